// bf16 weight GEMM on the 5th-generation tensor cores (sm_100a): y[M, N] (+)= x[M, K] * W[N, K]^T.
//
// The weight matrix is the streamed operand, so it takes the 128-row side of the instruction:
// each CTA owns a tile of 128 output features (rows of W) and MT rows of x, and computes
// D^T[128, MT] = W_tile[128, K] * x_tile[MT, K]^T with tcgen05.mma (A = W tile, B = x tile, both
// K-major in shared memory under the 128-byte swizzle, staged by TMA; accumulator in TMEM).  With
// MT = 16..64 the same kernel is a bandwidth-bound skinny GEMM for decode (weights read once, MMA
// cost hidden); with MT = 256 it is the dense GEMM of prefill / PRM scoring / catch-up.
//
// Roles inside a CTA of 7 warps: warps 0-3 read the accumulator out of TMEM (lane = output feature,
// column = x row) and write y, warp 4 issues the TMA loads of the weights and warp 6 those of x through a ring
// of shared-memory stages, warp 5 allocates TMEM and issues the MMAs.  Small problems are split along K across
// CTAs; the partial tiles go to scratch and are added in split order by the consumer or a reduction kernel
// (deterministic).
// Every wait on an mbarrier is bounded; on expiry the CTA raises an error flag and leaves cleanly.
#include <cuda.h>

#include <atomic>
#include <mutex>
#include <unordered_map>

#include "common.cuh"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace rsd {

static std::atomic<uint64_t> g_launches{0};
cudaError_t launched(int n_kernels) {
  g_launches.fetch_add((uint64_t)n_kernels, std::memory_order_relaxed);
  return cudaGetLastError();
}
uint64_t launches_total() { return g_launches.load(std::memory_order_relaxed); }
void note_replayed_launches(uint64_t n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

namespace {

using namespace tc;

constexpr int kTileN = 128;        // W rows per CTA (UMMA M)
constexpr int kTileK = 64;         // bf16 elements per 128-byte swizzled row
constexpr int kUmmaK = 16;
constexpr int kCounterBytes = 4096;
constexpr int kMaxSplitTiles = kCounterBytes / 4;
constexpr int kMaxSplitCtas = 640;
constexpr int kTcThreads = 224;    // four epilogue warps, weight producer, MMA issuer, x producer
// Ring stages of the decode pass's products of up to 16 rows into a fresh array (qkv, lm head), and of such gate/up tiles: enough to keep a
// stream going, and small enough that CTAs of the products after them (of three head tiles) find room beside these on an SM and
// have their first weights there when their turn comes.  14-layer iterations, us, full rings / these: 1.5B shape at 1 row 538 / 514, at 8
// 577 / 546; 7B shape 1391 / 1336 and 1418 / 1370.  Rings cut to the k-blocks of a CTA throughout spread the CTAs badly (16 rows 600 / 628); at 32 rows
// light rings cost the 7B shape's qkv product 8.4 -> 9.8 us.
constexpr int kLightStages = 4, kGuStages = 6;

// DEEP: a ring of eight (six for 128-row x tiles) stages for one CTA per SM, for grids that do not reach two CTAs per SM anyway (a lone
// CTA needs about twice the bytes in flight to keep its share of the HBM stream going).
template <int MT, bool DEEP = false> struct TcCfg {
  // tiles of up to 128 x-rows leave room for two CTAs per SM (one streams while the other starts
  // up or drains); the 256-row tile of the dense regime takes the SM alone
  static constexpr int kCtasPerSm = DEEP ? 1 : (MT <= 128 ? 2 : 1);
  static constexpr int kStages = DEEP ? (MT <= 64 ? 8 : 6) : (MT == 16 ? 6 : (MT == 32 ? 5 : (MT == 64 ? 4 : (MT == 128 ? 3 : 4))));
  static constexpr int kABytes = kTileN * kTileK * 2;
  static constexpr int kBBytes = MT * kTileK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kTmemCols = MT < 32 ? 32 : MT;
  static constexpr size_t smem_bytes(int stages) { return 1024 + (size_t)stages * kStageBytes + 256 + 512; }   // barriers, row scales
  static constexpr size_t kSmemBytes = smem_bytes(kStages);
  // gate/up mode: two exchange buffers [64 features][MT / 4 rows + 1] between the gate and the up warps; they
  // reuse the pipeline stages once the last MMA has read them
  static constexpr size_t kXchBytes = 2 * 64 * (size_t)(MT / 4 + 1) * 4;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
  static_assert(kXchBytes <= (size_t)(kStages < kGuStages ? kStages : kGuStages) * kStageBytes, "exchange buffers must fit in the stage ring");
  // instruction descriptor: fp32 accumulate, bf16 A and B, both K-major, N = MT, M = 128
  static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(MT >> 3) << 17) | ((uint32_t)(kTileN >> 4) << 24);
};

// SPLIT: the x operand is a pair (hi, lo) of bf16 matrices whose sum is the activation; the tile
// holds MT/2 rows of hi followed by the same MT/2 rows of lo, and the epilogue adds the two halves.
// GU (gate/up mode, SPLIT only): W is the stacked matrix [Wgate | Wup] of 2 * N rows; a CTA's 128-row tile is
// 64 gate rows and the 64 up rows of the same features (two TMA boxes of 64 rows), there is no K split, and the
// epilogue writes act = silu(gate) * up as the bf16 hi + lo operand pair [M, N] of the down projection instead
// of Y.  The gate values sit in TMEM lanes 0-63 (warps 0, 1), the up values in lanes 64-127 (warps 2, 3); the
// two warp pairs swap one half of the x rows each through shared memory, so all four warps compute.
// PROBE (one instantiation, reached only through the wait-probe entry): the producer warp issues NO copy, so the
// first stage never fills; the MMA warp's wait, cut to a few thousand polls, runs out, and the kernel must take its
// failure path -- error flag raised, epilogue warps released, tensor memory freed, clean return -- with nothing in
// flight.  This is how the failure path is exercised without a fault or an endless wait.
template <int MT, bool SPLIT, bool GU = false, bool DEEP = false, bool PROBE = false>
__global__ void __launch_bounds__(kTcThreads, TcCfg<MT, DEEP>::kCtasPerSm)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
               const __grid_constant__ CUtensorMap tm_x_lo, float* Y,
               int M, int N, int K, int accumulate, int splits, int kb_per_split, float* partials,
               int* err, const int32_t* n_active, RowScale rs, int n_stages,
               __nv_bfloat16* act_hi = nullptr, __nv_bfloat16* act_lo = nullptr, int f16 = 0) {
  // Programmatic dependent launch: the next kernel may be scheduled at once; this kernel sets itself
  // up and starts streaming its WEIGHT tiles (never written by any kernel) while its predecessors are
  // still running, and only then waits for them (griddepcontrol.wait) before it touches activations
  // or outputs.  The idle flag is a constant of the decode pass (see RSD_PDL_SYNC_LATE): requested here, looked at
  // after the first weight copies went out.  0: every row of the phase has finished.
  RSD_PDL_TRIGGER();
  const int active = n_active != nullptr ? ld_cg(n_active) : 1;
  using Cfg = TcCfg<MT, DEEP>;
  const uint32_t idesc = f16 ? (Cfg::kIdesc & ~((1u << 7) | (1u << 10))) : Cfg::kIdesc;   // both operands fp16 instead of bf16
  constexpr int kRows = SPLIT ? MT / 2 : MT;   // distinct x rows per tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + (size_t)n_stages * Cfg::kStageBytes);
  uint64_t* empty = full + n_stages;
  uint64_t* tmem_full = empty + n_stages;
  uint32_t* tmem_slot = (uint32_t*)(tmem_full + 1);
  volatile uint32_t* flags = tmem_slot + 1;   // [0] abort
  float* row_scale = (float*)(smem + (size_t)n_stages * Cfg::kStageBytes + 256);   // [kRows <= 128]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tile order.  CTAs start in the order of their linear index; with n fastest, the CTAs in flight together would
  // hold as many different weight tiles as there are SMs and the weight matrix would come from HBM once per row
  // tile of x.  With several row tiles the index is therefore walked in groups of eight row tiles, row tile
  // fastest: the CTAs in flight share eight x tiles and a few weight tiles, both of which stay in L2.
  int tile_n = blockIdx.x, tile_m = blockIdx.y;
  if (gridDim.y > 1) {
    constexpr int kGroup = 8;
    const int lin = blockIdx.y * gridDim.x + blockIdx.x, per_group = kGroup * gridDim.x;
    const int g0 = (lin / per_group) * kGroup, rem = lin % per_group;
    const int gsz = min(kGroup, (int)gridDim.y - g0);
    tile_m = g0 + rem % gsz;
    tile_n = rem / gsz;
  }
  const int n0 = tile_n * (GU ? kTileN / 2 : kTileN), m0 = tile_m * kRows, split = blockIdx.z;
  float* xch = (float*)smem;   // GU only: the exchange buffers reuse the pipeline stages, which are drained by then
  const int total_kb = (K + kTileK - 1) / kTileK;
  const int kb0 = split * kb_per_split;
  const int kb1 = min(total_kb, kb0 + kb_per_split);
  const int n_kb = kb1 - kb0;   // >= 1 by construction of the grid

  if (threadIdx.x == 128) {                    // the weight producer's first lane
    for (int s = 0; s < n_stages; ++s) { mbar_init(&full[s], 2); mbar_init(&empty[s], 1); }
    mbar_init(tmem_full, 1);
    flags[0] = 0; flags[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (threadIdx.x == 192) {             // the x producer's: its tensor maps are on their way under the wait
    tma_prefetch_map(&tm_x);
    if (SPLIT) tma_prefetch_map(&tm_x_lo);
  }
  if (warp == 5) tmem_alloc(tmem_slot, Cfg::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 4 || warp == 6) {
    // ---------------- TMA producers: warp 4 the weight tiles, warp 6 the x tiles ----------------
    // Two threads, since one pays 100+ cycles for every box it issues: the weight stream runs ahead under the wait for
    // the predecessors as far as the ring reaches, the x tiles follow after it.
    if (lane == 0 && !PROBE) {
      const int pre = min(n_kb, n_stages);
      int n_issue = n_kb;
      if (warp == 4) {
        if (active == 0) n_issue = pre;
      } else {
        RSD_PDL_WAIT();
        if (active == 0) {                     // close the stages of the weight copies that went out
          n_issue = 0;
          for (int i = 0; i < pre; ++i) mbar_arrive(&full[i]);
        }
      }
      int issued = 0, s = 0;
      uint32_t phase = 1;                      // of empty[s]: a fresh barrier passes for the parity before its first
      bool ok = true, ready = true;
      for (int i = 0; i < n_issue; ++i) {
        if (!ready && (!mbar_wait(&empty[s], phase) || flags[0])) { ok = false; break; }
        uint8_t* a = smem + (size_t)s * Cfg::kStageBytes;
        if (warp == 4) {
          mbar_expect_tx(&full[s], Cfg::kABytes);
          tma_load_2d(a, &tm_w, &full[s], (kb0 + i) * kTileK, n0);
          if (GU) tma_load_2d(a + Cfg::kABytes / 2, &tm_w, &full[s], (kb0 + i) * kTileK, N + n0);
        } else {
          mbar_expect_tx(&full[s], Cfg::kBBytes);
          tma_load_2d(a + Cfg::kABytes, &tm_x, &full[s], (kb0 + i) * kTileK, m0);
          if (SPLIT) tma_load_2d(a + Cfg::kABytes + kRows * kTileK * 2, &tm_x_lo, &full[s], (kb0 + i) * kTileK, m0);
        }
        issued = i + 1;
        if (++s == n_stages) { s = 0; phase ^= 1u; }
        ready = mbar_test(&empty[s], phase);
      }
      if (active == 0) {
        for (int i = 0; i < issued; ++i) mbar_wait(&full[i], 0);
      }
      if (!ok) {
        if (flags[0] == 0) {
          if (err) atomicCAS(err, 0, -5);
          flags[0] = 1;
        }
        // let the copies already in flight land before the CTA goes away (a stage that only one producer has reached
        // does not complete: the polls run out, long after the copy)
        for (int i = max(0, issued - n_stages); i < issued; ++i)
          mbar_wait(&full[i % n_stages], (i / n_stages) & 1, 1u << 16);
      }
    }
  } else if (warp == 5) {
    // ---------------- MMA issuer: the whole warp walks the ring, one lane issues ----------------
    // What a lone CTA gets through a second hangs on this loop.  Issued by a diverged thread, a narrow MMA took 140 cycles
    // (its descriptors were moved into uniform registers one by one), the wait 127 even when the data were there: 0.32 us
    // per k-block, 51 GB/s of weights a SM, whatever the ring's depth or the tile's width.  Converged and with the look ahead: 0.23 us.
    if (active != 0) {
      bool ok = true, ready = false;
      int s = 0;
      uint32_t phase = 0;
      const uint32_t on = elect_one();
      for (int i = 0; i < n_kb; ++i) {
        if (!ready) {
          ok = mbar_wait(&full[s], phase, PROBE ? 4096u : kWaitLimit);
          ok = __all_sync(0xFFFFFFFFu, ok && !flags[0]);
          if (!ok) break;
        }
        tc_fence_after();
        const int s1 = s + 1 == n_stages ? 0 : s + 1;
        const uint32_t phase1 = s1 == 0 ? phase ^ 1u : phase;
        // a look ahead at the next stage under this one's MMAs: even when the data are there, a wait takes 127 cycles
        ready = __all_sync(0xFFFFFFFFu, i + 1 < n_kb && mbar_test(&full[s1], phase1));
        const uint32_t a = smem_u32(smem + (size_t)s * Cfg::kStageBytes);
        const uint32_t b = a + Cfg::kABytes;
#pragma unroll
        for (int k = 0; k < kTileK / kUmmaK; ++k) {
          umma_bf16_if(on, tmem_base, smem_desc_sw128(a + k * kUmmaK * 2), smem_desc_sw128(b + k * kUmmaK * 2), idesc,
                       (i > 0 || k > 0) ? 1u : 0u);
        }
        umma_commit_if(on, &empty[s]);   // frees the stage once these MMAs have read it
        s = s1;
        phase = phase1;
      }
      if (ok) {
        umma_commit_if(on, tmem_full);
      } else if (lane == 0 && flags[0] == 0) {      // a wait expired (flags[0] != 0: someone else stopped the CTA)
        if (err) atomicCAS(err, 0, -5);
        flags[0] = 1;
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> registers -> global ----------------
    RSD_PDL_WAIT();                            // y and the partial sums belong to earlier kernels until now
    if (rs.ssq != nullptr && active != 0) {
      if (rs.n_chunks > 32) {
        // few rows in many chunks (gemm_rows.cu): a warp per row
        for (int r = warp; r < kRows && m0 + r < M; r += 4) {
          const float* src = rs.ssq + (size_t)(m0 + r) * rs.n_chunks;
          float sum = 0.f;
#pragma unroll 8
          for (int c = lane; c < rs.n_chunks; c += 32) sum += src[c];
          sum = warp_sum(sum);
          if (lane == 0) row_scale[r] = rsqrtf(sum * rs.inv_d + rs.eps);
        }
      } else {
        // RMSNorm denominators of this tile's x rows while the MMAs run: 128 / kRows threads per row, so that a row's
        // chunk sums are one round of loads, or two, instead of a chain as long as the row is wide
        constexpr int kLanes = kRows >= 128 ? 1 : (kRows >= 8 ? 128 / kRows : 16);
        const int r = threadIdx.x / kLanes, sub = threadIdx.x % kLanes;
        float sum = 0.f;
        if (r < kRows && m0 + r < M) {
          const float* src = rs.ssq + (size_t)(m0 + r) * rs.n_chunks;
#pragma unroll 8
          for (int c = sub; c < rs.n_chunks; c += kLanes) sum += src[c];
        }
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (sub == 0 && r < kRows) row_scale[r] = rsqrtf(sum * rs.inv_d + rs.eps);
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");   // the four epilogue warps only
    }
    // the four epilogue warps sleep in hardware between polls (about 1 us at most): busy polling by 128 threads
    // crowds the shared-memory pipe that the producer and the MMA issuer need for their own barriers
    bool ok = active != 0 && mbar_try_wait(tmem_full, 0);
    for (uint32_t i = 0; i < (1u << 21) && !ok && active != 0; ++i) {
      ok = mbar_try_wait_sleep(tmem_full, 0, 1000);
      if (!ok && flags[0]) break;                        // the CTA was stopped (an expired wait)
    }
    ok = __all_sync(0xFFFFFFFFu, ok);          // one answer for the warp: it goes on to tensor-memory loads together
    if (!ok && active != 0 && flags[0] == 0) {
      if (err) atomicCAS(err, 0, -5);
      flags[0] = 1;
    }
    tc_fence_after();
    const int n_local = warp * 32 + lane;
    const int n = n0 + n_local;
    const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16);
    const int m_valid = min(kRows, M - m0);
    if (GU) {
      // SwiGLU epilogue.  Rows [0, half) of the tile are finished by the gate warps (they receive the up values
      // of those rows), rows [half, kRows) by the up warps (they receive the gate values).
      constexpr int kHalf = kRows / 2, kLd = kHalf + 1, kCols = kHalf < 16 ? kHalf : 16;   // rows at a time
      // hi + lo of rows [at, at + kCols) of the tile
      auto rows_of = [&](int at, float (&v)[kCols]) {
        if (kRows == 8) {                                      // hi in columns 0..7, lo in columns 8..15 of the same load
          float w[16];
          tmem_ld16(taddr, w);
#pragma unroll
          for (int j = 0; j < kCols; ++j) v[j] = at == 0 ? w[j] + w[(j + 8) & 15] : w[(j + 4) & 15] + w[(j + 12) & 15];
        } else if (kRows == 16) {
          float w[2][16];
          tmem_ld16n<2>({taddr, taddr + 16}, w);
#pragma unroll
          for (int j = 0; j < kCols; ++j) v[j] = at == 0 ? w[0][j] + w[1][j] : w[0][(j + 8) & 15] + w[1][(j + 8) & 15];
        } else {
          float w[2][16];
          tmem_ld16n<2>({taddr + at, taddr + kRows + at}, w);
#pragma unroll
          for (int j = 0; j < kCols; ++j) v[j] = w[0][j & 15] + w[1][j & 15];
        }
      };
      const bool is_gate = warp < 2;
      const int l = (warp & 1) * 32 + lane;                    // feature within the 64-row half
      float* send = xch + (is_gate ? 64 * kLd : 0) + l * kLd;  // [0]: up values of the low rows, [1]: gate values of the high rows
      const float* recv = xch + (is_gate ? 0 : 64 * kLd) + l * kLd;
      const int send0 = is_gate ? kHalf : 0, own0 = is_gate ? 0 : kHalf;
      if (ok) {
#pragma unroll 1
        for (int c = 0; c < kHalf; c += kCols) {
          float v[kCols];
          rows_of(send0 + c, v);
#pragma unroll
          for (int j = 0; j < kCols; ++j) send[c + j] = v[j];
        }
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (ok && n0 + l < N) {
#pragma unroll 1
        for (int c = 0; c < kHalf; c += kCols) {
          if (own0 + c >= m_valid) break;
          float v[kCols];
          rows_of(own0 + c, v);
          // all sixteen, whether the row counts or not, and stores under predicates: a branch per row and a division per
          // element kept the elements from overlapping (32 rows: 4250 cycles behind the exchange, now 1760)
#pragma unroll
          for (int j = 0; j < kCols; ++j) {
            const float sc = rs.ssq != nullptr ? row_scale[own0 + c + j] : 1.f;
            const float mine = v[j] * sc, other = recv[c + j] * sc;
            v[j] = swiglu(is_gate ? mine : other, is_gate ? other : mine);
          }
          const size_t o = (size_t)(m0 + own0 + c) * N + n0 + l;
#pragma unroll
          for (int j = 0; j < kCols; ++j) {
            __nv_bfloat16 h, w;
            store_operand<__nv_bfloat16>(&h, &w, 0, v[j]);
            store_if(own0 + c + j < m_valid, act_hi + o + (size_t)j * N, h);
            store_if(own0 + c + j < m_valid, act_lo + o + (size_t)j * N, w);
          }
        }
      }
    } else if (ok) {
      // with several K-splits each CTA stores its partial sums as rows of a [split][M][N] array;
      // a reduction kernel adds the splits in order afterwards (deterministic)
      float* dst = splits == 1 ? Y : partials + (size_t)split * M * N;
      constexpr int kC = kRows >= 32 ? 32 : 16;    // rows at a time
      for (int c = 0; c < m_valid; c += kC) {
        float v[kC];
        if (SPLIT && kRows == 8) {                   // hi in columns 0..7, lo in columns 8..15 of the same load
          tmem_ld16(taddr, v);
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] += v[j + 8];
        } else {
          constexpr int G = kC / 16 * (SPLIT ? 2 : 1);
          float t[G][16];
          uint32_t at[G];
#pragma unroll
          for (int g = 0; g < G; ++g) at[g] = taddr + c + (SPLIT ? (g & 1) * kRows + (g >> 1) * 16 : g * 16);
          tmem_ld16n<G>(at, t);
#pragma unroll
          for (int j = 0; j < kC; ++j) v[j] = SPLIT ? t[j / 16 * 2][j % 16] + t[j / 16 * 2 + 1][j % 16] : t[j / 16][j % 16];
        }
        if (rs.ssq != nullptr) {
#pragma unroll
          for (int j = 0; j < kC; ++j) v[j] *= row_scale[(c + j) & 127];
        }
        if (n < N) {
          float* to = dst + (size_t)(m0 + c) * N + n;
          // when adding into y, all old values are requested before the first store: written as "*y += v" row by row,
          // every load would wait for the store before it (the compiler cannot rule out that two rows alias) and the
          // epilogue would crawl at one memory round trip per element
          if (accumulate && splits == 1) {
            float old[kC];
#pragma unroll
            for (int j = 0; j < kC; ++j) old[j] = c + j < m_valid ? to[(size_t)j * N] : 0.f;
#pragma unroll
            for (int j = 0; j < kC; ++j) v[j] += old[j];
          }
#pragma unroll
          for (int j = 0; j < kC; ++j) store_if(c + j < m_valid, to + (size_t)j * N, v[j]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::kTmemCols);
  }
}

// ---------------------------------------------------------------------------------------------------------
// Persistent form of the kernel above for the dense regime (more than 128 rows of x, no K split) and, with pairs, for the
// decode products of 65 to 128 rows that have more weight tiles than the chip has SMs (rs and n_active then as above; a
// single row tile): a CTA per SM walks the output tiles (128 weight rows x 128 x rows, the same grouped order), the TMA
// ring runs on from tile to tile, and the accumulator alternates between the two halves of tensor memory, so
// the epilogue of one tile (TMEM -> registers -> global) overlaps the MMAs of the next instead of ending the CTA.
// GU: gate/up tiles with the SwiGLU epilogue as above; the exchange buffers get shared memory of their own, since
// the ring is busy with the next tile.
// ---------------------------------------------------------------------------------------------------------
// SPLIT: the x tile is 128 rows of hi followed by the same 128 rows of lo (the epilogue adds the halves); otherwise it is
// 256 plain rows.  Either way the instruction's N is 256 and an accumulator takes 256 columns of tensor memory.
template <bool SPLIT, bool GU> struct PersistCfg {
  static constexpr int kMT = 256, kRows = SPLIT ? 128 : 256;
  static constexpr int kHalf = kRows / 2, kLd = kHalf + 1;
  static constexpr size_t kXchBytes = GU ? 2 * 64 * (size_t)kLd * 4 : 0;
  // the exchange buffers of the plain gate/up tile (2 x 64 x 129 floats) leave room for three stages
  static constexpr int kStages = (GU && !SPLIT) ? 3 : 4;
  static constexpr int kABytes = kTileN * kTileK * 2, kBBytes = kMT * kTileK * 2, kStageBytes = kABytes + kBBytes;
  static constexpr size_t kSmemBytes = 1024 + (size_t)kStages * kStageBytes + 256 + 512 + kXchBytes;   // barriers, row scales
  static constexpr uint32_t kIdesc = TcCfg<256>::kIdesc;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
};

// An instruction descriptor with n columns, and the operand formats fp16 where asked for.
__device__ __forceinline__ uint32_t tile_idesc(uint32_t idesc, int n, int f16) {
  idesc = (idesc & ~(0x3Fu << 17)) | ((uint32_t)(n >> 3) << 17);
  return f16 ? idesc & ~((1u << 7) | (1u << 10)) : idesc;
}

// warps 0..7: epilogue, warp 8: TMA producer, warp 9: MMA issuer and owner of the tensor-memory allocation
constexpr int kPersistEpiWarps = 8, kPersistThreads = 32 * (kPersistEpiWarps + 2);

// One output tile out of tensor memory, by the eight epilogue warps of a persistent kernel: warp w reads the lanes of
// quarter w % 4 (the hardware's rule), the two warps of a quarter take alternate groups of sixteen columns, which halves
// the time an accumulator stays occupied.  release() hands the accumulator back; it is called by one lane of every warp.
template <bool GU, bool SPLIT, typename Release>
__device__ __forceinline__ void persist_epilogue(uint32_t taddr, bool ok, int quarter, int lane, int col0, int n0, int m0, int M, int N,
                                                 float* Y, int accumulate, __nv_bfloat16* act_hi, __nv_bfloat16* act_lo, int f16,
                                                 float* xch, const float* row_scale, int rows, Release release) {
  using C = PersistCfg<SPLIT, GU>;
  constexpr int kColStep = 16 * (kPersistEpiWarps / 4);
  const int m_valid = min(rows, M - m0);
  auto ld = [&](int c, float (&v)[16]) {             // sixteen columns, the low halves' results added
    if (SPLIT) {
      float t[2][16];
      tmem_ld16n<2>({taddr + c, taddr + C::kRows + c}, t);
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = t[0][j] + t[1][j];
    } else {
      tmem_ld16(taddr + c, v);
    }
  };
  if (!GU) {
    const int n = n0 + quarter * 32 + lane;
    if (ok) {
      for (int c = col0; c < m_valid; c += kColStep) {
        float v[16];
        ld(c, v);
        if (row_scale != nullptr) {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] *= row_scale[(c + j) & 127];
        }
        if (n < N) {
          // all sixteen old values first, then the stores (see the one-tile kernel's epilogue)
          if (accumulate) {
            float old[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) old[j] = c + j < m_valid ? Y[(size_t)(m0 + c + j) * N + n] : 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += old[j];
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (c + j < m_valid) Y[(size_t)(m0 + c + j) * N + n] = v[j];
          }
        }
      }
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) release();
  } else {
    const bool is_gate = quarter < 2;
    const int l = (quarter & 1) * 32 + lane;
    float* send = xch + (is_gate ? 64 * C::kLd : 0) + l * C::kLd;
    const float* recv = xch + (is_gate ? 0 : 64 * C::kLd) + l * C::kLd;
    const int half = rows / 2, send0 = is_gate ? half : 0, own0 = is_gate ? 0 : half;
    if (ok) {
#pragma unroll 1
      for (int c = col0; c < half; c += kColStep) {
        float v[16];
        ld(send0 + c, v);
#pragma unroll
        for (int j = 0; j < 16; ++j) send[c + j] = v[j];
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kPersistEpiWarps) : "memory");
    if (ok && n0 + l < N) {
#pragma unroll 1
      for (int c = col0; c < half; c += kColStep) {
        if (own0 + c >= m_valid) break;
        float v[16];
        ld(own0 + c, v);
        // all sixteen, then the stores: see the one-tile kernel's epilogue
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float sc = row_scale != nullptr ? row_scale[(own0 + c + j) & 127] : 1.f;
          const float mine = v[j] * sc, other = recv[c + j] * sc;
          v[j] = swiglu(is_gate ? mine : other, is_gate ? other : mine);
        }
        const size_t o = (size_t)(m0 + own0 + c) * N + n0 + l;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (own0 + c + j < m_valid) {
            if (!SPLIT && f16) store_operand<__half>(reinterpret_cast<__half*>(act_hi), nullptr, o + (size_t)j * N, v[j]);
            else store_operand<__nv_bfloat16>(act_hi, SPLIT ? act_lo : nullptr, o + (size_t)j * N, v[j]);
          }
        }
      }
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) release();
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kPersistEpiWarps) : "memory");   // the exchange buffers are free for the next tile
  }
}

template <bool GU, bool SPLIT>
__global__ void __launch_bounds__(kPersistThreads, 1)
gemm_tc_persistent_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                          const __grid_constant__ CUtensorMap tm_x_lo, float* Y, int M, int N, int K,
                          int accumulate, int n_tiles_n, int n_tiles_m, int* err,
                          __nv_bfloat16* act_hi, __nv_bfloat16* act_lo, int f16, const int32_t* n_active, RowScale rs, int tile_rows) {
  RSD_PDL_TRIGGER();
  if (n_active != nullptr && ld_cg(n_active) == 0) {      // every row of the decode phase has finished
    RSD_PDL_WAIT();
    return;
  }
  using C = PersistCfg<SPLIT, GU>;
  // f16: both operands are fp16 (weights re-encoded at load, one fp16 activation operand); the MMA's operand-format
  // fields become 0 and a gate/up tile writes its activations as fp16.  Otherwise bf16 throughout.
  const int rows = SPLIT ? C::kRows : tile_rows;           // x rows of a tile: of plain operands the launch's choice
  const uint32_t idesc = tile_idesc(C::kIdesc, SPLIT ? C::kMT : rows, f16);
  const uint32_t stage_bytes = C::kABytes + (SPLIT ? C::kMT : rows) * kTileK * 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + (size_t)C::kStages * C::kStageBytes);
  uint64_t* empty = full + C::kStages;
  uint64_t* acc_full = empty + C::kStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  volatile uint32_t* stop = tmem_slot + 1;
  float* row_scale = (float*)(smem + (size_t)C::kStages * C::kStageBytes + 256);   // [128]
  float* xch = row_scale + 128;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total_kb = (K + kTileK - 1) / kTileK, n_tiles = n_tiles_n * n_tiles_m;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], kPersistEpiWarps); }
    *stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kPersistEpiWarps + 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // tile t -> (row tile of x, tile of W): groups of eight row tiles, row tile fastest
  auto tile_of = [&](int t, int& tm, int& tn) {
    const int per_group = 8 * n_tiles_n, g0 = (t / per_group) * 8, rem = t % per_group, gsz = min(8, n_tiles_m - g0);
    tm = g0 + rem % gsz;
    tn = rem / gsz;
  };
  auto fail = [&]() { if (*stop == 0) { if (err) atomicCAS(err, 0, -5); *stop = 1; } };

  if (warp == kPersistEpiWarps) {
    // ---------------- TMA producer: the whole warp walks the ring, one lane issues ----------------
    const uint32_t on = elect_one();
    uint32_t it = 0, s = 0, phase = 1;
    bool ready = true;
    auto load_w = [&](uint32_t st, int kb, int n0) {
      uint8_t* a = smem + (size_t)st * C::kStageBytes;
      mbar_expect_tx_if(on, &full[st], stage_bytes);
      tma_load_2d_if(on, a, &tm_w, &full[st], kb * kTileK, n0);
      if (GU) tma_load_2d_if(on, a + C::kABytes / 2, &tm_w, &full[st], kb * kTileK, N + n0);
    };
    // the weight tiles of the first ring of stages go out before the predecessors have finished
    uint32_t ahead = 0;
    if (blockIdx.x < n_tiles) {
      int tm, tn;
      tile_of(blockIdx.x, tm, tn);
      for (; ahead < (uint32_t)min(C::kStages, total_kb); ++ahead) load_w(ahead, ahead, tn * (GU ? kTileN / 2 : kTileN));
    }
    RSD_PDL_WAIT();
    bool ok = true;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
      int tm, tn;
      tile_of(t, tm, tn);
      const int n0 = tn * (GU ? kTileN / 2 : kTileN), m0 = tm * rows;
      for (int kb = 0; kb < total_kb; ++kb, ++it) {
        if (it >= ahead) {
          if (!ready) {
            ok = mbar_wait(&empty[s], phase);
            ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
            if (!ok) break;
          }
          load_w(s, kb, n0);
        }
        uint8_t* b = smem + (size_t)s * C::kStageBytes + C::kABytes;
        tma_load_2d_if(on, b, &tm_x, &full[s], kb * kTileK, m0);
        if (SPLIT) tma_load_2d_if(on, b + C::kRows * kTileK * 2, &tm_x_lo, &full[s], kb * kTileK, m0);
        if (++s == (uint32_t)C::kStages) { s = 0; phase ^= 1u; }
        ready = __all_sync(0xFFFFFFFFu, mbar_test(&empty[s], phase));
      }
    }
    if (!ok) {
      if (on) fail();
      // copies in flight must land before the CTA goes away
      for (uint32_t i = (it > (uint32_t)C::kStages ? it - C::kStages : 0); i < it; ++i)
        for (uint32_t k = 0; k < (1u << 16); ++k)
          if (mbar_try_wait(&full[i % C::kStages], (i / C::kStages) & 1u)) break;
    }
  } else if (warp == kPersistEpiWarps + 1) {
    // ---------------- MMA issuer, likewise ----------------
    const uint32_t on = elect_one();
    uint32_t s = 0, phase = 0, n_acc = 0;
    bool ok = true, ready = false;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++n_acc) {
      const uint32_t b = n_acc & 1u;
      ok = mbar_wait(&acc_empty[b], ((n_acc >> 1) & 1u) ^ 1u);
      ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + b * (uint32_t)C::kMT;
      for (int kb = 0; kb < total_kb; ++kb) {
        if (!ready) {
          ok = mbar_wait(&full[s], phase);
          ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
          if (!ok) break;
        }
        tc_fence_after();
        const uint32_t s1 = s + 1 == (uint32_t)C::kStages ? 0u : s + 1, phase1 = s1 == 0 ? phase ^ 1u : phase;
        ready = __all_sync(0xFFFFFFFFu, mbar_test(&full[s1], phase1));        // under this stage's MMAs
        const uint32_t a = smem_u32(smem + (size_t)s * C::kStageBytes), bb = a + C::kABytes;
#pragma unroll
        for (int k = 0; k < kTileK / kUmmaK; ++k)
          umma_bf16_if(on, d_tmem, smem_desc_sw128(a + k * kUmmaK * 2), smem_desc_sw128(bb + k * kUmmaK * 2), idesc,
                       (kb > 0 || k > 0) ? 1u : 0u);
        umma_commit_if(on, &empty[s]);
        s = s1;
        phase = phase1;
      }
      if (ok) umma_commit_if(on, &acc_full[b]);
    }
    if (!ok && on) fail();
  } else {
    // ---------------- epilogue warps ----------------
    const int quarter = warp & 3, col0 = (warp >> 2) * 16;
    uint32_t n_acc = 0;
    RSD_PDL_WAIT();                            // y, the activations' sums of squares and act belong to earlier kernels until now
    const bool scaled = SPLIT && rs.ssq != nullptr;
    if (scaled) {
      // RMSNorm denominators of the single row tile, two threads per row
      const int r = threadIdx.x >> 1, sub = threadIdx.x & 1;
      float sum = 0.f;
      if (r < M) {
#pragma unroll 8
        for (int c = sub; c < rs.n_chunks; c += 2) sum += rs.ssq[(size_t)r * rs.n_chunks + c];
      }
      sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 1);
      if (sub == 0) row_scale[r] = rsqrtf(sum * rs.inv_d + rs.eps);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kPersistEpiWarps) : "memory");
    }
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++n_acc) {
      int tm, tn;
      tile_of(t, tm, tn);
      const int n0 = tn * (GU ? kTileN / 2 : kTileN), m0 = tm * rows;
      const uint32_t b = n_acc & 1u;
      bool ok = mbar_try_wait(&acc_full[b], (n_acc >> 1) & 1u);
      for (uint32_t i = 0; i < (1u << 21) && !ok && !*stop; ++i) ok = mbar_try_wait_sleep(&acc_full[b], (n_acc >> 1) & 1u, 1000);
      ok = __all_sync(0xFFFFFFFFu, ok);        // one answer for the warp
      if (!ok) fail();
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + b * (uint32_t)C::kMT;
      persist_epilogue<GU, SPLIT>(taddr, ok, quarter, lane, col0, n0, m0, M, N, Y, accumulate, act_hi, act_lo, f16, xch,
                                  scaled ? row_scale : nullptr, rows, [&]() { mbar_arrive(&acc_empty[b]); });
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kPersistEpiWarps + 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ---------------------------------------------------------------------------------------------------------
// The persistent kernel for pairs of CTAs (cta_group::2): two neighbouring SMs share one tile of 256 weight rows x 256
// operand rows (256 plain rows of x, or 128 rows as hi | lo).  Each holds its 128 weight rows and HALF of the operand rows,
// and one thread of the leading CTA issues 256 x 256 x 16 MMAs that read both halves from both shared memories.
// Why: a lone CTA's 128 x 256 x 16 MMA takes 128 cycles and reads 12 KB, and the copies bring 48 KB every four MMAs:
// together 192 bytes a cycle against the 128 that an SM's shared memory delivers.  In a pair each SM reads 8 KB and
// receives 32 KB instead, 128 bytes a cycle, and L2 delivers two thirds of the bytes; the ring also gets deeper.
// The accumulator, 256 columns in each SM's tensor memory (lanes = its own weight rows), alternates as above, and the
// epilogues are those of the lone CTA, each SM finishing its own 128 weight rows (64 features in the gate/up mode).
// Barriers: full[s] and acc_empty[b] of the leader count for both CTAs (the follower's copies and epilogue warps report
// there), empty[s] and acc_full[b] are signalled in both by the MMAs' commits.  Every wait is bounded.
// ---------------------------------------------------------------------------------------------------------
template <bool SPLIT, bool GU> struct PairCfg {
  using P = PersistCfg<SPLIT, GU>;
  static constexpr int kStages = (GU && !SPLIT) ? 5 : 6;   // beside the exchange buffers of the plain gate/up tile: five
  static constexpr int kABytes = kTileN * kTileK * 2, kBBytes = 128 * kTileK * 2, kStageBytes = kABytes + kBBytes;
  static constexpr size_t kSmemBytes = 1024 + (size_t)kStages * kStageBytes + 256 + P::kXchBytes;
  // as for the lone CTA, with M = 256
  static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
  static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
};

template <bool GU, bool SPLIT>
__global__ void __launch_bounds__(kPersistThreads, 1)
gemm_tc_pair_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                    const __grid_constant__ CUtensorMap tm_x_lo, float* Y, int M, int N, int K, int accumulate, int n_tiles_n,
                    int n_tiles_m, int* err, __nv_bfloat16* act_hi, __nv_bfloat16* act_lo, int f16, int tile_rows) {
  RSD_PDL_TRIGGER();
  using C = PairCfg<SPLIT, GU>;
  const int rows = SPLIT ? C::P::kRows : tile_rows;        // x rows of a tile: of plain operands the launch's choice
  const int half = SPLIT ? 128 : rows / 2;                 // operand rows of one CTA
  const uint32_t idesc = tile_idesc(C::kIdesc, 2 * half, f16), stage_bytes = C::kABytes + half * kTileK * 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + (size_t)C::kStages * C::kStageBytes);
  uint64_t* empty = full + C::kStages;
  uint64_t* acc_full = empty + C::kStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  volatile uint32_t* stop = tmem_slot + 1;
  float* xch = (float*)(smem + (size_t)C::kStages * C::kStageBytes + 256);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int total_kb = (K + kTileK - 1) / kTileK, n_tiles = n_tiles_n * n_tiles_m;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * kPersistEpiWarps); }
    *stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == kPersistEpiWarps + 1) tmem_alloc_pair(tmem_slot, 512);
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();                          // both CTAs' barriers and tensor memory are set up
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // tile t -> (row tile of x, pair of weight tiles): groups of eight row tiles, row tile fastest
  auto tile_of = [&](int t, int& tm, int& tn) {
    const int per_group = 8 * n_tiles_n, g0 = (t / per_group) * 8, rem = t % per_group, gsz = min(8, n_tiles_m - g0);
    tm = g0 + rem % gsz;
    tn = rem / gsz;
  };
  constexpr int kFeat = GU ? kTileN / 2 : kTileN;          // output features of one CTA's tile
  auto first_feature = [&](int tn) { return (2 * tn + (int)rank) * kFeat; };
  auto fail = [&]() { if (*stop == 0) { if (err) atomicCAS(err, 0, -5); *stop = 1; } };

  if (warp == kPersistEpiWarps) {
    // ---------------- producer: this CTA's weight rows and its half of the operand rows; one lane issues ----------------
    const uint32_t on = elect_one(), lead = on && rank == 0 ? 1u : 0u;
    if (on) tma_prefetch_map(&tm_x);
    uint32_t it = 0, s = 0, phase = 1, ahead = 0;
    bool ready = true, ok = true;
    auto load_w = [&](uint32_t st, int kb, int n0) {
      uint8_t* a = smem + (size_t)st * C::kStageBytes;
      const uint32_t bar = cluster_addr(&full[st], 0);
      mbar_expect_tx_if(lead, &full[st], 2 * stage_bytes);        // both CTAs' bytes
      tma_load_2d_pair_if(on, a, &tm_w, bar, kb * kTileK, n0);
      if (GU) tma_load_2d_pair_if(on, a + C::kABytes / 2, &tm_w, bar, kb * kTileK, N + n0);
    };
    // the weight tiles of the first ring of stages go out before the predecessors have finished
    if (pair < n_tiles) {
      int tm, tn;
      tile_of(pair, tm, tn);
      for (; ahead < (uint32_t)min(C::kStages, total_kb); ++ahead) load_w(ahead, ahead, first_feature(tn));
    }
    RSD_PDL_WAIT();
    for (int t = pair; t < n_tiles && ok; t += n_pairs) {
      int tm, tn;
      tile_of(t, tm, tn);
      const int n0 = first_feature(tn), m0 = tm * rows;
      for (int kb = 0; kb < total_kb; ++kb, ++it) {
        if (it >= ahead) {
          if (!ready) {
            ok = mbar_wait(&empty[s], phase);
            ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
            if (!ok) break;
          }
          load_w(s, kb, n0);
        }
        uint8_t* b = smem + (size_t)s * C::kStageBytes + C::kABytes;
        const uint32_t bar = cluster_addr(&full[s], 0);
        if (SPLIT) tma_load_2d_pair_if(on, b, rank == 0 ? &tm_x : &tm_x_lo, bar, kb * kTileK, m0);
        else tma_load_2d_pair_if(on, b, &tm_x, bar, kb * kTileK, m0 + (int)rank * half);
        if (++s == (uint32_t)C::kStages) { s = 0; phase ^= 1u; }
        ready = __all_sync(0xFFFFFFFFu, mbar_test(&empty[s], phase));
      }
    }
    if (!ok) {
      if (on) fail();
      // the copies still in flight report to the leader's barriers, which a follower cannot poll: a few milliseconds are far
      // longer than any of them takes
      for (int i = 0; i < 4096; ++i) __nanosleep(1000);
    }
  } else if (warp == kPersistEpiWarps + 1) {
    // ---------------- MMA issuer: one lane of the leading CTA ----------------
    if (rank == 0) {
      const uint32_t on = elect_one();
      uint32_t s = 0, phase = 0, n_acc = 0;
      bool ok = true, ready = false;
      for (int t = pair; t < n_tiles && ok; t += n_pairs, ++n_acc) {
        const uint32_t b = n_acc & 1u;
        ok = mbar_wait(&acc_empty[b], ((n_acc >> 1) & 1u) ^ 1u);
        ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + b * 256u;
        for (int kb = 0; kb < total_kb; ++kb) {
          if (!ready) {
            ok = mbar_wait(&full[s], phase);
            ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t s1 = s + 1 == (uint32_t)C::kStages ? 0u : s + 1, phase1 = s1 == 0 ? phase ^ 1u : phase;
          ready = __all_sync(0xFFFFFFFFu, mbar_test(&full[s1], phase1));      // under this stage's MMAs
          const uint32_t a = smem_u32(smem + (size_t)s * C::kStageBytes), bb = a + C::kABytes;
#pragma unroll
          for (int k = 0; k < kTileK / kUmmaK; ++k)
            umma_f16_pair_if(on, d_tmem, smem_desc_sw128(a + k * kUmmaK * 2), smem_desc_sw128(bb + k * kUmmaK * 2), idesc,
                             (kb > 0 || k > 0) ? 1u : 0u);
          umma_commit_pair_if(on, &empty[s]);
          s = s1;
          phase = phase1;
        }
        if (ok) umma_commit_pair_if(on, &acc_full[b]);
      }
      if (!ok && on) fail();
    }
  } else {
    // ---------------- epilogue warps of both CTAs ----------------
    const int quarter = warp & 3, col0 = (warp >> 2) * 16;
    uint32_t n_acc = 0;
    RSD_PDL_WAIT();                            // y and act belong to earlier kernels until now
    for (int t = pair; t < n_tiles; t += n_pairs, ++n_acc) {
      int tm, tn;
      tile_of(t, tm, tn);
      const uint32_t b = n_acc & 1u;
      bool ok = mbar_try_wait(&acc_full[b], (n_acc >> 1) & 1u);
      for (uint32_t i = 0; i < (1u << 21) && !ok && !*stop; ++i) ok = mbar_try_wait_sleep(&acc_full[b], (n_acc >> 1) & 1u, 1000);
      ok = __all_sync(0xFFFFFFFFu, ok);        // one answer for the warp
      if (!ok) fail();
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + b * 256u;
      persist_epilogue<GU, SPLIT>(taddr, ok, quarter, lane, col0, first_feature(tn), tm * rows, M, N, Y, accumulate, act_hi, act_lo,
                                  f16, xch, nullptr, rows, [&]() { mbar_arrive_cluster(cluster_addr(&acc_empty[b], 0)); });
    }
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();                          // nobody leaves while the other CTA may still signal its barriers
  if (warp == kPersistEpiWarps + 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// y[m, n] (+)= sum over splits of partials[s][m][n], splits added in order; 4 columns per thread, or one where a caller's y or
// scratch does not start on a 16-byte boundary.
__global__ void __launch_bounds__(256)
splitk_reduce_kernel(const float* __restrict__ partials, float* __restrict__ Y, int M, int N, int splits, int accumulate,
                     const int32_t* __restrict__ n_active) {
  RSD_PDL_SYNC();
  if (n_active != nullptr && *n_active == 0) return;
  if (((uintptr_t)Y | (uintptr_t)partials) & 15) {
    const size_t total = (size_t)M * N;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
      float acc = accumulate ? Y[i] : 0.f;
      for (int sidx = 0; sidx < splits; ++sidx) acc += __ldcg(partials + (size_t)sidx * total + i);
      Y[i] = acc;
    }
    return;
  }
  const size_t total4 = (size_t)M * N / 4, stride = (size_t)M * N / 4;
  const float4* p4 = reinterpret_cast<const float4*>(partials);
  float4* y4 = reinterpret_cast<float4*>(Y);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total4; i += (size_t)gridDim.x * blockDim.x) {
    float4 acc = accumulate ? y4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    int sidx = 0;
    for (; sidx + 4 <= splits; sidx += 4) {
      const float4 a = __ldcg(p4 + (size_t)sidx * stride + i), b = __ldcg(p4 + (size_t)(sidx + 1) * stride + i);
      const float4 c = __ldcg(p4 + (size_t)(sidx + 2) * stride + i), d = __ldcg(p4 + (size_t)(sidx + 3) * stride + i);
      acc.x += a.x; acc.y += a.y; acc.z += a.z; acc.w += a.w;
      acc.x += b.x; acc.y += b.y; acc.z += b.z; acc.w += b.w;
      acc.x += c.x; acc.y += c.y; acc.z += c.z; acc.w += c.w;
      acc.x += d.x; acc.y += d.y; acc.z += d.z; acc.w += d.w;
    }
    for (; sidx < splits; ++sidx) {
      const float4 a = __ldcg(p4 + (size_t)sidx * stride + i);
      acc.x += a.x; acc.y += a.y; acc.z += a.z; acc.w += a.w;
    }
    y4[i] = acc;
  }
}

// ---- tensor maps (host) -----------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  });
  return fn;
}

struct MapKey {
  const void* ptr; int rows, cols, box_rows;
  bool operator==(const MapKey& o) const { return ptr == o.ptr && rows == o.rows && cols == o.cols && box_rows == o.box_rows; }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    size_t h = std::hash<const void*>()(k.ptr);
    h ^= std::hash<long long>()(((long long)k.rows << 32) ^ ((long long)k.cols << 8) ^ k.box_rows) + 0x9e3779b97f4a7c15ull + (h << 6) + (h >> 2);
    return h;
  }
};

// Row-major bf16 matrix [rows, cols]; box = 64 columns x box_rows rows; 128-byte swizzle.  Maps are
// cached by (pointer, shape): weights and activation buffers keep their addresses for a context's life.
bool get_map(const void* ptr, int rows, int cols, int box_rows, CUtensorMap* out) {
  static std::mutex mu;
  static std::unordered_map<MapKey, CUtensorMap, MapKeyHash> cache;
  std::lock_guard<std::mutex> lock(mu);
  MapKey key{ptr, rows, cols, box_rows};
  auto it = cache.find(key);
  if (it != cache.end()) { *out = it->second; return true; }
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (cache.size() > 65536) cache.clear();
  cache.emplace(key, m);
  *out = m;
  return true;
}

// Rows of x per tile: the smallest tile that holds M, up to 128 (split operand) or 256 (plain).
int pick_rows(int M, bool split_operand) {
  if (split_operand && M <= 8) return 8;
  if (M <= 16) return 16;
  if (M <= 32) return 32;
  if (M <= 64) return 64;
  if (M <= 128 || split_operand) return 128;
  return 256;
}

struct TcPlan { int rows, mt, n_tiles, m_tiles, splits, kb_per_split; };

TcPlan plan_tc(int M, int N, int K, bool split_operand) {
  TcPlan p;
  p.rows = pick_rows(M, split_operand);
  p.mt = split_operand ? 2 * p.rows : p.rows;
  p.n_tiles = (N + kTileN - 1) / kTileN;
  p.m_tiles = (M + p.rows - 1) / p.rows;
  const int tiles = p.n_tiles * p.m_tiles;
  const int total_kb = (K + kTileK - 1) / kTileK;
  int splits = 1;
  if (tiles < 148 && tiles <= kMaxSplitTiles && N % 4 == 0 && (p.rows <= 64 || (split_operand && M <= 128))) {
    // aim at one wave, each CTA with at least two k-blocks: of two CTAs per SM where the partial sums are small, of one where
    // pairs of more than 16 rows make them larger than what a second CTA saves (an iteration of 14 layers, 1.5B / 7B shapes:
    // 32 rows 726 / 1661 us with two, 710 / 1641 with one; 64 rows 905 / 1942 and 872 / 1900).  Plain rows (in the step
    // loop: short passes of the PRM) keep two: neither is better throughout (two / one, the reduction included: 32 x 1536 x 8960
    // 8.3 / 7.1 us, 32 x 4608 x 3584 7.0 / 7.1, 64 x 3584 x 18944 28.1 / 30.3).
    // 65 to 128 rows with pairs are the decode passes of large batches: without the split the 12 tiles of a
    // 1536 x 8960 product leave 136 SMs idle (58 us at 128 rows; 11 us with 12 splits).
    splits = std::max(1, (p.rows <= 16 || !split_operand ? 2 * 148 : 148) / tiles);
    // (Splits of four k-blocks instead of two for the qkv product of up to 16 rows, whose sums the rotation adds up: an iteration of 14 layers of the
    // 1.5B shape at 4 / 6 / 8 / 12 / 16 rows 496 / 505 / 530 / 558 / 569 us, with two 496 / 508 / 532 / 558 / 567; and the sums' error against fp64
    // grows with the chain of MMAs, 1.4 -> 2.4e-7.)
    splits = std::min(splits, std::max(1, total_kb / 2));
    splits = std::min(splits, kMaxSplitCtas / tiles);
    splits = std::max(splits, 1);
  }
  p.kb_per_split = (total_kb + splits - 1) / splits;
  p.splits = (total_kb + p.kb_per_split - 1) / p.kb_per_split;   // no empty split
  return p;
}

template <int MT, bool SPLIT, bool DEEP = false>
cudaError_t launch_mt(const CUtensorMap& tw, const CUtensorMap& tx, const CUtensorMap& txl, float* y, int M, int N, int K,
                      int accumulate, const TcPlan& p, float* partials, int* err, const int32_t* n_active,
                      bool defer_reduce, RowScale rs, cudaStream_t s, int f16 = 0) {
  using Cfg = TcCfg<MT, DEEP>;
  static OncePerDevice configured;
  const cudaError_t set = allow_smem(configured, gemm_tc_kernel<MT, SPLIT, false, DEEP>, Cfg::kSmemBytes);
  if (set != cudaSuccess) return set;
  dim3 grid(p.n_tiles, p.m_tiles, p.splits);
  const int stages = MT <= 32 && !accumulate && rs.ssq != nullptr ? std::min(Cfg::kStages, kLightStages) : Cfg::kStages;
  RSD_LAUNCH((gemm_tc_kernel<MT, SPLIT, false, DEEP>), grid, kTcThreads, Cfg::smem_bytes(stages), s, tw, tx, txl, y, M, N, K, accumulate, p.splits,
                                                                     p.kb_per_split, partials, err, n_active, rs, stages,
                                                                     (__nv_bfloat16*)nullptr, (__nv_bfloat16*)nullptr, f16);
  if (p.splits > 1 && !defer_reduce) {
    const size_t total4 = (size_t)M * N / 4;
    const int blocks = (int)std::min<size_t>((total4 + 255) / 256, 148 * 8);
    RSD_LAUNCH((splitk_reduce_kernel), blocks, 256, 0, s, partials, y, M, N, p.splits, accumulate, n_active);
    return launched(2);
  }
  return launched(1);
}

}  // namespace

// Row-major bf16 matrix [rows, cols] as a TMA tensor map with a 64-column x box_rows box under the 128-byte swizzle.
bool tc_tensor_map(const void* ptr, int rows, int cols, int box_rows, CUtensorMap* out) {
  return get_map(ptr, rows, cols, box_rows, out);
}

bool tc_tensor_map_rows(const void* ptr, bool f32, int rows, int cols, CUtensorMap* out) {
  EncodeTiledFn fn = encode_fn();
  if (!fn || ((uintptr_t)ptr & 15) || cols % (f32 ? 4 : kTileK) != 0) return false;
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r;
  if (f32) {
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)cols * 4};
    const cuuint32_t box[2] = {256, 8};
    r = fn(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    const cuuint64_t dims[3] = {kTileK, (cuuint64_t)rows, (cuuint64_t)cols / kTileK}, strides[2] = {(cuuint64_t)cols * 2, kTileK * 2};
    const cuuint32_t box[3] = {kTileK, 8, 8};
    r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  return r == CUDA_SUCCESS;
}

// One layer's slab of fp16 KV pages as a tensor of 4096-byte blocks (per page: the keys of every KV head
// [16 tokens][128 dims], then the values [128 dims][16 tokens]), one box per block:
//   keys    (64 dims, 8 tokens, 2 dim halves, 2 token groups, block)   128-byte swizzle: lands as
//           [token group][dim half][8 tokens][64 dims], the order the score MMA wants its operand in
//   values  (16 tokens, 128 dims, block)                               32-byte swizzle
// The block extent is a bound on what a coordinate may name, not an allocation size: only the boxes a kernel asks
// for are touched.
bool tc_tensor_map_kv(const void* pool_layer, int values, CUtensorMap* out) {
  static std::mutex mu;
  static std::unordered_map<MapKey, CUtensorMap, MapKeyHash> cache;
  std::lock_guard<std::mutex> lock(mu);
  MapKey key{pool_layer, values, 0, 0};
  auto it = cache.find(key);
  if (it != cache.end()) { *out = it->second; return true; }
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  CUtensorMap m;
  const cuuint64_t blocks = 1ull << 30;
  CUresult r;
  if (values) {
    cuuint64_t dims[3] = {16, 128, blocks};
    cuuint64_t strides[2] = {32, 4096};
    cuuint32_t box[3] = {16, 128, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(pool_layer), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    cuuint64_t dims[5] = {64, 8, 2, 2, blocks};
    cuuint64_t strides[4] = {256, 128, 2048, 4096};      // token, dim half, token group, block
    cuuint32_t box[5] = {64, 8, 2, 2, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<void*>(pool_layer), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  if (r != CUDA_SUCCESS) return false;
  if (cache.size() > 65536) cache.clear();
  cache.emplace(key, m);
  *out = m;
  return true;
}

// Launches the PROBE instantiation on a 128 x 16 x 64 problem whose copies are never issued (W and x are mapped but
// not read): the kernel's bounded wait expires and *err (the int at byte 4096 of the scratch) becomes -5.
cudaError_t launch_gemm_wait_probe(const void* W, const void* x, float* y, void* scratch, size_t scratch_bytes, cudaStream_t s) {
  if (!scratch || scratch_bytes < gemm_scratch_bytes(16)) return cudaErrorInvalidValue;
  CUtensorMap tw, tx;
  if (!get_map(W, 128, 64, kTileN, &tw) || !get_map(x, 16, 64, 16, &tx)) return cudaErrorNotSupported;
  static OncePerDevice configured;
  const cudaError_t set = allow_smem(configured, gemm_tc_kernel<16, false, false, false, true>, TcCfg<16>::kSmemBytes);
  if (set != cudaSuccess) return set;
  int* err = (int*)((char*)scratch + kCounterBytes);
  float* partials = (float*)((char*)scratch + kCounterBytes + 256);
  RSD_LAUNCH((gemm_tc_kernel<16, false, false, false, true>), dim3(1, 1, 1), kTcThreads, TcCfg<16>::kSmemBytes, s, tw, tx, tx, y, 16, 128, 64, 0, 1, 1,
             partials, err, (const int32_t*)nullptr, RowScale(), TcCfg<16>::kStages, (__nv_bfloat16*)nullptr, (__nv_bfloat16*)nullptr, 0);
  return launched(1);
}

bool gemm_tc_supported(int dtype, int M, int N, int K) {
  return dtype == 1 && M >= 1 && N >= 1 && K >= 8 && K % 8 == 0;
}

static int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 0;
  }
  return n;
}

// Dense regime (M > 128 rows, no K split, no row scale, no idle flag) and wide decode products: persistent kernel.
template <bool GU, bool SPLIT>
static cudaError_t launch_persistent(const CUtensorMap& tw, const CUtensorMap& tx, const CUtensorMap& txl, float* y, int M, int N,
                                     int K, int accumulate, int* err, __nv_bfloat16* act_hi, __nv_bfloat16* act_lo, cudaStream_t s,
                                     int f16 = 0, const int32_t* n_active = nullptr, RowScale rs = RowScale(), int rows = PersistCfg<SPLIT, GU>::kRows) {
  using C = PersistCfg<SPLIT, GU>;
  constexpr size_t smem = C::kSmemBytes;
  static OncePerDevice configured;
  const cudaError_t set = allow_smem(configured, gemm_tc_persistent_kernel<GU, SPLIT>, smem);
  if (set != cudaSuccess) return set;
  const int n_sm = sm_count();
  if (n_sm <= 0) return cudaErrorInvalidDevice;
  const int tiles_n = GU ? N / 64 : (N + kTileN - 1) / kTileN, tiles_m = (M + rows - 1) / rows;
  const int grid = std::min(tiles_n * tiles_m, n_sm);
  RSD_LAUNCH((gemm_tc_persistent_kernel<GU, SPLIT>), grid, kPersistThreads, smem, s, tw, tx, txl, y, M, N, K, accumulate, tiles_n,
             tiles_m, err, act_hi, act_lo, f16, n_active, rs, rows);
  return launched(1);
}

template <bool GU, bool SPLIT>
static cudaError_t configure_pair() {
  static OncePerDevice configured;
  return allow_smem(configured, gemm_tc_pair_kernel<GU, SPLIT>, PairCfg<SPLIT, GU>::kSmemBytes);
}

// Pairs of CTAs that fit the device at once.
template <bool GU, bool SPLIT>
static int query_pairs() {
  if (configure_pair<GU, SPLIT>() != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2048); cfg.blockDim = dim3(kPersistThreads); cfg.dynamicSmemBytes = PairCfg<SPLIT, GU>::kSmemBytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, gemm_tc_pair_kernel<GU, SPLIT>, &cfg) == cudaSuccess ? n : 0;
}
template <bool GU, bool SPLIT>
static int max_pairs() {
  static const int pairs = query_pairs<GU, SPLIT>();
  return pairs;
}

// The map of x has a box of half the tile's operand rows.
template <bool GU, bool SPLIT>
static cudaError_t launch_pair(const CUtensorMap& tw, const CUtensorMap& tx, const CUtensorMap& txl, float* y, int M, int N, int K,
                               int accumulate, int* err, __nv_bfloat16* act_hi, __nv_bfloat16* act_lo, cudaStream_t s, int f16, int rows) {
  constexpr size_t smem = PairCfg<SPLIT, GU>::kSmemBytes;
  const cudaError_t set = configure_pair<GU, SPLIT>();
  if (set != cudaSuccess) return set;
  const int pairs = max_pairs<GU, SPLIT>();
  if (pairs <= 0) return cudaErrorNotSupported;
  const int feat = GU ? kTileN : 2 * kTileN, tiles_n = (N + feat - 1) / feat, tiles_m = (M + rows - 1) / rows;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * std::min(tiles_n * tiles_m, pairs)); cfg.blockDim = dim3(kPersistThreads); cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_tc_pair_kernel<GU, SPLIT>, tw, tx, txl, y, M, N, K, accumulate, tiles_n, tiles_m,
                                           err, act_hi, act_lo, f16, rows);
  return e != cudaSuccess ? e : launched(1);
}

// Whether a dense product goes to pairs of CTAs: it has as many pair tiles as the chip has pairs, and where it adds into y a K
// long enough for the main loop to matter beside the epilogues.  Lone CTAs / pairs, us: 8192 x 3584 x 18944 857 / 817,
// 8192 x 1536 x 8960 182 / 158, 8192 x 2048 x 1536 55 / 51, gate/up 1000 x 18944 x 3584 226 / 193, 8192 x 18944 x 3584
// 1636 / 1501; adding, 4096 x 1536 x 1536 41 / 43.  (The paired gate/up tile of hi + lo operands gains nothing, 3180 / 3160
// at 8192 x 18944 x 3584, and keeps the lone CTAs.)
static bool pair_pays(int M, int n_features, int K, int feat, int rows, bool adds) {
  return K >= (adds ? 3072 : 1024) && ((n_features + feat - 1) / feat) * ((M + rows - 1) / rows) >= 74;
}

// x rows of a tile for plain operands in the persistent kernels: 256, or fewer where the waves then cost less.  A smaller tile costs
// more per row (the weight half of a stage is read as often): kCost, in 256-row units, fitted to 8192 x 18944 x 3584 (gate/up, full waves:
// 1387 / 1460 / 1583 / 1826 us with 256 / 224 / 192 / 160 rows; 128 rows, 2355, never pay).  Where the last wave of 256-row tiles is
// nearly empty (4096 x 3584: 224 tiles on 74 pairs of SMs) fewer rows win; us at 256 / 224 / 192 / 160: 4096 x 3584 x 18944 576 / 506 / 545 / 509,
// 1300 x 3584 x 18944 260 / 229 / 204 / 192, 4096 x 1536 x 8960 140 / 125 / 113 / 144, 8192 x 1536 x 1536 (lone CTAs) 55.8 / 50.8 / 55.8 / 57.9,
// 1300 x 4608 x 3584 55 / 50 / 45 / 54; and 4096 x 2048 x 1536, two full waves, stays at 256 (29.5 / 35.0 / 32.1 / 29.5).
// slots: the pairs of CTAs, or CTAs, that the launch has at once.
static int wave_rows(int M, int n_tiles, int slots) {
  slots = std::max(slots, 1);              // (none: the launch reports it)
  constexpr int kRows[4] = {256, 224, 192, 160}, kCost[4] = {256, 233, 217, 206};
  int best = 0;
  long cost = 0;
  for (int i = 0; i < 4; ++i) {
    const long c = (((long)n_tiles * ((M + kRows[i] - 1) / kRows[i]) + slots - 1) / slots) * kCost[i];
    if (i == 0 || c < cost) { best = i; cost = c; }
  }
  return kRows[best];
}
static int pair_tiles(int n_features, int feat) { return (n_features + feat - 1) / feat; }

// Rows of x per tile for a dense product with one operand (bf16 or fp16): 256, or 128 or 64 while the tiles of the larger
// size leave half of the SMs (of 256) or some (of 128) without one.  Every size sums along K in the same order: the
// results are the same bits.  us with 256 / 128 / 64 rows, adding into y (fp16, graph replays, operands in L2): 455 x 2048 x 1536
// 18.7 / 11.1 / 9.1, 1000 x 1536 x 1536 18.8 / 11.5 / 11.8, 1000 x 3584 x 3584, 112 tiles of 256, 30.3 / 29.9 / 39.5.  Adding at a short K
// the epilogue is most of a tile and one wave of 256-row tiles hides none of it, while two CTAs of 128 rows hide each other's:
// 2048 x 1536 x 1536, 96 tiles, 19.8 / 17.0 / 19.6; 3000 x 1536 x 1536, 144 tiles, 20.0 / 17.4 / 23.4; from two waves on the
// persistent kernel does as well or better (4096 x 1536 x 1536 30.2 / 28.9 / 33.1, 8192 x 1536 x 1536 47.4 / 52.2 / 66.6).
static int dense_rows(int M, int N, int K, bool adds) {
  const int n_tiles = (N + kTileN - 1) / kTileN;
  int rows = 256;
  while (rows > 64 && n_tiles * ((M + rows - 1) / rows) < (rows == 256 && !(adds && K < 3072) ? 74 : 148)) rows /= 2;
  return rows;
}

// ... one tile per CTA; with at most one CTA per SM the deep ring (a lone CTA is bound by the latency of its stages).
static cudaError_t launch_dense_small(const CUtensorMap& tw, const CUtensorMap& tx, float* y, int M, int N, int K, int accumulate,
                                      int rows, int* err, cudaStream_t s, int f16) {
  TcPlan p;
  p.rows = p.mt = rows;
  p.n_tiles = (N + kTileN - 1) / kTileN;
  p.m_tiles = (M + rows - 1) / rows;
  p.splits = 1;
  p.kb_per_split = (K + kTileK - 1) / kTileK;
  const bool deep = p.n_tiles * p.m_tiles <= 148;
#define RSD_DENSE(MT, DEEP) return launch_mt<MT, false, DEEP>(tw, tx, tx, y, M, N, K, accumulate, p, nullptr, err, nullptr, false, RowScale(), s, f16)
  if (rows == 64) { if (deep) RSD_DENSE(64, true); RSD_DENSE(64, false); }
  if (deep) RSD_DENSE(128, true);
  RSD_DENSE(128, false);
#undef RSD_DENSE
}

// 65 to 128 rows with pairs take an SM per tile: with more tiles than SMs the persistent kernel hides the epilogues and
// evens out the last wave (the 1187 tiles of a 151936-row head at 128 rows: 140 us one CTA per tile, 93 us persistent).
static bool wide_decode(int M, int n_tiles) { return M > 64 && M <= 128 && n_tiles > 148; }

template <int MT, bool DEEP>
static cudaError_t launch_gu_mt(const CUtensorMap& tw, const CUtensorMap& tx, const CUtensorMap& txl, int M, int F, int K, int rows,
                                int* err, const int32_t* n_active, RowScale rs, __nv_bfloat16* act_hi, __nv_bfloat16* act_lo,
                                cudaStream_t s) {
  static OncePerDevice configured;
  const cudaError_t set = allow_smem(configured, gemm_tc_kernel<MT, true, true, DEEP>, TcCfg<MT, DEEP>::kSmemBytes);
  if (set != cudaSuccess) return set;
  const int total_kb = (K + kTileK - 1) / kTileK;
  const int stages = MT <= 32 ? std::min(TcCfg<MT, DEEP>::kStages, kGuStages) : TcCfg<MT, DEEP>::kStages;
  const size_t smem = TcCfg<MT, DEEP>::smem_bytes(stages);
  dim3 grid(F / 64, (M + rows - 1) / rows, 1);
  RSD_LAUNCH((gemm_tc_kernel<MT, true, true, DEEP>), grid, kTcThreads, smem, s, tw, tx, txl, (float*)nullptr, M, F, K, 0, 1, total_kb,
             (float*)nullptr, err, n_active, rs, stages, act_hi, act_lo, 0);
  return launched(1);
}

bool gemm_gu_supported(int dtype, int M, int F, int K) {
  return dtype == 1 && M >= 1 && F >= 64 && F % 64 == 0 && K >= 8 && K % 8 == 0;
}

// act (hi + lo, bf16 [M, F]) = silu(g) * u with [g | u] = rowscale * (x_hi + x_lo)[M, K] * Wgu[2F, K]^T.
cudaError_t launch_gemm_gu(const void* Wgu, const void* x, const void* x_lo, void* act_hi, void* act_lo, int M, int F, int K,
                           void* scratch, size_t scratch_bytes, const int32_t* n_active, cudaStream_t s, RowScale rs) {
  if (M <= 0) return cudaSuccess;
  if (!gemm_gu_supported(1, M, F, K) || !act_hi) return cudaErrorNotSupported;
  if (!scratch || scratch_bytes < (size_t)kCounterBytes + 256) return cudaErrorInvalidValue;
  if (((uintptr_t)Wgu & 15) || ((uintptr_t)x & 15) || ((uintptr_t)x_lo & 15)) return cudaErrorMisalignedAddress;
  int* err = (int*)((char*)scratch + kCounterBytes);
  CUtensorMap tw, tx, txl;
  if (x_lo == nullptr) {
    // plain bf16 operand: the persistent kernel only (more than 128 rows, no row scale, no idle flag)
    if (!(M > 128 && rs.ssq == nullptr && n_active == nullptr)) return cudaErrorNotSupported;
    const bool pair = pair_pays(M, F, K, kTileN, 256, false);
    const int tile_rows = pair ? wave_rows(M, pair_tiles(F, kTileN), max_pairs<true, false>()) : wave_rows(M, F / 64, sm_count());
    if (!get_map(Wgu, 2 * F, K, kTileN / 2, &tw) || !get_map(x, M, K, pair ? tile_rows / 2 : tile_rows, &tx)) return cudaErrorNotSupported;
    if (pair) return launch_pair<true, false>(tw, tx, tx, nullptr, M, F, K, 0, err, (__nv_bfloat16*)act_hi, nullptr, s, 0, tile_rows);
    return launch_persistent<true, false>(tw, tx, tx, nullptr, M, F, K, 0, err, (__nv_bfloat16*)act_hi, nullptr, s, 0, nullptr, RowScale(), tile_rows);
  }
  if (!act_lo) return cudaErrorNotSupported;
  // each warp pair finishes one half of the rows, up to 16 at a time
  const int rows = M <= 8 ? 8 : (M <= 16 ? 16 : (M <= 32 ? 32 : (M <= 64 ? 64 : 128)));
  if (rs.ssq != nullptr && rows > 128) return cudaErrorInvalidValue;
  if (!get_map(Wgu, 2 * F, K, kTileN / 2, &tw) || !get_map(x, M, K, rows, &tx) || !get_map(x_lo, M, K, rows, &txl))
    return cudaErrorNotSupported;
  if (M > 128 && rs.ssq == nullptr && n_active == nullptr)
    return launch_persistent<true, true>(tw, tx, txl, nullptr, M, F, K, 0, err, (__nv_bfloat16*)act_hi, (__nv_bfloat16*)act_lo, s);
  auto* hi = (__nv_bfloat16*)act_hi;
  auto* lo = (__nv_bfloat16*)act_lo;
  if (wide_decode(M, F / 64)) return launch_persistent<true, true>(tw, tx, txl, nullptr, M, F, K, 0, err, hi, lo, s, 0, n_active, rs);
  // fewer than ~1.5 CTAs per SM: one CTA per SM with a deep ring streams faster than a thin second wave
  const bool deep = (F / 64) * ((M + rows - 1) / rows) <= 222;
  switch (rows) {
    case 8: return deep ? launch_gu_mt<16, true>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s)
                        : launch_gu_mt<16, false>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s);
    case 16: return deep ? launch_gu_mt<32, true>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s)
                         : launch_gu_mt<32, false>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s);
    case 32: return deep ? launch_gu_mt<64, true>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s)
                         : launch_gu_mt<64, false>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s);
    case 64: return deep ? launch_gu_mt<128, true>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s)
                         : launch_gu_mt<128, false>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s);
    default: return launch_gu_mt<256, false>(tw, tx, txl, M, F, K, rows, err, n_active, rs, hi, lo, s);
  }
}

// Layout of the scratch: [0, 4096) tile counters (kept zero between launches), then one int error
// flag region of 256 bytes, then split-K partial tiles.
size_t gemm_scratch_bytes(int M) {
  const int rows = pick_rows(M, false);
  const size_t part = rows <= 128 ? (size_t)kMaxSplitCtas * kTileN * std::min(64, std::max(rows, 16)) * 4 : 0;
  return kCounterBytes + 256 + part;
}

// Enough for any M (split-K is only used with up to 128 rows of x, and beyond 64 with half as many CTAs).
size_t gemm_scratch_bytes_any() { return gemm_scratch_bytes(64); }

const float* gemm_partials(const void* scratch) { return (const float*)((const char*)scratch + kCounterBytes + 256); }

cudaError_t launch_gemm_tc(const void* W, const void* x, const void* x_lo, float* y, int M, int N, int K, int accumulate,
                           void* scratch, size_t scratch_bytes, const int32_t* n_active, int* deferred_splits,
                           cudaStream_t s, RowScale rs, bool no_k_split) {
  if (deferred_splits) *deferred_splits = 1;
  if (M <= 0) return cudaSuccess;
  if (rs.ssq != nullptr && accumulate) return cudaErrorInvalidValue;
  if (!scratch || scratch_bytes < gemm_scratch_bytes(M)) return cudaErrorInvalidValue;
  if (((uintptr_t)W & 15) || ((uintptr_t)x & 15) || ((uintptr_t)x_lo & 15)) return cudaErrorMisalignedAddress;
  const bool split_operand = x_lo != nullptr;
  TcPlan p = plan_tc(M, N, K, split_operand);
  if (no_k_split) { p.splits = 1; p.kb_per_split = (K + kTileK - 1) / kTileK; }
  if (rs.ssq != nullptr && p.rows > 128) return cudaErrorInvalidValue;   // one epilogue thread per x row of the tile
  if (deferred_splits) *deferred_splits = p.splits;
  const bool defer = deferred_splits != nullptr;
  CUtensorMap tw, tx, txl;
  const bool dense = M > 128 && p.splits == 1 && rs.ssq == nullptr && n_active == nullptr;
  const bool pair = dense && pair_pays(M, N, K, 2 * kTileN, p.rows, accumulate != 0);
  int rows = dense && !split_operand && !pair && !no_k_split ? dense_rows(M, N, K, accumulate != 0) : p.rows;
  const bool small = dense && !pair && !split_operand && rows < 256;
  if (dense && !split_operand && !small) rows = pair ? wave_rows(M, pair_tiles(N, 2 * kTileN), max_pairs<false, false>()) : wave_rows(M, p.n_tiles, sm_count());
  if (!get_map(W, N, K, kTileN, &tw) || !get_map(x, M, K, pair ? (split_operand ? 128 : rows / 2) : rows, &tx)) return cudaErrorNotSupported;
  if (split_operand) { if (!get_map(x_lo, M, K, p.rows, &txl)) return cudaErrorNotSupported; }
  else txl = tx;
  int* err = (int*)((char*)scratch + kCounterBytes);
  float* partials = (float*)((char*)scratch + kCounterBytes + 256);
  if (dense) {
    if (pair && split_operand) return launch_pair<false, true>(tw, tx, txl, y, M, N, K, accumulate, err, nullptr, nullptr, s, 0, p.rows);
    if (pair) return launch_pair<false, false>(tw, tx, txl, y, M, N, K, accumulate, err, nullptr, nullptr, s, 0, rows);
    if (small) return launch_dense_small(tw, tx, y, M, N, K, accumulate, rows, err, s, 0);
    if (split_operand) return launch_persistent<false, true>(tw, tx, txl, y, M, N, K, accumulate, err, nullptr, nullptr, s);
    return launch_persistent<false, false>(tw, tx, txl, y, M, N, K, accumulate, err, nullptr, nullptr, s, 0, nullptr, RowScale(), rows);
  }
  if (split_operand && p.splits == 1 && wide_decode(M, p.n_tiles))
    return launch_persistent<false, true>(tw, tx, txl, y, M, N, K, accumulate, err, nullptr, nullptr, s, 0, n_active, rs);
#define RSD_TC(MT, SP) return launch_mt<MT, SP>(tw, tx, txl, y, M, N, K, accumulate, p, partials, err, n_active, defer, rs, s)
  // a grid of at most one CTA per SM: the deep ring (a lone CTA needs more bytes in flight to keep its stream going)
  if (split_operand && p.n_tiles * p.m_tiles * p.splits <= 148 && p.mt <= 128) {
#define RSD_TCD(MT) return launch_mt<MT, true, true>(tw, tx, txl, y, M, N, K, accumulate, p, partials, err, n_active, defer, rs, s)
    switch (p.mt) {
      case 16: RSD_TCD(16);
      case 32: RSD_TCD(32);
      case 64: RSD_TCD(64);
      default: RSD_TCD(128);
    }
#undef RSD_TCD
  }
  if (split_operand) {
    switch (p.mt) {
      case 16: RSD_TC(16, true);
      case 32: RSD_TC(32, true);
      case 64: RSD_TC(64, true);
      case 128: RSD_TC(128, true);
      default: RSD_TC(256, true);
    }
  }
  switch (p.mt) {
    case 16: RSD_TC(16, false);
    case 32: RSD_TC(32, false);
    case 64: RSD_TC(64, false);
    case 128: RSD_TC(128, false);
    default: RSD_TC(256, false);
  }
#undef RSD_TC
}

// Dense products (more than 128 rows) with fp16 weights and ONE fp16 activation operand: the persistent kernel with
// the operand formats switched.  y [M, N] fp32 (+)= x [M, K] W [N, K]^T.
cudaError_t launch_gemm_f16_dense(const void* W16, const void* x16, float* y, int M, int N, int K, int accumulate,
                                  void* scratch, size_t scratch_bytes, cudaStream_t s) {
  if (M <= 128 || !gemm_tc_supported(1, M, N, K)) return cudaErrorNotSupported;
  if (!scratch || scratch_bytes < gemm_scratch_bytes(M)) return cudaErrorInvalidValue;
  if (((uintptr_t)W16 & 15) || ((uintptr_t)x16 & 15)) return cudaErrorMisalignedAddress;
  const bool pair = pair_pays(M, N, K, 2 * kTileN, 256, accumulate != 0);
  CUtensorMap tw, tx;
  int rows = pair ? 256 : dense_rows(M, N, K, accumulate != 0);
  const bool small = rows < 256;
  if (!small) rows = pair ? wave_rows(M, pair_tiles(N, 2 * kTileN), max_pairs<false, false>()) : wave_rows(M, (N + kTileN - 1) / kTileN, sm_count());
  if (!get_map(W16, N, K, kTileN, &tw) || !get_map(x16, M, K, pair ? rows / 2 : rows, &tx)) return cudaErrorNotSupported;
  int* err = (int*)((char*)scratch + kCounterBytes);
  if (small) return launch_dense_small(tw, tx, y, M, N, K, accumulate, rows, err, s, 1);
  if (pair) return launch_pair<false, false>(tw, tx, tx, y, M, N, K, accumulate, err, nullptr, nullptr, s, 1, rows);
  return launch_persistent<false, false>(tw, tx, tx, y, M, N, K, accumulate, err, nullptr, nullptr, s, 1, nullptr, RowScale(), rows);
}

// act [M, F] fp16 = silu(g) * u with [g | u] = x [M, K] Wgu [2F, K]^T, fp16 operands, more than 128 rows.
cudaError_t launch_gemm_gu_f16_dense(const void* Wgu16, const void* x16, void* act16, int M, int F, int K, void* scratch,
                                     size_t scratch_bytes, cudaStream_t s) {
  if (M <= 128 || !gemm_gu_supported(1, M, F, K) || !act16) return cudaErrorNotSupported;
  if (!scratch || scratch_bytes < (size_t)kCounterBytes + 256) return cudaErrorInvalidValue;
  if (((uintptr_t)Wgu16 & 15) || ((uintptr_t)x16 & 15)) return cudaErrorMisalignedAddress;
  int* err = (int*)((char*)scratch + kCounterBytes);
  CUtensorMap tw, tx;
  const bool pair = pair_pays(M, F, K, kTileN, 256, false);
  const int rows = pair ? wave_rows(M, pair_tiles(F, kTileN), max_pairs<true, false>()) : wave_rows(M, F / 64, sm_count());
  if (!get_map(Wgu16, 2 * F, K, kTileN / 2, &tw) || !get_map(x16, M, K, pair ? rows / 2 : rows, &tx)) return cudaErrorNotSupported;
  if (pair) return launch_pair<true, false>(tw, tx, tx, nullptr, M, F, K, 0, err, (__nv_bfloat16*)act16, nullptr, s, 1, rows);
  return launch_persistent<true, false>(tw, tx, tx, nullptr, M, F, K, 0, err, (__nv_bfloat16*)act16, nullptr, s, 1, nullptr, RowScale(), rows);
}

cudaError_t launch_gemm(int dtype, const void* W, const void* x, const void* x_lo, float* y, int M, int N, int K,
                        int accumulate, int impl, void* scratch, size_t scratch_bytes, const int32_t* n_active,
                        int* deferred_splits, cudaStream_t s, RowScale rs) {
  if (deferred_splits) *deferred_splits = 1;
  const bool tc_ok = gemm_tc_supported(dtype, M, N, K) && scratch && scratch_bytes >= gemm_scratch_bytes(M);
  // the tensor-core path wins for every M (an M = 1 GEMV included: TMA streaming beats the SIMT loads)
  if (impl == 2 || impl == 3 || (impl == 0 && tc_ok))
    return launch_gemm_tc(W, x, x_lo, y, M, N, K, accumulate, scratch, scratch_bytes, n_active, deferred_splits, s, rs, impl == 3);
  if (rs.ssq != nullptr) return cudaErrorNotSupported;
  return launch_gemm_simt(dtype, W, x, dtype == 1 ? x_lo : nullptr, y, M, N, K, accumulate, n_active, s);
}

}  // namespace rsd
