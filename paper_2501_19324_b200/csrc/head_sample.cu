// The lm head of a decode pass with the sampling in its epilogue (bf16 weights x hi + lo operand pairs, up to 128 rows): the best id of every slot
// comes out, the logits stay in tensor memory.
//
// As two launches the head was one tile of 128 ids a CTA and the sampling read the logits back: in the step loop 151936 ids of 3584 columns took
// 154-201 us at 8 to 64 rows for a weight stream of 149, of 1536 columns 67-115 at 8 to 128 for 64, and the sampling 11 us at 20 rows, 15-19 at 32 to
// 40, 48 at 128.  Here both take 168-185 us at 16 to 64 rows, and 71 at 16, 80 at 40, 128 at 128.
//   - 1187 tiles are 8.02 for each of 148 SMs (4.01 rounds of two): the last round is nearly empty.  Here a CTA per SM walks the same number
//     of whole tiles as every other and then one smaller tile, whose rows are the remainder shared out by sixteens.
//   - Two tiles of 128 ids are multiplied at once with the same x tile (up to 64 rows): from 16 rows on the copies of x are what the head waits for,
//     64 rows of 3584 columns are 0.92 MB a tile, as many bytes in all as the weights.
//   - The ring runs on from tile to tile and the accumulators alternate, so the sampling of a tile runs beside the products of the next.
// The ids are sample_kernel's: ids whose logits cannot win against the best so far draw no noise, the others a quick one first, and only
// what comes near the best an exact one.  A thread holds one id of sixteen rows; the four words of a Philox block belong to four neighbouring
// ids, so four lanes take a block each of four rows and swap words.
// What bounds it: the weights up to 64 rows; at 128 the copies of x (a tile at a time, 0.79 MB each of 1536 columns) and the noise beside them.
// Roles: warps 0-7 epilogue, 8 weights, 9 MMAs, 10 x.  Every wait is bounded, as in gemm_tc.cu.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "sampling.cuh"
#include "tc_ptx.cuh"

namespace rsd {

namespace {

using namespace tc;

constexpr int kTile = 128, kTileK = 64, kUmmaK = 16, kPiece = 16;      // ids of an instruction; of the smallest copy
constexpr int kEpiWarps = 8, kThreads = 32 * (kEpiWarps + 3);

// MT: columns of an instruction, the slots' hi rows and then their lo rows.
template <int MT> struct HeadCfg {
  static constexpr int kRows = MT / 2;
  static constexpr int kWide = MT <= 128 ? 2 : 1;                      // tiles of 128 ids at once: two accumulators of them fit tensor memory
  static constexpr int kIds = kWide * kTile;
  static constexpr int kABytes = kIds * kTileK * 2, kBBytes = MT * kTileK * 2, kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = MT <= 32 ? 6 : (MT == 64 ? 5 : 4);
  static constexpr int kAccCols = kWide * MT, kTmemCols = 2 * kAccCols;
  static constexpr size_t kSmemBytes = 1024 + (size_t)kStages * kStageBytes + 256;
  static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(MT >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
  static_assert(kSmemBytes + 3584 <= 227 * 1024 && kTmemCols <= 512 && kTmemCols >= 32, "what an SM has");
};

// What CTA `b` of `g` walks: `whole` tiles of `ids` ids, and the rows that do not fill a round of them in pieces of `rest` ids a CTA.
struct Walk {
  int ids, whole, first_rest, rest, n;
  __device__ __forceinline__ Walk(int n_ids, int ids_, int g, int b) : ids(ids_) {
    whole = n_ids / (ids * g);
    first_rest = whole * ids * g;
    const int left = n_ids - first_rest;
    rest = ((left + g - 1) / g + kPiece - 1) / kPiece * kPiece;
    n = whole + (first_rest + b * rest < n_ids ? 1 : 0);
  }
  __device__ __forceinline__ int row(int t, int g, int b) const { return t < whole ? (t * g + b) * ids : first_rest + b * rest; }
  __device__ __forceinline__ int height(int t) const { return t < whole ? ids : rest; }
};

// v[s] = v[q ^ s]
template <typename T> __device__ __forceinline__ void by_lane(T (&v)[4], int q) {
  const T a = (q & 1) ? v[1] : v[0], b = (q & 1) ? v[0] : v[1], c = (q & 1) ? v[3] : v[2], d = (q & 1) ? v[2] : v[3];
  v[0] = (q & 2) ? c : a; v[1] = (q & 2) ? d : b; v[2] = (q & 2) ? a : c; v[3] = (q & 2) ? b : d;
}
__device__ __forceinline__ float pick(const float (&v)[4], int i) { return (i & 2) ? ((i & 1) ? v[3] : v[2]) : ((i & 1) ? v[1] : v[0]); }

template <int MT>
__global__ void __launch_bounds__(kThreads, 1)
head_sample_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_piece, const __grid_constant__ CUtensorMap tm_x,
                   const __grid_constant__ CUtensorMap tm_x_lo, int N, int K, int* err, RowScale rs, const __grid_constant__ SampleArgs a) {
  RSD_PDL_TRIGGER();
  using C = HeadCfg<MT>;
  if (a.n_active != nullptr && ld_cg(a.n_active) == 0) {
    RSD_PDL_WAIT();
    return;
  }
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + (size_t)C::kStages * C::kStageBytes);
  uint64_t* empty = full + C::kStages;
  uint64_t* acc_full = empty + C::kStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  volatile uint32_t* stop = tmem_slot + 1;
  __shared__ float s_scale[C::kRows];
  __shared__ volatile float s_run[C::kRows];   // best exact score of a row that this CTA knows of; NaN for a slot without a row
  __shared__ unsigned long long s_best[C::kRows];    // packed, of this CTA
  __shared__ int s_row[C::kRows], s_pos[C::kRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, M = a.n_slots;
  const int n_kb = (K + kTileK - 1) / kTileK, g = gridDim.x, b = blockIdx.x;
  const Walk walk(N, C::kIds, g, b);
  if (threadIdx.x == 32 * kEpiWarps) {
    for (int s = 0; s < C::kStages; ++s) { mbar_init(&full[s], 2); mbar_init(&empty[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], kEpiWarps); }
    *stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (threadIdx.x == 32 * (kEpiWarps + 2)) {
    tma_prefetch_map(&tm_x);
    tma_prefetch_map(&tm_x_lo);
  }
  if (warp == kEpiWarps + 1) tmem_alloc(tmem_slot, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  auto fail = [&]() { if (*stop == 0) { if (err) atomicCAS(err, 0, -5); *stop = 1; } };

  if (warp == kEpiWarps || warp == kEpiWarps + 2) {
    // ---------------- producers: weights ahead of the wait as far as the ring reaches, x behind it ----------------
    if (lane == 0) {
      const bool weights = warp == kEpiWarps;
      if (!weights) RSD_PDL_WAIT();
      int issued = 0, s = 0;
      uint32_t phase = 1;
      bool ok = true, ready = true;
      for (int t = 0; t < walk.n && ok; ++t) {
        const int row = walk.row(t, g, b), height = walk.height(t);
        for (int kb = 0; kb < n_kb; ++kb) {
          if (!ready && (!mbar_wait(&empty[s], phase) || *stop)) { ok = false; break; }
          uint8_t* dst = smem + (size_t)s * C::kStageBytes;
          if (weights) {
            mbar_expect_tx(&full[s], height * kTileK * 2);
            int r = 0;
            for (; r + kTile <= height; r += kTile) tma_load_2d(dst + r * kTileK * 2, &tm_w, &full[s], kb * kTileK, row + r);
            for (; r < height; r += kPiece) tma_load_2d(dst + r * kTileK * 2, &tm_piece, &full[s], kb * kTileK, row + r);
          } else {
            mbar_expect_tx(&full[s], C::kBBytes);
            tma_load_2d(dst + C::kABytes, &tm_x, &full[s], kb * kTileK, 0);
            tma_load_2d(dst + C::kABytes + C::kRows * kTileK * 2, &tm_x_lo, &full[s], kb * kTileK, 0);
          }
          ++issued;
          if (++s == C::kStages) { s = 0; phase ^= 1u; }
          ready = mbar_test(&empty[s], phase);
        }
      }
      if (!ok) {
        fail();
        for (int i = max(0, issued - C::kStages); i < issued; ++i) mbar_wait(&full[i % C::kStages], (i / C::kStages) & 1, 1u << 16);
      }
    }
  } else if (warp == kEpiWarps + 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t on = elect_one();
    int s = 0;
    uint32_t phase = 0;
    bool ok = true, ready = false;
    for (int t = 0; t < walk.n && ok; ++t) {
      const uint32_t buf = t & 1;
      ok = mbar_wait(&acc_empty[buf], ((t >> 1) & 1) ^ 1u);
      ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d0 = tmem_base + buf * C::kAccCols;
      const bool both = C::kWide == 2 && walk.height(t) > kTile;
      for (int kb = 0; kb < n_kb; ++kb) {
        if (!ready) {
          ok = mbar_wait(&full[s], phase);
          ok = __all_sync(0xFFFFFFFFu, ok && !*stop);
          if (!ok) break;
        }
        tc_fence_after();
        const int s1 = s + 1 == C::kStages ? 0 : s + 1;
        const uint32_t phase1 = s1 == 0 ? phase ^ 1u : phase;
        ready = __all_sync(0xFFFFFFFFu, mbar_test(&full[s1], phase1));       // under this stage's MMAs
        const uint32_t at = smem_u32(smem + (size_t)s * C::kStageBytes), bt = at + C::kABytes;
#pragma unroll
        for (int k = 0; k < kTileK / kUmmaK; ++k) {
          const uint64_t bd = smem_desc_sw128(bt + k * kUmmaK * 2);
          const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
          umma_bf16_if(on, d0, smem_desc_sw128(at + k * kUmmaK * 2), bd, C::kIdesc, acc);
          if (both) umma_bf16_if(on, d0 + MT, smem_desc_sw128(at + kTile * kTileK * 2 + k * kUmmaK * 2), bd, C::kIdesc, acc);
        }
        umma_commit_if(on, &empty[s]);
        s = s1;
        phase = phase1;
      }
      if (ok) umma_commit_if(on, &acc_full[buf]);
    }
    if (!ok && on) fail();
  } else {
    // ---------------- epilogue ----------------
    constexpr int kEpiThreads = 32 * kEpiWarps;
    RSD_PDL_WAIT();
    if (threadIdx.x < C::kRows) {
      const int row = threadIdx.x < M ? ld_cg(a.slot_row + threadIdx.x) : -1;
      s_row[threadIdx.x] = row;
      s_best[threadIdx.x] = 0ull;
      s_pos[threadIdx.x] = row >= 0 ? ld_cg(a.slot_pos + threadIdx.x) + 1 : 0;
      s_run[threadIdx.x] = row >= 0 ? -INFINITY : __int_as_float(0x7FC00000);
    }
    {
      // RMSNorm's denominators, as in gemm_tc_kernel
      constexpr int kLanes = kEpiThreads / C::kRows < 32 ? kEpiThreads / C::kRows : 32;
      const int r = threadIdx.x / kLanes, sub = threadIdx.x % kLanes;
      float sum = 0.f;
      if (r < M && rs.ssq != nullptr) {
        const float* src = rs.ssq + (size_t)r * rs.n_chunks;
#pragma unroll 8
        for (int c = sub; c < rs.n_chunks; c += kLanes) sum += src[c];
      }
#pragma unroll
      for (int o = kLanes / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
      if (sub == 0 && r < C::kRows) s_scale[r] = rs.ssq != nullptr ? rsqrtf(sum * rs.inv_d + rs.eps) : 1.f;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
    const bool noisy = a.temperature > 0.f;
    const float inv_t = noisy ? 1.f / a.temperature : 1.f;
    const uint2 key = make_uint2((uint32_t)(a.seed & 0xFFFFFFFFull), (uint32_t)(a.seed >> 32));
    const int quarter = warp & 3, half = warp >> 2, q = lane & 3;
    constexpr int kCols = C::kRows < 16 ? C::kRows : 16;
    // An exact score.  The warps of the CTA meet in shared memory; what they have found goes out between tiles (an atomic with an answer for every
    // candidate of the first tile took as long as the weights).
    auto offer = [&](int r, float score, int id) {
      atomicMax(&s_best[r], pack_best(score, id));
      if (!(s_run[r] >= score)) s_run[r] = score;  // (of several at once any may stay: each is a score that the row's best has reached)
    };
    // sixteen rows (or eight) from c on of the 128 ids whose accumulators begin at `acc`; id: this thread's, in the race if `in`
    auto sample = [&](uint32_t acc, int c, int id, bool in) {
      float v[kCols];
      if (C::kRows == 8) {
        float w[16];
        tmem_ld16(acc, w);
#pragma unroll
        for (int j = 0; j < kCols; ++j) v[j] = w[j] + w[(j + 8) & 15];
      } else {
        float w[2][16];
        tmem_ld16n<2>({acc + c, acc + C::kRows + c}, w);
#pragma unroll
        for (int j = 0; j < kCols; ++j) v[j] = w[0][j & 15] + w[1][j & 15];
      }
#pragma unroll
      for (int j = 0; j < kCols; ++j) v[j] = in ? v[j] * s_scale[c + j] : __int_as_float(0x7FC00000);   // NaN: never wins a comparison
      if (!noisy) {
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
          const float run = s_run[c + j];
          if (!__any_sync(0xFFFFFFFFu, v[j] >= run)) continue;         // (equal: the lower id wins)
          const uint32_t mine = v[j] == v[j] ? score_key(v[j]) : 0u, top = __reduce_max_sync(0xFFFFFFFFu, mine);
          const unsigned who = __ballot_sync(0xFFFFFFFFu, mine == top);
          if (top != 0u && lane == __ffs(who) - 1) offer(c + j, v[j], id);
        }
        return;
      }
#pragma unroll
      for (int i = 0; i < kCols; i += 4) {
        if (c + i >= M) break;
        // step s of four: row c + i + (q ^ s), for which lane q ^ s of the four holds the block with this lane's word
        // need: what a quick score has to reach.  Like sample_kernel's it leaves room for an ulp of the exact score, which is what decides: of two ids that
        // round to the same score the lower one wins, whichever was found first
        float lg[4] = {v[i], v[i + 1], v[i + 2], v[i + 3]}, need[4], u[4];
        by_lane(lg, q);
        bool near = false, first = false;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float run = s_run[c + i + (q ^ s)];
          need[s] = score_needed(run);
          near = near || lg[s] * inv_t >= need[s] - kNoiseMax || run == -INFINITY;
          first = first || fabsf(run) == INFINITY;
        }
        if (!__any_sync(0xFFFFFFFFu, near)) continue;
        const uint4 ph = philox4x32_10(make_uint4((uint32_t)id / 4u, (uint32_t)s_pos[c + i + q], (uint32_t)s_row[c + i + q], (uint32_t)a.model_id), key);
        uint32_t word[4] = {ph.x, ph.y, ph.z, ph.w};
        by_lane(word, q);
#pragma unroll
        for (int s = 0; s < 4; ++s) u[s] = uniform_from_bits(__shfl_xor_sync(0xFFFFFFFFu, word[s], s));
        unsigned may = 0;
        if (!__any_sync(0xFFFFFFFFu, first)) {
          // -log(-log u) + x >= need  <=>  u >= exp(-exp(x - need)).  __expf errs by 2 + 1.173 |argument| ulp, and beyond 17 either way no u
          // decides: 2.6e-6 of the bound, which the factor covers, and as much of the inner exponential, which is a shift of the score by 2.6e-6: need has 1e-3 of room
#pragma unroll
          for (int s = 0; s < 4; ++s)
            may |= u[s] >= __expf(-__expf(fmaf(lg[s], inv_t, -need[s]))) * (1.f - 4e-6f) ? 1u << s : 0u;
        } else {
          float sc[4], top[4];
#pragma unroll
          for (int s = 0; s < 4; ++s) top[s] = sc[s] = fmaf(lg[s], inv_t, fast_gumbel(u[s]));
#pragma unroll
          for (int x = 4; x < 32; x <<= 1)
#pragma unroll
            for (int s = 0; s < 4; ++s) top[s] = fmaxf(top[s], __shfl_xor_sync(0xFFFFFFFFu, top[s], x));   // of the eight lanes with the same row (a NaN drops out)
#pragma unroll
          for (int s = 0; s < 4; ++s) may |= (sc[s] >= fmaxf(need[s], score_needed(top[s])) && need[s] == need[s]) ? 1u << s : 0u;
        }
        while (may != 0u) {
          const int s = __ffs(may) - 1;
          may &= may - 1;
          offer(c + i + (q ^ s), fmaf(pick(lg, s), inv_t, -logf(-logf(pick(u, s)))), id);
        }
      }
    };
    // what this CTA has found so far to the others, and theirs
    unsigned long long sent = 0ull;
    auto exchange = [&]() {
      if (threadIdx.x < C::kRows && s_row[threadIdx.x] >= 0) {
        const unsigned long long mine = *reinterpret_cast<volatile unsigned long long*>(&s_best[threadIdx.x]);
        if (mine > sent) { atomicMax(a.best + threadIdx.x, mine); sent = mine; }
        const unsigned long long seen = *reinterpret_cast<volatile unsigned long long*>(a.best + threadIdx.x);
        if (seen != 0ull && !(s_run[threadIdx.x] >= unpack_score(seen))) s_run[threadIdx.x] = unpack_score(seen);
      }
    };
    for (int t = 0; t < walk.n; ++t) {
      const uint32_t buf = t & 1;
      exchange();
      bool ok = mbar_try_wait(&acc_full[buf], (t >> 1) & 1);
      for (uint32_t i = 0; i < (1u << 21) && !ok && !*stop; ++i) ok = mbar_try_wait_sleep(&acc_full[buf], (t >> 1) & 1, 1000);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) { fail(); break; }
      tc_fence_after();
      const int row0 = walk.row(t, g, b), height = walk.height(t);
      const uint32_t acc = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * C::kAccCols;
      // few rows: a half of the warps per 128 ids; else alternate groups of sixteen rows
      constexpr bool kById = C::kRows <= 16 && C::kWide == 2;
#pragma unroll 1
      for (int w = kById ? half : 0; w < C::kWide; w += kById ? 2 : 1) {
        const int in = w * kTile + quarter * 32;
        if (in >= height) continue;
        const int id = row0 + in + lane;
        const bool counts = in + lane < height && id < a.v_limit;
#pragma unroll 1
        for (int c = kById ? 0 : half * 16; c < C::kRows && c < M; c += kById ? C::kRows : 32) sample(acc + w * MT, c, id, counts);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
    exchange();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kEpiWarps + 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, C::kTmemCols);
  }
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return n;
}

template <int MT>
cudaError_t launch_as(const void* W, const void* x, const void* x_lo, int M, int N, int K, int* err, RowScale rs, const SampleArgs& a, cudaStream_t s) {
  using C = HeadCfg<MT>;
  CUtensorMap tw, tp, tx, txl;
  if (!tc_tensor_map(W, N, K, kTile, &tw) || !tc_tensor_map(W, N, K, kPiece, &tp) || !tc_tensor_map(x, M, K, C::kRows, &tx) ||
      !tc_tensor_map(x_lo, M, K, C::kRows, &txl))
    return cudaErrorNotSupported;
  static OncePerDevice configured;
  const cudaError_t set = allow_smem(configured, head_sample_kernel<MT>, C::kSmemBytes);
  if (set != cudaSuccess) return set;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  RSD_LAUNCH((head_sample_kernel<MT>), std::min(sms, (N + kPiece - 1) / kPiece), kThreads, C::kSmemBytes, s, tw, tp, tx, txl, N, K, err, rs, a);
  return launched(1);
}

}  // namespace

bool head_sample_supported(int M, int N, int K) { return M >= 1 && M <= 128 && N >= 1 && K >= 8 && K % 8 == 0; }

// From two rounds of 256 ids on all SMs on, so that there is a tile under whose products the sampling of another runs.  us, head and sampling / here, T = 0.7:
// 19000 ids of 1536 columns at 9 / 64 / 128 rows 19 / 25, 28 / 40, 39 / 51; 38000 33 / 34, 48 / 48, 61 / 63; 76000 51 / 47, 78 / 60, 101 / 89; 151936
// 91 / 80 at 16 rows, 104 / 80 at 32, 129 / 92 at 64, 175 / 141 at 128, of 3584 columns 183 / 171, 200 / 174, 230 / 187, 347 / 265; two layers of 512
// columns with 4096 ids, 9 rows, 54 / 60 an iteration.  Up to eight rows the head's CTAs of few stages, three to an SM, are there before their
// turn and stream as well: an iteration of 14 layers of the 7B shape at 1 / 4 / 8 rows 1289 / 1297, 1330 / 1337, 1369 / 1374, of the 1.5B shape 482 / 483,
// 493 / 491, 539 / 532.
bool head_sample_pays(int M, int N, int K) { return head_sample_supported(M, N, K) && N >= 65536 && (M > 8 || K <= 2048); }

cudaError_t launch_head_sample(const void* W, const void* x, const void* x_lo, int N, int K, int* err, RowScale rs, const SampleArgs& a, cudaStream_t s) {
  const int M = a.n_slots;
  if (!head_sample_supported(M, N, K) || !x_lo || a.token != nullptr) return cudaErrorNotSupported;
  if (((uintptr_t)W & 15) || ((uintptr_t)x & 15) || ((uintptr_t)x_lo & 15)) return cudaErrorMisalignedAddress;
  if (M <= 8) return launch_as<16>(W, x, x_lo, M, N, K, err, rs, a, s);
  if (M <= 16) return launch_as<32>(W, x, x_lo, M, N, K, err, rs, a, s);
  if (M <= 32) return launch_as<64>(W, x, x_lo, M, N, K, err, rs, a, s);
  if (M <= 64) return launch_as<128>(W, x, x_lo, M, N, K, err, rs, a, s);
  return launch_as<256>(W, x, x_lo, M, N, K, err, rs, a, s);
}

}  // namespace rsd
