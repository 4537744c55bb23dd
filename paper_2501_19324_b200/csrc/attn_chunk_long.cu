// Causal attention of a long chunk of new tokens over paged fp16 KV on the 5th-generation tensor cores: prompts being
// cached, and prefixes of hundreds of keys and more.  head_dim 128, up to 8 query heads per KV head.
//
// A CTA takes two tiles of QT = 128 / G consecutive entries of the pass list and one KV head; the 128 rows of a tile are
// (entry, query head) pairs, row = entry * G + head.  Entries of different sequences are handled one run ("segment") at a
// time, the rows outside the segment masked.  Per segment the keys go by ONCE, in tiles of 128 (eight pages), and the two
// query tiles share every key and value tile that comes in:
//   S_j = Q_j K^T          tcgen05.mma, both operands in shared memory, S_j (128 columns of tensor memory)
//   softmax                a warpgroup per query tile, a thread per row: no exchange between threads.  p = 2^(s - m) with
//                          a REFERENCE maximum m that is raised only when a tile's maximum exceeds it by more than 8
//                          (p <= 2^8 fits fp16 easily): only then are the row's output and sum rescaled, by its own
//                          thread, in place.  After the first tile that is rare, so O stays in tensor memory.
//   O_j += P_j V           P_j overwrites S_j as fp16 and is the left operand straight from tensor memory.
// While one tile's softmax runs, the tensor cores work for the other tile: the issue order is PV_0(i) S_0(i+1) PV_1(i)
// S_1(i+1), and the barriers are two per tile and key tile (scores ready, weights ready).
//
// What bounds it: the exponentials (128 x 128 per tile and key tile take 1024 cycles of an SM's 16 per cycle) and the MMAs
// (1024 cycles per query tile and key tile) are about even.  The older kernel (attn_chunk_tc.cu) walks the keys twice in
// tiles of 64 and hands every tile through five roles; it stays for short passes and few CTAs, see attn_chunk_long_pays.  One row of 4096
// tokens over a prefix of 4000, 28 / 4 heads: 935 us (380 TFLOP/s algorithmic) there, 426 us (833) here; 16 rows of 256
// over 3072: 627 us, 379 us.
//
// Roles: warps 0-3 and 4-7 softmax of tile 0 and 1, warp 8 issues every MMA, warp 9 fetches pages (the boxes and the
// treatment of the last, partly cached page are those of attn_chunk_tc.cu).  Every wait is bounded; on expiry the CTA
// raises an error flag, waits for its copies in flight, frees its tensor memory and leaves.
#include <cuda.h>

#include "attn_chunk_tc.cuh"
#include "common.cuh"
#include "kernels.cuh"

namespace rsd {

namespace {

using namespace tc;
using namespace chunk;

constexpr int kKeys = 128, kTilePages = kKeys / kPageTokens;     // keys per tile: eight pages
constexpr int kSlots = 4;                                        // ring slots: K, V, K, V (so a slot only ever holds one kind)
constexpr int kSlotBytes = kTilePages * kBlockBytes;             // 32 KB
constexpr int kQBytes = 128 * kHd * 2;                           // one query tile: [2 dim halves][128 rows][64 dims], 128-byte swizzle
constexpr int kMetaBytes = 4096;
constexpr size_t kSmemBytes = 1024 + 2 * kQBytes + kSlots * kSlotBytes + kMetaBytes;
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
constexpr int kMmaWarp = 8, kFetchWarp = 9, kThreads = 320;
// kind::f16: fp32 accumulate, fp16 A and B, both K-major, M = 128, N = 128
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
constexpr uint32_t kColS = 0, kColO = 256, kTmemCols = 512;      // S_j (and P_j) at 128 j, O_j at 256 + 128 j
constexpr float kRaise = 8.f;

struct Meta {
  uint64_t kv_full[kSlots], kv_empty[kSlots], s_full[2], p_full[2], o_full[2];
  uint32_t tmem_slot, stop;
  int32_t row[256], pos[256];
};
static_assert(sizeof(Meta) <= kMetaBytes, "metadata block");

// A run of entries of one sequence: [seg, e), and how many key tiles each query tile has to see.
struct Segment { int e, row, pos_last, n[2]; };

__device__ __forceinline__ Segment segment_at(const Meta* mt, int seg, int n_ent, int QT) {
  Segment s;
  s.row = mt->row[seg];
  s.e = seg + 1;
  while (s.e < n_ent && mt->row[s.e] == s.row) ++s.e;
  s.pos_last = mt->pos[s.e - 1];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int lo = max(seg, j * QT), hi = min(s.e, (j + 1) * QT);
    s.n[j] = hi > lo ? mt->pos[hi - 1] / kKeys + 1 : 0;
  }
  return s;
}

template <typename OT, bool PROBE = false>
__global__ void __launch_bounds__(kThreads, 1)
attn_chunk_long_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v, const float* q, PassView p,
                       const __half* pool, const int32_t* page_table, int max_pages, OT* out, OT* out_lo, int H, int KV, int QT,
                       int* err) {
  RSD_PDL_TRIGGER();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* ring = smem + 2 * kQBytes;
  Meta* mt = reinterpret_cast<Meta*>(ring + kSlots * kSlotBytes);
  volatile uint32_t* stop = &mt->stop;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = H / KV, kvh = blockIdx.y, h0 = kvh * G;
  // the last entries of a row see the most keys: they start first
  const int t0 = (int)(gridDim.x - 1 - blockIdx.x) * 2 * QT;
  const int n_ent = min(2 * QT, p.T - t0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) { mbar_init(&mt->kv_full[s], 1); mbar_init(&mt->kv_empty[s], 1); }
    for (int j = 0; j < 2; ++j) { mbar_init(&mt->s_full[j], 1); mbar_init(&mt->p_full[j], 4); mbar_init(&mt->o_full[j], 1); }
    mt->stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) tmem_alloc(&mt->tmem_slot, kTmemCols);
  // the value slots start zeroed: a buffer no page was fetched into is multiplied by weights that are exactly zero
  for (int i = threadIdx.x; i < 2 * (kSlotBytes / 16); i += kThreads)
    *reinterpret_cast<uint4*>(ring + (size_t)(2 * (i / (kSlotBytes / 16)) + 1) * kSlotBytes + (size_t)(i % (kSlotBytes / 16)) * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  RSD_PDL_WAIT();
  if (threadIdx.x < 256) {
    const int i = threadIdx.x;
    mt->row[i] = i < n_ent ? p.tok_row[t0 + i] : -1;
    mt->pos[i] = i < n_ent ? p.tok_pos[t0 + i] : 0;
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = mt->tmem_slot;
  // Q_j: row r = entry j QT + r / G, head r % G; 1 / sqrt(head_dim) and log2(e) folded in, so the scores come out in
  // units of log 2.  Rows beyond the tile's entries are zero.
  const int wg = warp >> 2, r = threadIdx.x & 127, qi = wg * QT + r / G, g = r % G;      // softmax threads' row
  const bool has_row = warp < 8 && r < QT * G && qi < n_ent && mt->row[qi] >= 0;
  if (warp < 8) {
    const float scale = rsqrtf((float)kHd) * 1.4426950408889634f;
    const float* src = q + ((size_t)(t0 + qi) * H + h0 + g) * kHd;
    uint8_t* dst = smem + wg * kQBytes + r * 128;
    // (a thread its own row: lines come through L1; a row per warp load, coalesced, measured 20 % slower on short prefixes)
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
      uint4 packed = make_uint4(0u, 0u, 0u, 0u);
      if (has_row) {
        const float4 a = *reinterpret_cast<const float4*>(src + 8 * c), b = *reinterpret_cast<const float4*>(src + 8 * c + 4);
        packed = make_uint4(pack_half2(a.x * scale, a.y * scale), pack_half2(a.z * scale, a.w * scale),
                            pack_half2(b.x * scale, b.y * scale), pack_half2(b.z * scale, b.w * scale));
      }
      *reinterpret_cast<uint4*>(dst + (c >> 3) * (kQBytes / 2) + (((c & 7) ^ (r & 7)) << 4)) = packed;
    }
  }
  fence_async_smem();
  __syncthreads();
  auto fail = [&]() { if (*stop == 0) { if (err) atomicCAS(err, 0, -5); *stop = 1; } };

  if (warp == kFetchWarp) {
    // ---------------- fetch warp: per key tile a slot of keys, then a slot of values ----------------
    uint32_t it = 0;
    int seg = 0;
    bool ok = true;
    while (!PROBE && seg < n_ent && ok) {
      const Segment sg = segment_at(mt, seg, n_ent, QT);
      if (sg.row >= 0) {
        const int n_tiles = max(sg.n[0], sg.n[1]), n_pages = sg.pos_last / kPageTokens + 1;
        const int tail = (sg.pos_last + 1) % kPageTokens;    // cached tokens of the last page when it is not full
        const int32_t* pt = page_table + (size_t)sg.row * max_pages;
        // page ids are read 32 at a time (four tiles), a batch ahead of their use
        int pg_cur = lane < n_pages ? pt[lane] : -1;
        int pg_nxt = 32 + lane < n_pages ? pt[32 + lane] : -1;
        for (int t = 0; t < n_tiles && ok; ++t) {
          if (t > 0 && (t & 3) == 0) {
            pg_cur = pg_nxt;
            const int ahead = (t / 4 + 1) * 32 + lane;
            pg_nxt = ahead < n_pages ? pt[ahead] : -1;
          }
          const int i = lane & 7, page = kTilePages * t + i;       // lanes 0-7 issue
          const int pg = __shfl_sync(0xFFFFFFFFu, pg_cur, page & 31);
          for (int kind = 0; kind < 2; ++kind, ++it) {             // keys, values
            const int sl = it % kSlots;
            bool got = true;
            if (lane == 0) got = wait_sleep(&mt->kv_empty[sl], ((it / kSlots) & 1u) ^ 1u, stop);
            got = __all_sync(0xFFFFFFFFu, got && !*stop);          // one decision for the whole warp
            if (!got) { ok = false; break; }
            uint8_t* dst = ring + (size_t)sl * kSlotBytes;
            const bool partial = kind == 1 && tail != 0 && page == n_pages - 1;
            if (__any_sync(0xFFFFFFFFu, partial && lane < 8)) {
              const int last = n_pages - 1, pg_last = __shfl_sync(0xFFFFFFFFu, pg_cur, last & 31);
              copy_partial_values(pool + ((size_t)pg_last * 2 * KV + KV + kvh) * (kPageTokens * kHd),
                                  dst + (last & 7) * kBlockBytes, tail, lane);
              __syncwarp();
            }
            const bool load = lane < 8 && page < n_pages && !partial;
            const uint32_t n_boxes = __popc(__ballot_sync(0xFFFFFFFFu, load));
            if (lane == 0) mbar_expect_tx(&mt->kv_full[sl], n_boxes * kBlockBytes);
            __syncwarp();
            const int blk = pg * 2 * KV + kvh;
            if (load && kind == 0) tma_load_block_5d(dst + i * kBlockBytes, &tm_k, &mt->kv_full[sl], blk);
            if (load && kind == 1) tma_load_block_3d(dst + i * kBlockBytes, &tm_v, &mt->kv_full[sl], blk + KV);
          }
        }
      }
      seg = sg.e;
    }
    // copies in flight must have landed before the CTA may leave
    if (lane == 0) {
      const uint32_t first = it > (uint32_t)kSlots ? it - kSlots : 0;
      for (uint32_t k = first; k < it; ++k) mbar_wait(&mt->kv_full[k % kSlots], (k / kSlots) & 1u, kProbeLimit);
      if (!ok) fail();
    }
  } else if (warp == kMmaWarp) {
    // ---------------- the one MMA issuer: a converged warp, one lane issues ----------------
    {
      const uint32_t on = elect_one();
      uint32_t it = 0, n_p[2] = {0, 0};
      bool ok = true;
      int seg = 0;
      auto wait = [&](uint64_t* bar, uint32_t parity) {
        const bool got = mbar_wait(bar, parity, PROBE ? kProbePolls : kProbeLimit);
        return __all_sync(0xFFFFFFFFu, got && !*stop) != 0;
      };
      auto scores = [&](int j, uint32_t k_it) {
        const uint32_t a = smem_u32(smem + j * kQBytes);
        const uint64_t k_desc = desc_sw128(smem_u32(ring + (size_t)(k_it % kSlots) * kSlotBytes), 2048);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_bf16_if(on, tmem_base + kColS + j * 128, smem_desc_sw128(a + hh * (kQBytes / 2) + kk * 32),
                         k_desc + (uint64_t)((hh * 1024 + kk * 32) >> 4), kIdesc, (hh > 0 || kk > 0) ? 1u : 0u);
        umma_commit_if(on, &mt->s_full[j]);
      };
      while (seg < n_ent && ok && !__any_sync(0xFFFFFFFFu, *stop)) {
        const Segment sg = segment_at(mt, seg, n_ent, QT);
        if (sg.row >= 0) {
          const int n_tiles = max(sg.n[0], sg.n[1]);
          // items of the ring: keys of tile i at it + 2 i, values at it + 2 i + 1
          ok = wait(&mt->kv_full[it % kSlots], (it / kSlots) & 1u);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (sg.n[j] > 0) scores(j, it);
          umma_commit_if(on, &mt->kv_empty[it % kSlots]);
          for (int i = 0; i < n_tiles && ok; ++i) {
            const uint32_t v_it = it + 2 * i + 1, k_it = v_it + 1;
            ok = wait(&mt->kv_full[v_it % kSlots], (v_it / kSlots) & 1u);
            if (ok && i + 1 < n_tiles) ok = wait(&mt->kv_full[k_it % kSlots], (k_it / kSlots) & 1u);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              if (!ok || i >= sg.n[j]) continue;
              ok = wait(&mt->p_full[j], n_p[j] & 1u);
              if (!ok) continue;
              ++n_p[j];
              tc_fence_after();
              const uint64_t v_desc = desc_sw32(smem_u32(ring + (size_t)(v_it % kSlots) * kSlotBytes));
#pragma unroll
              for (int kk = 0; kk < kTilePages; ++kk)
                umma_f16_ts_if(on, tmem_base + kColO + j * 128, tmem_base + kColS + j * 128 + kk * 8,
                               v_desc + (uint64_t)((kk * kBlockBytes) >> 4), kIdesc, (i > 0 || kk > 0) ? 1u : 0u);
              if (i + 1 < sg.n[j]) scores(j, k_it);
              else umma_commit_if(on, &mt->o_full[j]);
            }
            if (!ok) break;
            umma_commit_if(on, &mt->kv_empty[v_it % kSlots]);
            if (i + 1 < n_tiles) umma_commit_if(on, &mt->kv_empty[k_it % kSlots]);
          }
          it += 2 * n_tiles;
        }
        seg = sg.e;
      }
      if (!ok && on) fail();
    }
  } else {
    // ---------------- softmax warps: thread = tile row = tensor-memory lane ----------------
    const uint32_t lanes = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_s = lanes + kColS + wg * 128, t_o = lanes + kColO + wg * 128;
    uint32_t n_s = 0, n_o = 0;
    bool ok = true;
    int seg = 0;
    while (seg < n_ent && ok) {
      const Segment sg = segment_at(mt, seg, n_ent, QT);
      const int n_tiles = sg.n[wg];
      if (sg.row >= 0 && n_tiles > 0) {
        const bool mine = has_row && qi >= seg && qi < sg.e;
        const int pq = mine ? mt->pos[qi] : -1;              // last visible key position; -1: the row is not of this segment
        float m = -INFINITY, l = 0.f;
        for (int t = 0; t < n_tiles; ++t, ++n_s) {
          ok = wait_sleep_warp(&mt->s_full[wg], n_s & 1u, stop);
          if (!ok) break;
          tc_fence_after();
          float v[128];
          tmem_ld128(t_s, v);
          const int k0 = t * kKeys;
          if (k0 + kKeys - 1 > pq) {
#pragma unroll
            for (int j = 0; j < 128; ++j)
              if (k0 + j > pq) v[j] = -INFINITY;
          }
          float mx[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
          for (int j = 4; j < 128; ++j) mx[j & 3] = fmaxf(mx[j & 3], v[j]);
          const float tile_max = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
          const bool raise = tile_max > m + kRaise;          // true for a row's first visible tile (m = -inf)
          if (__any_sync(0xFFFFFFFFu, raise)) {
            const float corr = !raise ? 1.f : (m == -INFINITY ? 0.f : ex2(m - tile_max));
            if (raise) { m = tile_max; l *= corr; }
            // every MMA issued before these scores has completed, O += P V of the previous tile included, and the next
            // one waits for this tile's weights: the accumulator is this warp's for now
            if (t > 0) {
#pragma unroll
              for (int c = 0; c < 128; c += 32) {
                float o[32];
                tmem_ld32(t_o + c, o);
                uint32_t u[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) u[k] = __float_as_uint(o[k] * corr);
                tmem_st32(t_o + c, u);
              }
            }
          }
          const float m_use = m == -INFINITY ? 0.f : m;
          float sum[4] = {0.f, 0.f, 0.f, 0.f};
          uint32_t w[64];
#pragma unroll
          for (int j = 0; j < 128; j += 2) {
            const float a = ex2(v[j] - m_use), b = ex2(v[j + 1] - m_use);     // 2^-inf = 0: masked keys
            sum[(j >> 1) & 3] += a + b;
            w[j >> 1] = pack_half2(a, b);
          }
          l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
          tmem_st32(t_s, w);
          tmem_st32(t_s + 32, w + 32);
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&mt->p_full[wg]);
        }
        if (!ok) break;
        ok = wait_sleep_warp(&mt->o_full[wg], n_o & 1u, stop);
        if (!ok) break;
        ++n_o;
        tc_fence_after();
        const float inv = l > 0.f ? 1.f / l : 0.f;
        const size_t o0 = ((size_t)(t0 + qi) * H + h0 + g) * kHd;
#pragma unroll
        for (int c = 0; c < 128; c += 32) {
          float v[32];
          tmem_ld32(t_o + c, v);
          if (mine) {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] *= inv;
            store16<OT>(out, out_lo, o0 + c, v);
            store16<OT>(out, out_lo, o0 + c + 16, v + 16);
          }
        }
        // the next segment's first O = P V overwrites the accumulator; it waits for weights that this warp posts after this
        tc_fence_before();
        __syncwarp();
      }
      seg = sg.e;
    }
    if (!ok) fail();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

template <typename OT, bool PROBE = false>
cudaError_t launch_long(const CUtensorMap& tm_k, const CUtensorMap& tm_v, const float* q, PassView p, KvView kv, void* out, void* out_lo,
                        int H, int KV, int* err, cudaStream_t s) {
  static OncePerDevice configured;
  const cudaError_t set = allow_smem(configured, attn_chunk_long_kernel<OT, PROBE>, kSmemBytes);
  if (set != cudaSuccess) return set;
  const int QT = 128 / (H / KV);
  RSD_LAUNCH((attn_chunk_long_kernel<OT, PROBE>), dim3((p.T + 2 * QT - 1) / (2 * QT), KV), kThreads, kSmemBytes, s, tm_k, tm_v, q, p,
             (const __half*)kv.pool_layer, kv.page_table, kv.max_pages, (OT*)out, (OT*)out_lo, H, KV, QT, err);
  return launched(1);
}

}  // namespace

cudaError_t launch_attn_chunk_long(const float* q, PassView p, KvView kv, void* out, void* out_lo, int out_dtype, int H, int KV, int* err,
                                   cudaStream_t s, bool probe) {
  if (p.T <= 0) return cudaSuccess;
  CUtensorMap tm_k, tm_v;
  if (!tc_tensor_map_kv(kv.pool_layer, 0, &tm_k) || !tc_tensor_map_kv(kv.pool_layer, 1, &tm_v)) return cudaErrorInvalidValue;
  if (probe) return launch_long<float, true>(tm_k, tm_v, q, p, kv, out, nullptr, H, KV, err, s);
  if (out_dtype == 2) return launch_long<__half>(tm_k, tm_v, q, p, kv, out, nullptr, H, KV, err, s);
  if (out_dtype == 1) return launch_long<__nv_bfloat16>(tm_k, tm_v, q, p, kv, out, out_lo, H, KV, err, s);
  return launch_long<float>(tm_k, tm_v, q, p, kv, out, nullptr, H, KV, err, s);
}

}  // namespace rsd
