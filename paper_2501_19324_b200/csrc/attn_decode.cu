// Paged-KV grouped-query decode attention (one query token per row), sm_100a.
//
// A CTA of 4 warps (16 in one form) serves one (row slot, KV head, context split): the G = H / KV query heads that
// share the KV head are the rows of a 16-row MMA tile, so every key / value is read once from HBM for
// the whole group.  Each warp walks its share of the 16-token pages through a ring of page buffers of its own in shared
// memory (16-byte cp.async, a page ahead):
//   S  = Q K^T   with mma.sync m16n8k16 (16-bit in, fp32 out): a key fragment is one 128-bit load (the order of
//        the head dims inside a 32-dim block is permuted identically for Q and K, which a dot product does not see);
//   softmax statistics per head are kept on line (running max / sum), reduced over the 4 lanes that
//        share a row with warp shuffles;
//   O += P V     with the same MMA: values are stored transposed inside a page ([hd][16 tokens]), so a
//        B fragment is one 64-bit load; the order of the tokens inside a page is permuted identically
//        for P and V.
// The warps' partial (max, sum, O) meet in shared memory.  With 2 to 8 context splits the splits of a (slot, KV
// head) are the CTAs of one thread-block cluster: each sends every other CTA its partial of the slice of the G x HD outputs
// that this one merges, and after a cluster barrier every CTA merges and writes its slice out of its own shared memory: no
// second launch and no trip through global memory.  With more splits than a cluster holds the CTA writes its partial to
// scratch and a second kernel merges them.
//
// In a decode pass only the pass's own tokens are written by the kernels just before: every page that ends ahead of the
// pass's first new position is older than the pass.  Lists, page ids and each warp's first pages are therefore
// requested before the wait for the preceding kernels and stream in while the qkv product and the rotation still run;
// at the step loop's contexts (a page or two per warp) the cache has arrived when the query has.  (Fragments loaded from
// global memory straight into registers had one page a warp in flight and none under the wait: 12.3 us a launch at 32
// rows x 400 tokens, 12 / 2 heads, and 330 us for 64 rows x 4096-16384 tokens, 28 / 4 heads.)
//
// What is left after the wait is a chain of short steps.  Of the 5.8 us from the wait to the end at one row (12 / 2 heads,
// a page per warp) 3.3 lay behind the last page: outputs stored with 8-way bank conflicts, one output dim a thread, loads
// from the other CTAs' shared memory and a running maximum over them, a second cluster barrier; and the products of a page
// formed one chain through the accumulators of the tile's padding rows.  As it stands: 3.8 us, 2.0 behind the last page;
// 64 rows x 4096-16384 tokens: 201 us, the copy bandwidth.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.cuh"

namespace rsd {

namespace {

namespace cg = cooperative_groups;

constexpr int kMaxSplits = 32;
constexpr int kClusterSplits = 8;   // the portable cluster size

// Two fp32 values rounded to the cache's 16-bit type and packed into one MMA operand register.
template <typename KT> __device__ __forceinline__ uint32_t pack2(float lo, float hi);
template <> __device__ __forceinline__ uint32_t pack2<__nv_bfloat16>(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
template <> __device__ __forceinline__ uint32_t pack2<__half>(float lo, float hi) {
  __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// The same pair split into a high and a low 16-bit part: (a, b) = hi + lo up to ~2^-22 relative.
template <typename KT> __device__ __forceinline__ void pack2_split(float a, float b, uint32_t& hi, uint32_t& lo) {
  const KT ah = from_f32<KT>(a), bh = from_f32<KT>(b);
  hi = pack2<KT>(to_f32(ah), to_f32(bh));
  lo = pack2<KT>(a - to_f32(ah), b - to_f32(bh));
}

// D += A B for a tile whose rows 8..15 are padding: their accumulators enter as zeros and what comes out is dropped, so
// that no product waits for another one's padding.
template <typename KT>
__device__ __forceinline__ void mma_16816(float& d0, float& d1, uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {
  float x, y;
  if (std::is_same<KT, __half>::value)
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%8,%5,%8}, {%6,%7}, {%0,%1,%9,%9};"
                 : "+f"(d0), "+f"(d1), "=f"(x), "=f"(y) : "r"(a0), "r"(a2), "r"(b0), "r"(b1), "r"(0u), "f"(0.f));
  else
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%8,%5,%8}, {%6,%7}, {%0,%1,%9,%9};"
                 : "+f"(d0), "+f"(d1), "=f"(x), "=f"(y) : "r"(a0), "r"(a2), "r"(b0), "r"(b1), "r"(0u), "f"(0.f));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Shared memory of a CTA: NW warps x kStages page buffers; the warps' outputs take its place after the loop.  An extended
// page (16 KB) gets one buffer a warp, a plain one (8 KB) two, so that three CTAs of four warps fit an SM either way; of sixteen warps
// one buffer each, one CTA an SM.
template <int HD, bool EXT, int NW> struct DecCfg {
  static constexpr int kPageBytes = (EXT ? 4 : 2) * kPageTokens * HD * 2;
  static constexpr int kStages = EXT || NW > 4 ? 1 : 2;
  static constexpr int kOutBytes = NW * 8 * (HD + 8) * 4;
  static constexpr int kRingBytes = NW * kStages * kPageBytes > kOutBytes ? NW * kStages * kPageBytes : kOutBytes;
};

// part_o: [slot][head][split][HD] un-normalised outputs; part_ml: [slot][head][split][2] (max, sum).
// EXT: queries and softmax weights enter the products as hi + lo pairs and every page carries the low
// halves of its keys and values in two more blocks: the attention is accurate to about 2^-20.
// new_tokens: how many of a row's last positions the pass itself writes.
// FUSE (one split; every row's only new position is its last): the kernel takes the qkv product itself, K-split partial sums or
// not, adds them up, rotates, and writes the new key and value to the cache: see new_token below.
// NW: warps, 4, or 16 where there is one CTA per SM at most (wide_ctas).
template <int HD, typename KT, typename OT, bool EXT, bool CL, bool FUSE, int NW>
__global__ void __launch_bounds__(32 * NW, NW == 4 ? 3 : 1)
attn_decode_kernel(const float* q, KT* pool, const int32_t* page_table, int max_pages, const int32_t* slot_row,
                   const int32_t* len_or_pos, int len_offset, OT* out, OT* out_lo, float* part_o, float* part_ml, int H, int KV,
                   int n_splits, const int32_t* n_active, int new_tokens, const float* partials, int k_splits, const float2* rope) {
  RSD_PDL_TRIGGER();
  if (n_active == nullptr) RSD_PDL_WAIT();   // a decode pass's lists and old pages may be read ahead of the wait, others not
  using Cfg = DecCfg<HD, EXT, NW>;
  constexpr int kThreads = 32 * NW;
  constexpr int KB = HD / 32;    // 32-dim blocks of the head dimension
  constexpr int NT = HD / 8;     // 8-dim output tiles
  constexpr int kBlock = kPageTokens * HD;       // elements of one head's keys (or values) in a page
  constexpr int kStages = Cfg::kStages, kParts = EXT ? 4 : 2;
  extern __shared__ __align__(128) uint8_t ring_raw[];
  __shared__ float s_m[NW][8], s_l[NW][8];
  auto s_o = reinterpret_cast<float(*)[8][HD + 8]>(ring_raw);   // rows 32 bytes apart modulo 128: the fragments' stores do not collide
  const int kvh = blockIdx.x, slot = blockIdx.y, split = blockIdx.z;
  const bool idle = n_active != nullptr && ld_cg(n_active) == 0;
  const int row = slot_row ? ld_cg(slot_row + slot) : slot;
  const int ctx = ld_cg(len_or_pos + slot) + len_offset;
  if (idle || row < 0 || ctx <= 0) { RSD_PDL_WAIT(); return; }
  const int G = H / KV, h0 = kvh * G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const float scale = rsqrtf((float)HD);

  const int n_pages = (ctx + kPageTokens - 1) / kPageTokens;
  const int pps = (n_pages + n_splits - 1) / n_splits;
  const int p_begin = split * pps, p_end = min(n_pages, p_begin + pps);
  const int32_t* pt = page_table + (size_t)row * max_pages;
  const size_t page_elems = (size_t)kParts * KV * kBlock;
  KT* ring = reinterpret_cast<KT*>(ring_raw) + (size_t)warp * kStages * kParts * kBlock;
  // Keys of token t: 16-byte chunk c of its row sits at chunk c ^ 4 (t & 1), so that the two rows a quarter warp reads
  // together fall on different banks.  Values as in the page.
  auto fetch = [&](int page, int stage) {
    const KT* src = pool + (size_t)page * page_elems + (size_t)kvh * kBlock + lane * 8;
    KT* dst = ring + stage * kParts * kBlock;
    constexpr int kChunks = kBlock / 8, kRow = HD / 8;
#pragma unroll
    for (int part = 0; part < kParts; ++part) {
#pragma unroll
      for (int i = 0; i < kChunks / 32; ++i) {
        const int c = i * 32 + lane, d = (part & 1) ? c : (c ^ (((c / kRow) & 1) << 2));
        cp_async16(dst + part * kBlock + d * 8, src + (size_t)part * KV * kBlock + i * 256);
      }
    }
  };
  // pages [0, n_old) may be read ahead of the wait: they are older than the pass, or (FUSE) all but the token that this
  // kernel fills in itself
  const int first = p_begin + warp, n_old = FUSE ? n_pages : (ctx - new_tokens) / kPageTokens;
  int next = first;                              // the page whose turn it is to be fetched
  int next_id = next < p_end ? ld_cg(pt + next) : 0;
  auto fetch_next = [&](int stage) {
    if (next < p_end) {
      fetch(next_id, stage);
      next += NW;
      if (next < p_end) next_id = ld_cg(pt + next);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  int fetched = 0;
  for (; fetched < kStages && next < min(p_end, n_old); ++fetched) fetch_next(fetched);
  for (; FUSE && fetched < kStages; ++fetched) fetch_next(fetched);
  // every CTA of the cluster runs before the others write to its shared memory
  if (CL) cg::this_cluster().barrier_arrive();
  RSD_PDL_WAIT();
  for (; fetched < kStages; ++fetched) fetch_next(fetched);

  // the group's queries, rounded once by the whole block
  constexpr int kLd = HD + 32;                   // rows 64 bytes apart modulo 128: the fragment loads below do not collide
  __shared__ __align__(16) KT s_q[EXT ? 2 : 1][8][kLd];
  __shared__ __align__(16) KT s_new[FUSE ? kParts : 1][HD];   // the new token's key and value (and their low halves)
  const int new_page = (ctx - 1) / kPageTokens, new_slot = (ctx - 1) % kPageTokens;
  if (FUSE) {
    // new_token.  A task is four neighbouring pairs (i, i + HD / 2) of a query head, of the key or of the value; P lanes of a warp
    // share its K splits, all of them in flight at once.
    constexpr int NQ = HD / 8, kAhead = 3, P = NW == 16 ? 2 : 1, R = kSumGroups / P, kPerWarp = 32 / P;
    const int n_tasks = (G + 2) * NQ, width = (H + 2 * KV) * HD;
    const size_t sstride = (size_t)gridDim.y * width;
    const int per = (k_splits + kSumGroups - 1) / kSumGroups;
    for (int idx = threadIdx.x; idx < (8 - G) * HD; idx += kThreads) {   // the tile's rows beyond the group
      s_q[0][G + idx / HD][idx % HD] = from_f32<KT>(0.f);
      if (EXT) s_q[EXT ? 1 : 0][G + idx / HD][idx % HD] = from_f32<KT>(0.f);
    }
    const int part = lane / kPerWarp;              // of the K splits: runs [part R, part R + R)
    // (P == 1: a task per thread; the loop over whole warps there cost registers, 80 bytes of spills instead of 48 with hi + lo caches)
    for (int task0 = P == 1 ? threadIdx.x : warp * kPerWarp; task0 < n_tasks; task0 += NW * kPerWarp) {
      const int task = P == 1 ? task0 : min(task0 + lane % kPerWarp, n_tasks - 1);   // whole warps: lanes beyond the last task repeat it
      const bool is_q = task < G * NQ;
      const int hh = is_q ? task / NQ : task / NQ - G, dd = 4 * (task % NQ);   // one of the group's heads, or 0 = the key, 1 = the value
      const size_t src = (size_t)slot * width + (size_t)(is_q ? h0 + hh : H + hh * KV + kvh) * HD + dd;
      float a[4] = {0.f, 0.f, 0.f, 0.f}, b[4] = {0.f, 0.f, 0.f, 0.f};
      if (k_splits <= 1) {
        *reinterpret_cast<float4*>(a) = ld_cg(reinterpret_cast<const float4*>(q + src));
        *reinterpret_cast<float4*>(b) = ld_cg(reinterpret_cast<const float4*>(q + src + HD / 2));
      } else {
        // the order of the additions is rope_kv_kernel's: kSumGroups runs of splits, then their sums
        float ga[R][4], gb[R][4];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int i = 0; i < 4; ++i) ga[r][i] = gb[r][i] = 0.f;
        for (int s0 = 0; s0 < per; s0 += kAhead) {
          float4 ta[R][kAhead], tb[R][kAhead];
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
              if (s0 + u < per && (part * R + r) * per + s0 + u < k_splits) {
                const float* at = partials + (size_t)((part * R + r) * per + s0 + u) * sstride + src;
                ta[r][u] = ld_cg(reinterpret_cast<const float4*>(at));
                tb[r][u] = ld_cg(reinterpret_cast<const float4*>(at + HD / 2));
              }
#pragma unroll
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
              if (s0 + u < per && (part * R + r) * per + s0 + u < k_splits) {
                ga[r][0] += ta[r][u].x; ga[r][1] += ta[r][u].y; ga[r][2] += ta[r][u].z; ga[r][3] += ta[r][u].w;
                gb[r][0] += tb[r][u].x; gb[r][1] += tb[r][u].y; gb[r][2] += tb[r][u].z; gb[r][3] += tb[r][u].w;
              }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          a[i] = ga[0][i]; b[i] = gb[0][i];
#pragma unroll
          for (int r = 1; r < R; ++r) { a[i] += ga[r][i]; b[i] += gb[r][i]; }
          if (P == 2) {                            // the other lane's runs, one after the other
#pragma unroll
            for (int r = 0; r < R; ++r) {
              a[i] += __shfl_down_sync(0xFFFFFFFFu, ga[r][i], kPerWarp & 31);
              b[i] += __shfl_down_sync(0xFFFFFFFFu, gb[r][i], kPerWarp & 31);
            }
          }
        }
      }
      if (P > 1 && (part > 0 || task0 + lane >= n_tasks)) continue;
      if (is_q || hh == 0) {
        const float2* cs = rope + (size_t)(ctx - 1) * (HD / 2) + dd;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float ra = rotate_lo(a[i], b[i], cs[i]), rb = rotate_hi(a[i], b[i], cs[i]);
          a[i] = ra; b[i] = rb;
        }
      }
      __align__(8) KT hi[2][4], lo[2][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        hi[0][i] = from_f32<KT>(a[i]); lo[0][i] = from_f32<KT>(a[i] - to_f32(hi[0][i]));
        hi[1][i] = from_f32<KT>(b[i]); lo[1][i] = from_f32<KT>(b[i] - to_f32(hi[1][i]));
      }
      if (is_q) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          *reinterpret_cast<uint2*>(&s_q[0][hh][half * (HD / 2) + dd]) = *reinterpret_cast<const uint2*>(hi[half]);
          if (EXT) *reinterpret_cast<uint2*>(&s_q[EXT ? 1 : 0][hh][half * (HD / 2) + dd]) = *reinterpret_cast<const uint2*>(lo[half]);
        }
      } else {
        KT* blk = pool + (size_t)ld_cg(pt + new_page) * page_elems + (size_t)hh * KV * kBlock + (size_t)kvh * kBlock;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int d0 = half * (HD / 2) + dd;
          *reinterpret_cast<uint2*>(&s_new[hh][d0]) = *reinterpret_cast<const uint2*>(hi[half]);
          if (EXT) *reinterpret_cast<uint2*>(&s_new[EXT ? hh + 2 : 0][d0]) = *reinterpret_cast<const uint2*>(lo[half]);
          if (hh == 0) {
            *reinterpret_cast<uint2*>(blk + new_slot * HD + d0) = *reinterpret_cast<const uint2*>(hi[half]);
            if (EXT) *reinterpret_cast<uint2*>(blk + (size_t)2 * KV * kBlock + new_slot * HD + d0) = *reinterpret_cast<const uint2*>(lo[half]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              blk[(d0 + i) * kPageTokens + new_slot] = hi[half][i];
              if (EXT) blk[(size_t)2 * KV * kBlock + (d0 + i) * kPageTokens + new_slot] = lo[half][i];
            }
          }
        }
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8 * HD / kThreads; ++i) {     // one coalesced round of loads
      const int idx = i * kThreads + threadIdx.x, gg = idx / HD, dd = idx % HD;
      const float v = gg < G ? q[((size_t)slot * H + h0 + gg) * HD + dd] : 0.f;
      const KT hi = from_f32<KT>(v);
      s_q[0][gg][dd] = hi;
      if (EXT) s_q[EXT ? 1 : 0][gg][dd] = from_f32<KT>(v - to_f32(hi));
    }
  }
  __syncthreads();
  // Q fragments (rows 8..15 of the tile are padding): dims 32j + 8t + e of head h0 + g
  __align__(16) uint32_t qa[KB][2][2], ql[EXT ? KB : 1][2][2];
#pragma unroll
  for (int j = 0; j < KB; ++j) {
    *reinterpret_cast<uint4*>(qa[j]) = *reinterpret_cast<const uint4*>(&s_q[0][g][32 * j + 8 * t]);
    if (EXT) *reinterpret_cast<uint4*>(ql[EXT ? j : 0]) = *reinterpret_cast<const uint4*>(&s_q[EXT ? 1 : 0][g][32 * j + 8 * t]);
  }
  float o[NT][2];
#pragma unroll
  for (int i = 0; i < NT; ++i) { o[i][0] = o[i][1] = 0.f; }
  float m_run = -INFINITY, l_run = 0.f;
  // tokens whose keys this lane loads: tile 0 -> 4(g/2) + g%2, tile 1 -> that + 2 (the same parity)
  const int tok0 = 4 * (g >> 1) + (g & 1), tok1 = tok0 + 2;
  const int key_off = ((t ^ ((g & 1) << 2))) * 8;

  int stage = 0;
  for (int p = first; p < p_end; p += NW) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
    __syncwarp();
    KT* kb = ring + stage * kParts * kBlock;
    KT* vb = kb + kBlock;
    if (FUSE && p == new_page) {
      // the page was fetched before its last token was known
#pragma unroll
      for (int part = 0; part < kParts; part += 2) {
        if (lane < HD / 8)
          *reinterpret_cast<uint4*>(kb + part * kBlock + new_slot * HD + (lane ^ ((new_slot & 1) << 2)) * 8) =
              *reinterpret_cast<const uint4*>(&s_new[part][lane * 8]);
#pragma unroll
        for (int i = 0; i < HD / 32; ++i)
          vb[part * kBlock + (i * 32 + lane) * kPageTokens + new_slot] = s_new[FUSE ? part + 1 : 0][i * 32 + lane];
      }
      __syncwarp();
    }
    float s0[2] = {0.f, 0.f}, s1[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < KB; ++j) {
      const int off = (32 * j) ^ key_off;        // chunk 4j + t, swizzled
      const uint4 k0 = *reinterpret_cast<const uint4*>(kb + tok0 * HD + off);
      const uint4 k1 = *reinterpret_cast<const uint4*>(kb + tok1 * HD + off);
      mma_16816<KT>(s0[0], s0[1], qa[j][0][0], qa[j][0][1], k0.x, k0.y);
      mma_16816<KT>(s0[0], s0[1], qa[j][1][0], qa[j][1][1], k0.z, k0.w);
      mma_16816<KT>(s1[0], s1[1], qa[j][0][0], qa[j][0][1], k1.x, k1.y);
      mma_16816<KT>(s1[0], s1[1], qa[j][1][0], qa[j][1][1], k1.z, k1.w);
      if (EXT) {
        const uint4 e0 = *reinterpret_cast<const uint4*>(kb + 2 * kBlock + tok0 * HD + off);
        const uint4 e1 = *reinterpret_cast<const uint4*>(kb + 2 * kBlock + tok1 * HD + off);
        mma_16816<KT>(s0[0], s0[1], qa[j][0][0], qa[j][0][1], e0.x, e0.y);
        mma_16816<KT>(s0[0], s0[1], qa[j][1][0], qa[j][1][1], e0.z, e0.w);
        mma_16816<KT>(s1[0], s1[1], qa[j][0][0], qa[j][0][1], e1.x, e1.y);
        mma_16816<KT>(s1[0], s1[1], qa[j][1][0], qa[j][1][1], e1.z, e1.w);
        mma_16816<KT>(s0[0], s0[1], ql[j][0][0], ql[j][0][1], k0.x, k0.y);
        mma_16816<KT>(s0[0], s0[1], ql[j][1][0], ql[j][1][1], k0.z, k0.w);
        mma_16816<KT>(s1[0], s1[1], ql[j][0][0], ql[j][0][1], k1.x, k1.y);
        mma_16816<KT>(s1[0], s1[1], ql[j][1][0], ql[j][1][1], k1.z, k1.w);
      }
    }
    // this lane's scores of head g: tokens 4t, 4t+1 (tile 0) and 4t+2, 4t+3 (tile 1) of the page
    const int n_valid = min(kPageTokens, ctx - p * kPageTokens);
    float sc[4] = {s0[0] * scale, s0[1] * scale, s1[0] * scale, s1[1] * scale};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (4 * t + e >= n_valid) sc[e] = -INFINITY;
    float mx = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
    const float m_new = fmaxf(m_run, mx);          // finite: token 0 of the page is always valid
    const float corr = __expf(m_run - m_new);
    float pr[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) pr[e] = __expf(sc[e] - m_new);
    l_run = l_run * corr + (pr[0] + pr[1] + pr[2] + pr[3]);
    m_run = m_new;
    uint32_t pa0, pa2, pl0 = 0u, pl2 = 0u;
    if (EXT) { pack2_split<KT>(pr[0], pr[1], pa0, pl0); pack2_split<KT>(pr[2], pr[3], pa2, pl2); }
    else { pa0 = pack2<KT>(pr[0], pr[1]); pa2 = pack2<KT>(pr[2], pr[3]); }
    // mask of the 16-bit halves of a value fragment that belong to cached tokens
    uint32_t mlo = 0xFFFFFFFFu, mhi = 0xFFFFFFFFu;
    if (n_valid < kPageTokens) {
      mlo = (4 * t < n_valid ? 0x0000FFFFu : 0u) | (4 * t + 1 < n_valid ? 0xFFFF0000u : 0u);
      mhi = (4 * t + 2 < n_valid ? 0x0000FFFFu : 0u) | (4 * t + 3 < n_valid ? 0xFFFF0000u : 0u);
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const uint2 vv = *reinterpret_cast<const uint2*>(vb + (8 * i + g) * kPageTokens + 4 * t);
      o[i][0] *= corr; o[i][1] *= corr;
      mma_16816<KT>(o[i][0], o[i][1], pa0, pa2, vv.x & mlo, vv.y & mhi);
      if (EXT) {
        const uint2 vl = *reinterpret_cast<const uint2*>(vb + 2 * kBlock + (8 * i + g) * kPageTokens + 4 * t);
        mma_16816<KT>(o[i][0], o[i][1], pl0, pl2, vv.x & mlo, vv.y & mhi);
        mma_16816<KT>(o[i][0], o[i][1], pa0, pa2, vl.x & mlo, vl.y & mhi);
      }
    }
    __syncwarp();                                // every lane has read the buffer
    fetch_next(stage);
    stage = stage + 1 == kStages ? 0 : stage + 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();                               // the ring is free: the outputs take its place
  // the 4 lanes of a row hold partial sums of l
  l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 1);
  l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 2);
  if (t == 0) { s_m[warp][g] = m_run; s_l[warp][g] = l_run; }
#pragma unroll
  for (int i = 0; i < NT; ++i) *reinterpret_cast<float2*>(&s_o[warp][g][8 * i + 2 * t]) = make_float2(o[i][0], o[i][1]);
  // Cluster mode: rank r of n merges the outputs [r * per, r * per + per) of the G x HD; every CTA leaves its partial of
  // them (and its max and sum per head) in r's shared memory, outside the ring, which r may still be reading pages from.
  constexpr int kRecv = CL ? 8 * HD : 4;
  __shared__ __align__(16) float r_o[kRecv + (CL ? 4 * kClusterSplits : 0)];
  __shared__ float2 r_ml[CL ? kClusterSplits : 1][8];
  const int n_rank = CL ? n_splits : 1, total = G * HD;
  const int per = 4 * ((total / 4 + n_rank - 1) / n_rank);
  if (CL) cg::this_cluster().barrier_wait();
  __syncthreads();
  for (int idx = 4 * threadIdx.x; idx < total; idx += 4 * kThreads) {
    const int gg = idx / HD, dd = idx % HD;
    float M = s_m[0][gg];
#pragma unroll
    for (int w = 1; w < NW; ++w) M = fmaxf(M, s_m[w][gg]);
    float L = 0.f, O[4] = {0.f, 0.f, 0.f, 0.f};
    if (M > -INFINITY) {
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float e = __expf(s_m[w][gg] - M);
        const float4 v = *reinterpret_cast<const float4*>(&s_o[w][gg][dd]);
        L += s_l[w][gg] * e;
        O[0] += v.x * e; O[1] += v.y * e; O[2] += v.z * e; O[3] += v.w * e;
      }
    }
    const int h = h0 + gg;
    if (CL) {
      const int r = idx / per;
      *reinterpret_cast<float4*>(cg::this_cluster().map_shared_rank(r_o, r) + split * per + idx - r * per) = make_float4(O[0], O[1], O[2], O[3]);
      if (dd < 4 * n_rank) *cg::this_cluster().map_shared_rank(&r_ml[split][gg], dd / 4) = make_float2(M, L);
    } else if (n_splits == 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) O[i] /= L;
      store_operand4_any<OT>(out, out_lo, ((size_t)slot * H + h) * HD + dd, O);
    } else {
      const size_t base = ((size_t)slot * H + h) * n_splits + split;
      store_operand4_any<float>(part_o, nullptr, base * HD + dd, O);     // the scratch is a caller's too
      if (dd == 0) { part_ml[base * 2] = M; part_ml[base * 2 + 1] = L; }
    }
  }
  if (CL) {
    // Every CTA of the cluster gets here (the early returns above depend on the slot alone, which the cluster shares),
    // and none touches another's shared memory after the barrier.
    cg::this_cluster().sync();
    const int idx = split * per + threadIdx.x, end = min(total, (split + 1) * per);
    for (int k = idx; k < end; k += kThreads) {
      const int gg = k / HD, dd = k % HD;
      float2 ml[kClusterSplits];
      float M = -INFINITY, L = 0.f, O = 0.f;
#pragma unroll
      for (int r = 0; r < kClusterSplits; ++r) {
        ml[r] = r < n_rank ? r_ml[CL ? r : 0][gg] : make_float2(-INFINITY, 0.f);
        M = fmaxf(M, ml[r].x);
      }
#pragma unroll
      for (int r = 0; r < kClusterSplits; ++r) {
        const float e = __expf(ml[r].x - M);     // a split without pages: max -inf, weight 0; split 0 always has some
        L += ml[r].y * e;
        O += (r < n_rank ? r_o[r * per + k - split * per] : 0.f) * e;
      }
      store_operand<OT>(out, out_lo, ((size_t)slot * H + h0 + gg) * HD + dd, O / L);
    }
  }
}

// One thread per output dim.  What it costs is trips to L2, so there is one: the lists, every split's max and sum (a lane each) and its outputs are
// requested together, and whether the slot counts is looked at when they are there.  us of a launch behind the attention, 32 splits, one row of 28 heads / five rows
// of 12: four splits at a time behind the lists 8.4 / 7.3, so 2.6 / 2.9; 14-layer iterations of the 1.5B / 7B shapes, one row, 4000 tokens, 563 / 1427 -> 524 / 1335.
template <int HD, typename OT>
__global__ void __launch_bounds__(HD)
attn_merge_kernel(const float* __restrict__ part_o, const float* __restrict__ part_ml, const int32_t* __restrict__ slot_row,
                  const int32_t* __restrict__ len_or_pos, int len_offset, OT* __restrict__ out, OT* __restrict__ out_lo,
                  int H, int n_splits, const int32_t* __restrict__ n_active) {
  static_assert(kMaxSplits == 32, "a lane of a warp per split");
  RSD_PDL_SYNC();
  const int slot = blockIdx.y, h = blockIdx.x, dd = threadIdx.x, lane = threadIdx.x & 31;
  const size_t base = ((size_t)slot * H + h) * n_splits;
  const int active = n_active != nullptr ? ld_cg(n_active) : 1, row = slot_row ? ld_cg(slot_row + slot) : 0, len = ld_cg(len_or_pos + slot);
  float2 ml = make_float2(-INFINITY, 0.f);
  if (lane < n_splits) ml = make_float2(ld_cg(part_ml + (base + lane) * 2), ld_cg(part_ml + (base + lane) * 2 + 1));
  float ov[kMaxSplits];
#pragma unroll
  for (int s = 0; s < kMaxSplits; ++s) {
    ov[s] = 0.f;
    if (s < n_splits) ov[s] = ld_cg(part_o + (base + s) * HD + dd);
  }
  if (active == 0 || row < 0 || len + len_offset <= 0) return;
  float M = ml.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
  const float e = __expf(ml.x - M);              // a split without pages: max -inf, weight 0; split 0 always has some
  const float L = warp_sum(ml.y * e);
  float O = 0.f;
#pragma unroll
  for (int s = 0; s < kMaxSplits; ++s) O += ov[s] * __shfl_sync(0xFFFFFFFFu, e, s);
  store_operand<OT>(out, out_lo, ((size_t)slot * H + h) * HD + dd, O / L);
}

__global__ void decode_slots_kernel(const int32_t* slot_row, const int32_t* len_or_pos, int len_offset, int32_t* row,
                                    int32_t* pos, int B) {
  RSD_PDL_SYNC();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B) return;
  const int r = slot_row ? slot_row[i] : i;
  const int ctx = len_or_pos[i] + len_offset;
  row[i] = (r >= 0 && ctx >= 1) ? r : -1;
  pos[i] = ctx - 1;
}

// Splits of a row's context.  One wave of at most three CTAs per SM when that leaves short splits: a second, partial wave
// would double the time (16 rows x 1000-2048 tokens, 28 / 4 heads: 21 us in one wave, 29 us with eight splits).  Splits
// of 64 pages and more are worth several waves instead, since rows of different lengths then even out (64 rows x
// 4096-16384 tokens, 28 / 4 heads: 261 us in one wave, 217 us = 93 % of the copy bandwidth with eight splits).
int pick_splits(int B, int KV, int max_ctx) {
  const int ctas = B * KV, max_pages = max_ctx / kPageTokens;
  int splits = (3 * 148) / ctas;
  while (splits < kClusterSplits && max_pages / std::max(1, splits) >= 64) ++splits;
  // At least 8 pages per split: two per warp, both on their way before the wait (4 and 8 pages: 714 and 706 ms for two
  // steps of 32 rows with contexts of a few hundred tokens).  Few CTAs leave the chip idle, and a warp that walks one page, or none, is done sooner:
  // a page a split for up to eight (slot, KV head) pairs, three for up to 32.  14-layer iterations, 8 pages a split / so, us: 1.5B shape, two pairs,
  // 80 / 140 / 250 / 700 tokens 470 / 475 / 483 / 486 -> 466 / 466 / 465 / 471, four, 250 490 / 469, eight, 250 490 / 476, 16, 170 / 250 / 500 517 / 526 / 544 ->
  // 513 / 513 / 528; 7B shape, four pairs, 100 / 250 / 500 1271 / 1272 / 1265 -> 1257 / 1254 / 1256, eight, 250 1307 / 1284, 16, 170 / 250 1324 / 1315 ->
  // 1301 / 1308, 32, 170 / 250 / 500 1328 / 1356 / 1362 -> 1326 / 1329 / 1365; 64 pairs no difference.  Below six pages, or 13, one split that takes the qkv product
  // itself is the better: two pairs, five pages 468 / 473, 16 and 32 pairs, nine pages 513 / 518 and 1336 / 1347.
  int in_cluster = max_pages / 8;
  if (ctas <= 8 && max_pages >= 6) in_cluster = max_pages;
  else if (ctas <= 32 && max_pages >= 13) in_cluster = max_pages / 3;
  splits = std::max(1, std::min(splits, std::max(std::min(in_cluster, kClusterSplits), max_pages / 8)));
  splits = std::min(splits, kMaxSplits);
  // more splits than a cluster holds cost a second launch: not worth it when 8 splits of 16 or more (slot, KV head)
  // pairs already put a CTA on most SMs, nor when 8 splits leave a warp at most six pages (full at 3000 tokens 8 splits / more 528 / 517 us, but these are the most tokens that a
  // row may come to: with 200 in that room 464 / 475)
  if (splits > kClusterSplits && (ctas * kClusterSplits >= 128 || max_pages <= kClusterSplits * 24)) splits = kClusterSplits;
  if (splits <= kClusterSplits) {              // none without pages
    const int pages = (max_pages + splits - 1) / splits;
    splits = std::max(1, (max_pages + pages - 1) / std::max(1, pages));
  }
  return splits;
}

// Launch with programmatic stream serialisation and, when cluster_z > 1, clusters of cluster_z CTAs along z.
template <typename... KArgs, typename... Args>
cudaError_t launch_decode(void (*kernel)(KArgs...), dim3 grid, int threads, int cluster_z, int smem, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 1;
  if (cluster_z > 1) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = (unsigned)cluster_z;
    cfg.numAttrs = 2;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(std::forward<Args>(args))...);
}

}  // namespace

size_t attn_decode_scratch_bytes(int B, int H, int hd, int max_ctx) {
  (void)max_ctx;
  const size_t partials = (size_t)B * H * kMaxSplits * (hd + 2) * sizeof(float);
  return sizeof(int32_t) * 2 * (size_t)B + 256 + partials;
}

// Whether a pass that takes the qkv product runs one CTA of sixteen warps per (slot, KV head): 97 to 148 of them, one per SM and no cluster,
// and few enough pages that a warp walks four at most.  14-layer iterations, us, split contexts with a rotation kernel ahead / so:
// 64 rows, 12 / 2 heads, 256 cached tokens 849 / 773, 500 tokens 844 / 805; 32 rows, 28 / 4 heads 1631 / 1598 and 1748 / 1725; near the lower
// limit 49 rows, 12 / 2 heads, 100 and 256 tokens 747 / 730 and 829 / 787, 100 rows, 8 / 1 heads 597 / 544, 25 rows, 28 / 4 heads 1588 / 1589, 13 rows, 64 / 8
// heads (8 layers) 2804 / 2740, 16 / 8 heads of 64 221 / 207.  Groups of one head mostly gain (8 layers: 37 rows, 4 / 4 heads, 420 tokens 282 / 245, 18
// rows, 8 / 8, 160 tokens 239 / 228) but not all (13 rows, 8 / 8, 64, 320 and 480 tokens 209 / 210, 236 / 242 and 261 / 250; 50 rows, 2 / 2, 64 tokens 198 / 203).  With
// fewer (slot, KV head) pairs nothing or a loss (32 rows, 12 / 2 heads, 500 tokens 688 / 703), with more, four warps are better (64 rows, 28 / 4
// heads 1951 / 2031).  Heads of 128 dims spill 108 bytes at the 128 registers that 512 threads leave; in those times.
static bool wide_ctas(int kv_dtype, int rows, int KV, int max_ctx) {
  return kv_dtype == 2 && rows * KV > 96 && rows * KV <= 148 && max_ctx <= 64 * kPageTokens;
}

bool attn_decode_takes_qkv(int kv_dtype, int out_dtype, int B, int H, int KV, int max_ctx, int active_rows, int new_tokens) {
  // With the context split over a cluster every CTA would add up the query for itself, or wait for its share from the
  // others: a rotation kernel ahead is faster there (iteration of 14 layers, 12 / 2 heads: 525 us at one row and 739 at 32
  // against 583 and 794; at 128 rows, in one split, 1275 with the rotation kernel and 1206 without).
  const int rows = active_rows > 0 ? std::min(active_rows, B) : B;
  return kv_dtype >= 2 && H / KV <= 8 && out_dtype == 1 && new_tokens == 1 &&
         (wide_ctas(kv_dtype, rows, KV, max_ctx) || pick_splits(rows, KV, max_ctx) == 1);
}

cudaError_t launch_attn_decode(int kv_dtype, const float* q, const void* pool_layer, const int32_t* page_table,
                               int max_pages, const int32_t* slot_row, const int32_t* len_or_pos, int len_offset,
                               void* out, void* out_lo, int out_dtype, int B, int H, int KV, int hd, int max_ctx,
                               void* scratch, size_t scratch_bytes, const int32_t* n_active, cudaStream_t s, int active_rows,
                               int new_tokens, const QkvSource* qkv) {
  if (B <= 0) return cudaSuccess;
  if (!scratch || scratch_bytes < attn_decode_scratch_bytes(B, H, hd, max_ctx)) return cudaErrorInvalidValue;
  const int G = H / KV;
  int32_t* row = (int32_t*)scratch;
  int32_t* pos = row + B;
  if (qkv != nullptr && !attn_decode_takes_qkv(kv_dtype, out_dtype, B, H, KV, max_ctx, active_rows, new_tokens)) return cudaErrorInvalidValue;
  if (kv_dtype == 0 || G > 8) {
    // fp32 caches and wide groups take the generic kernel
    PassView p{nullptr, slot_row, len_or_pos, B, n_active};
    if (!slot_row || len_offset != 1) {        // else the slots are a pass's rows and positions already
      RSD_LAUNCH((decode_slots_kernel), (B + 255) / 256, 256, 0, s, slot_row, len_or_pos, len_offset, row, pos, B);
      launched(1);
      p = PassView{nullptr, row, pos, B, nullptr};   // written a kernel ago: nothing to read ahead of the wait
    }
    KvView kv{const_cast<void*>(pool_layer), page_table, max_pages, kv_dtype == 3 ? 1 : 0};
    return launch_attn_generic(kv_dtype == 3 ? 2 : kv_dtype, q, p, kv, out, out_lo, out_dtype, H, KV, hd, s);
  }
  const size_t head = ((sizeof(int32_t) * 2 * (size_t)B + 255) / 256) * 256;
  float* part_ml = (float*)((char*)scratch + head);
  float* part_o = part_ml + (size_t)B * H * kMaxSplits * 2;
  const int rows = active_rows > 0 ? std::min(active_rows, B) : B;
  const bool wide = qkv != nullptr && wide_ctas(kv_dtype, rows, KV, max_ctx);
  const int splits = wide ? 1 : pick_splits(rows, KV, max_ctx);
  const bool clustered = splits >= 2 && splits <= kClusterSplits;
  dim3 grid(KV, B, splits);
#define RSD_DEC_K(HD, KT, OT, EXTV, CLV, FUSEV, NW)                                                                    \
  do {                                                                                                               \
    static OncePerDevice configured_;                                                                                \
    constexpr int smem_ = DecCfg<HD, EXTV, NW>::kRingBytes;                                                          \
    const cudaError_t set_ = allow_smem(configured_, attn_decode_kernel<HD, KT, OT, EXTV, CLV, FUSEV, NW>, smem_);    \
    if (set_ != cudaSuccess) return set_;                                                                            \
    (void)launch_decode(attn_decode_kernel<HD, KT, OT, EXTV, CLV, FUSEV, NW>, grid, 32 * NW, clustered ? splits : 1, smem_, s, \
                        FUSEV ? qkv->qkv : q, (KT*)pool_layer, page_table, max_pages, slot_row, len_or_pos, len_offset, (OT*)out, \
                        (OT*)out_lo, part_o, part_ml, H, KV, splits, n_active, new_tokens, FUSEV ? qkv->pending.partials : nullptr, \
                        FUSEV ? qkv->pending.splits : 1, FUSEV ? qkv->rope : nullptr);                               \
  } while (0)
#define RSD_DEC(HD, KT, OT, EXTV, FUSEV)                                                                              \
  do {                                                                                                               \
    if (clustered) RSD_DEC_K(HD, KT, OT, EXTV, true, false, 4);                                                       \
    else RSD_DEC_K(HD, KT, OT, EXTV, false, FUSEV, 4);                                                                \
    if (splits > 1 && !clustered)                                                                                    \
      RSD_LAUNCH((attn_merge_kernel<HD, OT>), dim3(H, B), HD, 0, s, part_o, part_ml, slot_row, len_or_pos, len_offset, (OT*)out, \
                                                          (OT*)out_lo, H, splits, n_active);                         \
  } while (0)
#define RSD_DEC_O(HD, KT, EXTV)                                                                                       \
  do {                                                                                                               \
    if (wide && !EXTV) RSD_DEC_K(HD, KT, __nv_bfloat16, false, false, true, 16);                                      \
    else if (qkv != nullptr) RSD_DEC(HD, KT, __nv_bfloat16, EXTV, true);                                              \
    else if (out_dtype == 1) RSD_DEC(HD, KT, __nv_bfloat16, EXTV, false);                                             \
    else RSD_DEC(HD, KT, float, EXTV, false);                                                                         \
  } while (0)
  // (a model of the engine has a 16-bit cache of fp16: bf16 caches come through the attention entry point alone)
  if (kv_dtype == 3) { if (hd == 128) RSD_DEC_O(128, __half, true); else RSD_DEC_O(64, __half, true); }
  else if (kv_dtype == 2) { if (hd == 128) RSD_DEC_O(128, __half, false); else RSD_DEC_O(64, __half, false); }
  else if (hd == 128) { if (out_dtype == 1) RSD_DEC(128, __nv_bfloat16, __nv_bfloat16, false, false); else RSD_DEC(128, __nv_bfloat16, float, false, false); }
  else { if (out_dtype == 1) RSD_DEC(64, __nv_bfloat16, __nv_bfloat16, false, false); else RSD_DEC(64, __nv_bfloat16, float, false, false); }
#undef RSD_DEC_O
#undef RSD_DEC
#undef RSD_DEC_K
  return launched(splits > 1 && !clustered ? 2 : 1);
}

}  // namespace rsd
