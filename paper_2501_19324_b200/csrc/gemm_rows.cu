// Decode products of few rows without a K split over CTAs, each in one launch with the small step behind it (bf16 weights x hi + lo
// operand pairs, up to eight rows, sixteen weight rows a CTA):
//   kResidual   x += in W^T; hi + lo = x * gain, the operand of the next product, and the sums of squares of x per eight columns for
//               that product's RowScale
//   kQkv        queries, keys and values: RMSNorm's denominator, rotation, queries to q_out, keys and values to the row's page
// A K split leaves partial sums that a launch of its own adds up (2.0-2.7 us); here the sums stay in the CTA.  The price is that every CTA
// reads the whole operand, so it pays while that is little (rows_gemm_pays).  Bound by latency: wait, operand from L2, a few
// hundred cycles of products, sums over the warps, store; the weights are there before the wait as far as the slots reach.
// Iterations us, before / with these: two layers of 512 columns 1 / 4 / 8 rows 51.6 / 51.9 / 54.2 -> 39.3 / 40.8 / 41.8, 14 layers of the
// 1.5B shape at 1 / 3 rows 503 / 509 -> 482 / 485.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace rsd {

namespace {

enum RowsEpilogue { kResidual, kQkv };
constexpr int kRowsMax = 8, kRowsWarps = 8, kRowsStages = 6, kChunk = 64, kGroups = 2;   // kGroups: of eight weight rows a CTA

struct RowsArgs {
  // kResidual
  float* x;
  const __nv_bfloat16* gain;
  __nv_bfloat16 *hi, *lo;
  float* ssq;
  // kQkv
  RowScale rs;
  PassView p;
  float* q_out;
  __half* pool;
  const int32_t* page_table;
  const float2* rope;
  int max_pages, H, KV, hd, ext;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The warps of a CTA share K in chunks of 64.  A chunk of a group of eight weight rows is four MMAs of 16 x 8 x 16: the operand's eight hi
// and eight lo rows are the 16 rows of the left side, the weight rows the eight columns.  (tcgen05 has no tile this narrow, and these few
// products are not what the time goes to.)  The order of the 32 values of K inside a half chunk is permuted for both alike, so that a
// lane's share of either is one 16-byte piece of a row; every lane copies the pieces that it multiplies itself, through slots of
// shared memory of its own: nothing to synchronise, no bank conflicts.
// LONG: more than kFold chunks a warp.  The MMAs' own additions are not rounded to nearest, so a long chain of them drifts: every kFold chunks the
// accumulators go into sums that are (relative error against fp64, K split / one chain / so: 2 x 512 x 8960 2.0 / 4.6 / 1.3e-7, 1 x 3584 x
// 3584 2.8 / 1.7 / 1.0e-7; at 1536 one chain of three chunks, 1.1 / 0.8).  The short form is one chain: with the sums in its loop an iteration
// of 14 layers of the 1.5B shape at one row took 489 us instead of 487, of the small models at eight rows 68.0 instead of 67.5.
constexpr int kFold = 4;

template <int EPI, bool LONG>
__global__ void __launch_bounds__(32 * kRowsWarps)
gemm_rows_kernel(const __nv_bfloat16* W, const __nv_bfloat16* in, const __nv_bfloat16* in_lo, int M, int K, int n_stages,
                 const int32_t* n_active, const __grid_constant__ RowsArgs a) {
  RSD_PDL_TRIGGER();
  const int active = n_active != nullptr ? ld_cg(n_active) : 1;
  extern __shared__ __align__(16) uint8_t ring_raw[];
  __shared__ float red[kRowsWarps][kGroups][8][8];
  __shared__ float s_inv[kRowsMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int chunks = K / kChunk, mine = (chunks - warp + kRowsWarps - 1) / kRowsWarps;
  const int x_part = M * 64, stage_bytes = kGroups * 1024 + 4 * x_part;      // weights; (half chunk, hi | lo) of the operand
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(ring_raw) + warp * n_stages * stage_bytes;
  const int half = EPI == kQkv ? a.hd / 2 : 0, per_head = EPI == kQkv ? a.hd / 8 : 1;
  const __nv_bfloat16* w_row[kGroups];
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    const int unit = blockIdx.x * kGroups + u;               // kQkv: four dims of a head and the four that they turn with
    const int row = EPI == kQkv ? (unit / per_head) * a.hd + (unit % per_head) * 4 + (g & 3) + (g >> 2) * half : unit * 8 + g;
    w_row[u] = W + (size_t)row * K + 8 * t;
  }
  auto fetch_w = [&](int i, int stage) {
    if (i < mine) {
      const int k0 = (i * kRowsWarps + warp) * kChunk;
#pragma unroll
      for (int u = 0; u < kGroups; ++u)
#pragma unroll
        for (int j = 0; j < 2; ++j) cp_async16(ring + stage * stage_bytes + (u * 2 + j) * 512 + lane * 16, w_row[u] + k0 + 32 * j);
    }
  };
  const bool has_row = g < M;
  const __nv_bfloat16 *xh = in + (size_t)(has_row ? g : 0) * K + 8 * t, *xl = in_lo + (size_t)(has_row ? g : 0) * K + 8 * t;
  auto fetch_x = [&](int i, int stage) {
    if (i < mine && has_row) {
      const int k0 = (i * kRowsWarps + warp) * kChunk;
      const uint32_t dst = ring + stage * stage_bytes + kGroups * 1024 + lane * 16;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        cp_async16(dst + 2 * j * x_part, xh + k0 + 32 * j);
        cp_async16(dst + (2 * j + 1) * x_part, xl + k0 + 32 * j);
      }
    }
  };
  auto commit = [&]() { asm volatile("cp.async.commit_group;" ::: "memory"); };
  if (n_active == nullptr) RSD_PDL_WAIT();     // outside a decode pass the weights and the lists may be an earlier kernel's output
#pragma unroll
  for (int i = 0; i < kRowsStages; ++i) { fetch_w(i, i); commit(); }         // (a warp with fewer chunks has fewer slots: mine <= n_stages)
  // what the epilogue needs beside the product: of the pass's lists and the weights before the wait, the rest after it
  const int em = EPI == kQkv ? (threadIdx.x >> 2) & 7 : (threadIdx.x >> 3) & 7, en = EPI == kQkv ? threadIdx.x & 3 : threadIdx.x & 7;
  const int eu = EPI == kQkv ? threadIdx.x >> 5 : threadIdx.x >> 6, e_unit = blockIdx.x * kGroups + eu;
  const bool owner = eu < kGroups && em < M;
  float gain = 0.f, old = 0.f, sq[4];
  float2 cs = make_float2(1.f, 0.f);
  int row = -1, pos = 0, page = 0;
  const int head = e_unit / per_head, dim = (e_unit % per_head) * 4 + en;      // kQkv: this thread's pair is (dim, dim + half)
  const int d = gridDim.x * kGroups * 8;
  const size_t o = (size_t)em * d + e_unit * 8 + en;
  if (owner) {
    if (EPI == kResidual) {
      gain = to_f32(a.gain[e_unit * 8 + en]);
    } else {
      row = ld_cg(a.p.tok_row + em);
      pos = ld_cg(a.p.tok_pos + em);
      if (row >= 0) {
        if (head >= a.H) page = ld_cg(a.page_table + (size_t)row * a.max_pages + pos / kPageTokens);
        if (head < a.H + a.KV) cs = a.rope[(size_t)pos * half + dim];
      }
    }
  }
  RSD_PDL_WAIT();
  if (active == 0) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    return;
  }
#pragma unroll
  for (int i = 0; i < kRowsStages; ++i) { fetch_x(i, i); commit(); }
  if (EPI == kResidual) {
    if (owner) old = a.x[o];
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) sq[c] = warp < M && c * 32 + lane < a.rs.n_chunks ? a.rs.ssq[(size_t)warp * a.rs.n_chunks + c * 32 + lane] : 0.f;
  }
  float acc[kGroups][2][4], sum[LONG ? kGroups : 1][2] = {};
#pragma unroll
  for (int u = 0; u < kGroups; ++u)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[u][j][i] = 0.f;
  int stage = 0;
  for (int i = 0; i < mine; ++i) {
    // groups in order: the weights of the first chunks, their operands, then one of both per chunk
    asm volatile("cp.async.wait_group %0;" ::"n"(kRowsStages - 1) : "memory");
    const uint32_t at = ring + stage * stage_bytes;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      uint4 h = make_uint4(0, 0, 0, 0), l = make_uint4(0, 0, 0, 0);
      if (has_row) {
        h = lds128(at + kGroups * 1024 + lane * 16 + 2 * j * x_part);
        l = lds128(at + kGroups * 1024 + lane * 16 + (2 * j + 1) * x_part);
      }
#pragma unroll
      for (int u = 0; u < kGroups; ++u) {
        const uint4 w = lds128(at + (u * 2 + j) * 512 + lane * 16);
        mma_bf16(acc[u][j], h.x, l.x, h.y, l.y, w.x, w.y);
        mma_bf16(acc[u][j], h.z, l.z, h.w, l.w, w.z, w.w);
      }
    }
    fetch_w(i + kRowsStages, stage);
    fetch_x(i + kRowsStages, stage);
    commit();
    stage = stage + 1 == kRowsStages ? 0 : stage + 1;
    if (LONG && i % kFold == kFold - 1) {
#pragma unroll
      for (int u = 0; u < kGroups; ++u) {
#pragma unroll
        for (int k = 0; k < 2; ++k) sum[LONG ? u : 0][k] += (acc[u][0][k] + acc[u][1][k]) + (acc[u][0][k + 2] + acc[u][1][k + 2]);
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[u][j][k] = 0.f;
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
  for (int u = 0; u < kGroups; ++u) {
    float2 v = make_float2((acc[u][0][0] + acc[u][1][0]) + (acc[u][0][2] + acc[u][1][2]), (acc[u][0][1] + acc[u][1][1]) + (acc[u][0][3] + acc[u][1][3]));
    if (LONG) v = make_float2(sum[LONG ? u : 0][0] + v.x, sum[LONG ? u : 0][1] + v.y);
    *reinterpret_cast<float2*>(&red[warp][u][g][2 * t]) = v;
  }
  if (EPI == kQkv) {
    float s = (sq[0] + sq[1]) + (sq[2] + sq[3]);
    if (warp < M)
      for (int c = 128 + lane; c < a.rs.n_chunks; c += 32) s += a.rs.ssq[(size_t)warp * a.rs.n_chunks + c];
    s = warp_sum(s);
    if (lane == 0) s_inv[warp] = rsqrtf(s * a.rs.inv_d + a.rs.eps);
  }
  __syncthreads();
  if (EPI == kResidual) {
    if (threadIdx.x >= 64 * kGroups) return;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kRowsWarps; ++w) v += red[w][eu][em][en];
    v += old;
    if (owner) {
      a.x[o] = v;
      store_operand<__nv_bfloat16>(a.hi, a.lo, o, v * gain);
    }
    float ss = v * v;
#pragma unroll
    for (int k = 4; k > 0; k >>= 1) ss += __shfl_xor_sync(0xFFFFFFFFu, ss, k);
    if (owner && en == 0) a.ssq[(size_t)em * (d / 8) + e_unit] = ss;
  } else {
    if (!owner || row < 0) return;
    float lo = 0.f, up = 0.f;
#pragma unroll
    for (int w = 0; w < kRowsWarps; ++w) { lo += red[w][eu][em][en]; up += red[w][eu][em][en + 4]; }
    lo *= s_inv[em]; up *= s_inv[em];
    if (head < a.H + a.KV) {
      const float r = rotate_lo(lo, up, cs);
      up = rotate_hi(lo, up, cs);
      lo = r;
    }
    if (head < a.H) {
      float* q = a.q_out + ((size_t)em * a.H + head) * a.hd + dim;
      q[0] = lo;
      q[half] = up;
      return;
    }
    // the page as rope_kv_kernel lays it out
    const size_t block = (size_t)a.KV * kPageTokens * a.hd;
    __half* at = a.pool + (size_t)page * (a.ext ? 4 : 2) * block;
    const int slot = pos % kPageTokens;
    size_t gap = half;
    if (head < a.H + a.KV) {
      at += ((size_t)(head - a.H) * kPageTokens + slot) * a.hd + dim;
    } else {
      at += block + ((size_t)(head - a.H - a.KV) * a.hd + dim) * kPageTokens + slot;
      gap *= kPageTokens;
    }
    const __half l16 = __float2half_rn(lo), u16 = __float2half_rn(up);
    at[0] = l16;
    at[gap] = u16;
    if (a.ext) {
      at[2 * block] = __float2half_rn(lo - __half2float(l16));
      at[2 * block + gap] = __float2half_rn(up - __half2float(u16));
    }
  }
}

template <int EPI>
cudaError_t launch_rows(const void* W, const void* in, const void* in_lo, int M, int N, int K, const int32_t* n_active, const RowsArgs& a, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (!rows_gemm_supported(M, N, K) || !in_lo) return cudaErrorNotSupported;
  if (((uintptr_t)W & 15) || ((uintptr_t)in & 15) || ((uintptr_t)in_lo & 15)) return cudaErrorMisalignedAddress;
  const int stages = std::min(kRowsStages, (K / kChunk + kRowsWarps - 1) / kRowsWarps);    // slots; the waits count kRowsStages groups
  const int smem = kRowsWarps * stages * (kGroups * 1024 + M * 256);
  constexpr int max_smem = kRowsWarps * kRowsStages * (kGroups * 1024 + kRowsMax * 256);
#define RSD_ROWS(LONG)                                                                                                                          \
  do {                                                                                                                                          \
    static OncePerDevice configured;                                                                                                            \
    const cudaError_t set = allow_smem(configured, gemm_rows_kernel<EPI, LONG>, max_smem);                                                       \
    if (set != cudaSuccess) return set;                                                                                                         \
    RSD_LAUNCH((gemm_rows_kernel<EPI, LONG>), N / (8 * kGroups), 32 * kRowsWarps, smem, s, (const __nv_bfloat16*)W, (const __nv_bfloat16*)in,    \
               (const __nv_bfloat16*)in_lo, M, K, stages, n_active, a);                                                                          \
  } while (0)
  if (K > kFold * kRowsWarps * kChunk) RSD_ROWS(true);
  else RSD_ROWS(false);
#undef RSD_ROWS
  return launched(1);
}

}  // namespace

bool rows_gemm_supported(int M, int N, int K) {
  return M >= 1 && M <= kRowsMax && N >= 8 * kGroups && N % (8 * kGroups) == 0 && K >= kChunk && K % kChunk == 0;
}

// What all CTAs read of the operand, N / 16 times M rows of 4 K bytes, within 3.5 MB; of the down projection, whose K split has long chains
// to hide its sums behind, within 1.7 MB.  Iterations us, K split / here: qkv and wo of 14 layers, 1.5B shape, 3 rows (2.4 and 1.8 MB) 510 / 486,
// 4 rows (3.1 and 2.4) 517 / 492; 7B shape, 1 row: wo (3.2 MB) 1311 / 1289, with qkv (4.1 MB) 1308; wo, 2 rows (6.4 MB) 1342 / 1367;
// down of 2 layers, 512 x 1408, 8 rows (1.4 MB) 45.5 / 41.8, 3 layers, 768 x 2048, 4 rows (1.6 MB) 65.2 / 60.8; 14 layers, 1536 x 8960, 1 row
// (3.4 MB) 509 / 528.
bool rows_gemm_pays(int M, int N, int K, bool long_k) {
  return rows_gemm_supported(M, N, K) && (size_t)(N / (8 * kGroups)) * M * K * 4 <= (long_k ? 1700000u : 3500000u);
}

cudaError_t launch_gemm_rows_residual(const void* W, const void* in, const void* in_lo, float* x, const void* gain, void* hi, void* lo,
                                      float* ssq, int M, int d, int K, const int32_t* n_active, cudaStream_t s) {
  RowsArgs a{};
  a.x = x; a.gain = (const __nv_bfloat16*)gain; a.hi = (__nv_bfloat16*)hi; a.lo = (__nv_bfloat16*)lo; a.ssq = ssq;
  return launch_rows<kResidual>(W, in, in_lo, M, d, K, n_active, a, s);
}

cudaError_t launch_gemm_rows_qkv(const void* W, const void* in, const void* in_lo, RowScale rs, PassView p, float* q_out, KvView kv,
                                 const float2* rope, int H, int KV, int hd, int K, cudaStream_t s) {
  RowsArgs a{};
  a.rs = rs; a.p = p; a.q_out = q_out; a.pool = (__half*)kv.pool_layer; a.page_table = kv.page_table; a.rope = rope;
  a.max_pages = kv.max_pages; a.H = H; a.KV = KV; a.hd = hd; a.ext = kv.v_extra;
  return launch_rows<kQkv>(W, in, in_lo, p.T, (H + 2 * KV) * hd, K, p.n_active, a, s);
}

}  // namespace rsd
