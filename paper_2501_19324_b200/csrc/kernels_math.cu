// Element-wise, normalisation, rotary, SIMT GEMV, attention, sampling and reward kernels of the RSD
// step loop (sm_100a).  The residual stream and every reduction are fp32; weights, GEMM inputs and
// the KV cache are stored in the model's element type (fp32 or bfloat16).
#include "common.cuh"
#include "kernels.cuh"
#include "sampling.cuh"

namespace rsd {

#define RSD_SKIP_IF_IDLE(n_active) \
  if ((n_active) != nullptr && *(n_active) == 0) return;

// ---------------------------------------------------------------------------------------------
// Embedding gather: x[t, :] = E[tok_id[t], :]
// ---------------------------------------------------------------------------------------------
template <typename WT>
__global__ void embed_kernel(const WT* __restrict__ E, PassView p, float* __restrict__ x, int d) {
  RSD_PDL_SYNC_LATE();
  RSD_SKIP_IF_IDLE(p.n_active);
  const int t = blockIdx.x;
  if (p.tok_row[t] < 0) return;
  const WT* src = E + (size_t)p.tok_id[t] * d;
  float* dst = x + (size_t)t * d;
  constexpr int N = Vec16<WT>::N;
  for (int i = threadIdx.x * N; i < d; i += blockDim.x * N) {
    Vec16<WT> v;
    v.load(src + i);
#pragma unroll
    for (int j = 0; j < N; ++j) dst[i + j] = v.v[j];
  }
}

cudaError_t launch_embed(int dtype, const void* embed, PassView p, float* x, int d, cudaStream_t s) {
  if (p.T <= 0) return cudaSuccess;
  if (dtype == 1) RSD_LAUNCH((embed_kernel<__nv_bfloat16>), p.T, 128, 0, s, (const __nv_bfloat16*)embed, p, x, d);
  else RSD_LAUNCH((embed_kernel<float>), p.T, 128, 0, s, (const float*)embed, p, x, d);
  return launched(1);
}

// ... of a decode pass of a bf16 model, with the first layer's un-normalised norm operand and sums of squares (see reduce_norm_kernel):
// one block per (token, 256-column chunk).  A launch of 1.4-1.7 us less an iteration.
__global__ void __launch_bounds__(64)
embed_norm_kernel(const __nv_bfloat16* __restrict__ E, PassView p, float* __restrict__ x, const __nv_bfloat16* __restrict__ gain,
                  __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo, float* __restrict__ ssq, int d) {
  RSD_PDL_SYNC_LATE();
  RSD_SKIP_IF_IDLE(p.n_active);
  __shared__ float red[2];
  const int t = blockIdx.y, col = blockIdx.x * 256 + threadIdx.x * 4;
  if (p.tok_row[t] < 0) return;
  float ss = 0.f;
  if (col < d) {
    float v[4], y[4];
    __align__(8) __nv_bfloat16 e[4];
    *reinterpret_cast<uint2*>(e) = *reinterpret_cast<const uint2*>(E + (size_t)p.tok_id[t] * d + col);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = to_f32(e[i]);
      y[i] = v[i] * to_f32(gain[col + i]);       // (a caller's gains may start anywhere)
    }
    const size_t o = (size_t)t * d + col;
    *reinterpret_cast<float4*>(x + o) = make_float4(v[0], v[1], v[2], v[3]);
    store_operand4<__nv_bfloat16>(hi, lo, o, y);
    ss = v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  }
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x == 0) ssq[(size_t)t * gridDim.x + blockIdx.x] = red[0] + red[1];
}

cudaError_t launch_embed_norm(const void* embed, PassView p, float* x, const void* gain, void* hi, void* lo, float* ssq, int d, cudaStream_t s) {
  if (p.T <= 0) return cudaSuccess;
  if (d % 4 != 0) return cudaErrorInvalidValue;
  RSD_LAUNCH((embed_norm_kernel), dim3(norm_chunks(d), p.T), 64, 0, s, (const __nv_bfloat16*)embed, p, x, (const __nv_bfloat16*)gain,
             (__nv_bfloat16*)hi, (__nv_bfloat16*)lo, ssq, d);
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// RMSNorm: out = x * gain / sqrt(mean(x^2) + eps), one block per token, x kept in registers
// ---------------------------------------------------------------------------------------------
// Bound by DRAM in the dense passes (8192 x 3584: 117 MB in, 59 MB out: 29.5 us from and to L2).  A thread keeps VECS
// vectors of four elements; the block has as many threads as that takes (launch_rmsnorm), so that narrow rows leave none idle.

// The roundings spelled out: the sum does not depend on what the compiler would fuse.
__device__ __forceinline__ float sum_squares(float4 v) { return fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.x, v.x, __fmul_rn(v.y, v.y)))); }

template <typename OT, typename GT>
__device__ __forceinline__ void norm_store(OT* out, OT* out_lo, size_t o, float4 v, float inv, const GT* gain) {
  const float y[4] = {v.x * inv * to_f32(gain[0]), v.y * inv * to_f32(gain[1]), v.z * inv * to_f32(gain[2]), v.w * inv * to_f32(gain[3])};
  store_operand4_any<OT>(out, out_lo, o, y);
}

template <typename OT, typename GT, int VECS>
__global__ void rmsnorm_kernel(const float* x, const GT* __restrict__ gain, OT* out, OT* out_lo, int d, float eps,
                               const int32_t* n_active) {
  RSD_PDL_SYNC_UNLESS_IDLE(n_active);
  __shared__ float red[33];
  const int t = blockIdx.x;
  const float* xr = x + (size_t)t * d;
  float ss = 0.f;
  // the row stays in registers between the two halves (wider ones are read again)
  float4 keep[VECS];
#pragma unroll
  for (int k = 0; k < VECS; ++k) {
    const int i = (k * blockDim.x + threadIdx.x) * 4;
    if (i < d) keep[k] = *reinterpret_cast<const float4*>(xr + i);
  }
#pragma unroll
  for (int k = 0; k < VECS; ++k) {
    const float4 v = keep[k];
    if ((k * (int)blockDim.x + (int)threadIdx.x) * 4 < d) ss += sum_squares(v);
  }
  for (int i = (VECS * blockDim.x + threadIdx.x) * 4; i < d; i += blockDim.x * 4) {
    ss += sum_squares(*reinterpret_cast<const float4*>(xr + i));
  }
  ss = block_sum(ss, red);
  const float inv = rsqrtf(ss / (float)d + eps);
  const size_t o = (size_t)t * d;
#pragma unroll
  for (int k = 0; k < VECS; ++k) {
    const int i = (k * blockDim.x + threadIdx.x) * 4;
    if (i < d) norm_store<OT>(out, out_lo, o + i, keep[k], inv, gain + i);
  }
  for (int i = (VECS * blockDim.x + threadIdx.x) * 4; i < d; i += blockDim.x * 4)
    norm_store<OT>(out, out_lo, o + i, *reinterpret_cast<const float4*>(xr + i), inv, gain + i);
}

// bf16 -> fp16, element by element (n a multiple of 8: weight matrices are).
__global__ void bf16_to_f16_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, size_t n8) {
  RSD_PDL_SYNC();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += (size_t)gridDim.x * blockDim.x) {
    uint4 v = src[i];
    const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&v);
    uint4 o;
    __half2* h = reinterpret_cast<__half2*>(&o);
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = __floats2half2_rn(__low2float(b[k]), __high2float(b[k]));
    dst[i] = o;
  }
}

cudaError_t launch_bf16_to_f16(const void* src, void* dst, size_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  if (n % 8 != 0 || ((uintptr_t)src & 15) || ((uintptr_t)dst & 15)) return cudaErrorInvalidValue;
  const size_t n8 = n / 8;
  const int blocks = (int)std::min<size_t>((n8 + 255) / 256, 148 * 16);
  RSD_LAUNCH((bf16_to_f16_kernel), blocks, 256, 0, s, (const uint4*)src, (uint4*)dst, n8);
  return launched(1);
}

cudaError_t launch_rmsnorm(int dtype, const float* x, const void* gain, void* out, void* out_lo, int T, int d, float eps,
                           const int32_t* n_active, cudaStream_t s, bool out_f16) {
  if (T <= 0) return cudaSuccess;
  // As few threads as keep the row in registers: more rows are in flight on an SM.  Up to 1024 columns a vector a thread (64 to
  // 256 threads), up to 4096 two or four and 256 threads, beyond 512 threads: 8192 x 256, bf16, 11.9 us with 256 threads and four
  // vectors, 9.0 with 64 and one; 2048 x 512 4.2 / 3.3, 8192 x 1536 16.0 / 13.2.
#define RSD_NORM(OT, GT, VECS, threads, lo) RSD_LAUNCH((rmsnorm_kernel<OT, GT, VECS>), T, threads, 0, s, x, (const GT*)gain, (OT*)out, lo, d, eps, n_active)
#define RSD_NORM_D(OT, GT, lo)                                       \
  do {                                                               \
    if (d <= 1024) RSD_NORM(OT, GT, 1, d <= 256 ? 64 : (d <= 512 ? 128 : 256), lo); \
    else if (d <= 2048) RSD_NORM(OT, GT, 2, 256, lo);                \
    else RSD_NORM(OT, GT, 4, d <= 4096 ? 256 : 512, lo);             \
  } while (0)
  if (dtype == 1 && out_f16) RSD_NORM_D(__half, __nv_bfloat16, (__half*)nullptr);
  else if (dtype == 1) RSD_NORM_D(__nv_bfloat16, __nv_bfloat16, (__nv_bfloat16*)out_lo);
  else RSD_NORM_D(float, float, (float*)nullptr);
#undef RSD_NORM_D
#undef RSD_NORM
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// Residual update + un-normalised RMSNorm operand (decode path of bf16 models).  One block per (row,
// 256-column chunk): x (+)= sum of the K-split partial sums of the GEMM that feeds the residual stream;
// hi + lo = x * gain (two bf16 arrays, the operand of the next GEMM); ssq[row][chunk] = sum of x^2
// over the chunk.  The next GEMM multiplies its result rows by rsqrt(sum_chunk ssq / d + eps)
// (RowScale), which is RMSNorm applied after the product instead of before it.
// ---------------------------------------------------------------------------------------------
// Bound by latency (a launch moves 1-5 MB, all of it in L2): the gain is fetched under the wait, and the partial sums are
// dealt over kSumGroups groups of 64 threads, so that up to kSumGroups * kSumAhead = 24 splits, the rule, are one
// round of loads.  The groups' sums meet in shared memory and are added in order.
constexpr int kSumAhead = 6;

__global__ void __launch_bounds__(64 * kSumGroups)
reduce_norm_kernel(const float* partials, int splits, float* x, const __nv_bfloat16* __restrict__ gain, __nv_bfloat16* hi,
                   __nv_bfloat16* lo, float* ssq, int M, int d, int n_chunks, const int32_t* n_active) {
  RSD_PDL_TRIGGER();
  __shared__ float red[2];
  __shared__ float4 s_part[kSumGroups - 1][64];
  const bool idle = n_active != nullptr && ld_cg(n_active) == 0;
  const int m = blockIdx.y, c = blockIdx.x;
  const int col = c * 256 + threadIdx.x * 4, grp = threadIdx.y;
  const size_t o = (size_t)m * d + col, stride = (size_t)M * d;
  float g[4] = {0.f, 0.f, 0.f, 0.f};
  if (col < d && grp == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) g[i] = to_f32(gain[col + i]);
  }
  RSD_PDL_WAIT();
  if (idle) return;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (col < d) {
    float4 old;
    if (grp == 0) old = *reinterpret_cast<const float4*>(x + o);
    if (splits > 1) {
      const int per = (splits + kSumGroups - 1) / kSumGroups, s_end = min(splits, (grp + 1) * per);
      for (int s0 = grp * per; s0 < s_end; s0 += kSumAhead) {
        float4 a[kSumAhead];
#pragma unroll
        for (int u = 0; u < kSumAhead; ++u)
          if (s0 + u < s_end) a[u] = ld_cg(reinterpret_cast<const float4*>(partials + (size_t)(s0 + u) * stride + o));
#pragma unroll
        for (int u = 0; u < kSumAhead; ++u)
          if (s0 + u < s_end) { v.x += a[u].x; v.y += a[u].y; v.z += a[u].z; v.w += a[u].w; }
      }
      if (grp > 0) s_part[grp - 1][threadIdx.x] = v;
    }
    if (grp == 0) { v.x += old.x; v.y += old.y; v.z += old.z; v.w += old.w; }
  }
  if (splits > 1) __syncthreads();
  if (grp > 0) return;
  float ss = 0.f;
  if (col < d) {
    if (splits > 1) {
#pragma unroll
      for (int i = 0; i < kSumGroups - 1; ++i) {
        const float4 a = s_part[i][threadIdx.x];
        v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
      }
      *reinterpret_cast<float4*>(x + o) = v;
    }
    ss = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    const float y[4] = {v.x * g[0], v.y * g[1], v.z * g[2], v.w * g[3]};
    __align__(8) __nv_bfloat16 h4[4], l4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) store_operand<__nv_bfloat16>(h4, l4, i, y[i]);
    *reinterpret_cast<uint2*>(hi + o) = *reinterpret_cast<const uint2*>(h4);
    *reinterpret_cast<uint2*>(lo + o) = *reinterpret_cast<const uint2*>(l4);
  }
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  asm volatile("bar.sync 1, 64;" ::: "memory");            // the two warps of group 0
  if (threadIdx.x == 0) ssq[(size_t)m * n_chunks + c] = red[0] + red[1];
}

cudaError_t launch_reduce_norm(const float* partials, int splits, float* x, const void* gain, void* hi, void* lo,
                               float* ssq, int M, int d, const int32_t* n_active, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (d % 4 != 0) return cudaErrorInvalidValue;
  const int n_chunks = norm_chunks(d);
  RSD_LAUNCH((reduce_norm_kernel), dim3(n_chunks, M), dim3(64, splits > 1 ? kSumGroups : 1), 0, s, partials, splits, x, (const __nv_bfloat16*)gain,
             (__nv_bfloat16*)hi, (__nv_bfloat16*)lo, ssq, M, d, n_chunks, n_active);
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// Split-K SIMT GEMV / skinny GEMM:  y[m, n] (+)= sum_k x[m, k] W[n, k]
// A block of 8 warps covers nb = 8/ks output columns; the ks warps of one column each stream a
// strided share of the row with 16-byte loads and their partial sums meet in shared memory, in a
// fixed order (deterministic).  Rows of x are taken MT at a time.
// Bound by latency at the sizes it serves (the fp32 test models: 0.3-5 MB of weights a launch, resident in L2): in a
// decode pass the first kGemvAhead weight vectors of a lane, and nearly always all of them, are requested before the
// wait for the preceding kernels, and the old y before the products.
// ---------------------------------------------------------------------------------------------
constexpr int kGemvAhead = 4;

template <typename WT, int MT, int AHEAD>
__global__ void __launch_bounds__(256)
gemv_splitk_kernel(const WT* __restrict__ W, const WT* X, const WT* X_lo, float* Y, int M, int N, int K, int ks, int accumulate,
                   const int32_t* n_active) {
  RSD_PDL_TRIGGER();
  constexpr int VN = Vec16<WT>::N;
  __shared__ float part[8][MT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = 8 / ks;
  const int col = warp / ks, split = warp % ks;
  const int n = blockIdx.x * nb + col;
  const int m0 = blockIdx.y * MT;
  const int nvec = n < N ? K / VN : 0, v0 = split * 32 + lane, step = ks * 32;
  const WT* wrow = W + (size_t)n * K;
  Vec16<WT> ahead[AHEAD > 0 ? AHEAD : 1];
  if (n_active == nullptr) RSD_PDL_WAIT();   // outside a decode pass W may be an earlier kernel's output
  const bool idle = n_active != nullptr && ld_cg(n_active) == 0;
#pragma unroll
  for (int i = 0; i < AHEAD; ++i)
    if (v0 + i * step < nvec) ahead[i].load_stream(wrow + (size_t)(v0 + i * step) * VN);
  RSD_PDL_WAIT();
  if (idle) return;
  // one thread per (column, m) finishes the sum and owns that element of y
  const int oc = threadIdx.x / MT, om = threadIdx.x % MT, on = blockIdx.x * nb + oc;
  const bool owner = threadIdx.x < nb * MT && on < N && m0 + om < M;
  float* y = Y + (size_t)(m0 + om) * N + on;
  const float old = owner && accumulate ? *y : 0.f;
  float acc[MT];
#pragma unroll
  for (int m = 0; m < MT; ++m) acc[m] = 0.f;
  auto fold = [&](const Vec16<WT>& w, int v) {
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      if (m0 + m < M) {
        Vec16<WT> xv;
        xv.load(X + (size_t)(m0 + m) * K + (size_t)v * VN);
        if (X_lo != nullptr) {
          Vec16<WT> xl;
          xl.load(X_lo + (size_t)(m0 + m) * K + (size_t)v * VN);
#pragma unroll
          for (int j = 0; j < VN; ++j) xv.v[j] += xl.v[j];
        }
#pragma unroll
        for (int j = 0; j < VN; ++j) acc[m] = fmaf(w.v[j], xv.v[j], acc[m]);
      }
    }
  };
#pragma unroll
  for (int i = 0; i < AHEAD; ++i)
    if (v0 + i * step < nvec) fold(ahead[i], v0 + i * step);
  for (int v = v0 + AHEAD * step; v < nvec; v += step) {
    Vec16<WT> w;
    w.load_stream(wrow + (size_t)v * VN);
    fold(w, v);
  }
#pragma unroll
  for (int m = 0; m < MT; ++m) acc[m] = warp_sum(acc[m]);
  if (lane == 0) {
#pragma unroll
    for (int m = 0; m < MT; ++m) part[warp][m] = acc[m];
  }
  __syncthreads();
  if (owner) {
    float sum = 0.f;
    for (int sidx = 0; sidx < ks; ++sidx) sum += part[oc * ks + sidx][om];
    *y = old + sum;
  }
}

// The decode products of fp32 models with the small steps around them: RMSNorm ahead (the gain goes into the weights as they arrive,
// the row's sum of squares is taken along with the products and its root divides the finished sum) and SwiGLU behind (GU: a warp
// streams the gate row and the up row of its column).  Geometry, reads ahead and order of the sums are those of the kernel above.
// Bound by latency like it; what this removes is a launch of 1.2-1.4 us for every norm and one for the SwiGLU.
template <int MT, int AHEAD, bool GU>
__global__ void __launch_bounds__(256)
gemv_norm_kernel(const float* W, const float* __restrict__ gain, const float* X, float* Y, int M, int N, int K, int ks, float eps,
                 const int32_t* n_active) {
  RSD_PDL_TRIGGER();
  constexpr int VN = 4, R = GU ? 2 : 1;
  __shared__ float part[8][R + 1][MT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = 8 / ks;
  const int col = warp / ks, split = warp % ks;
  const int n = blockIdx.x * nb + col;
  const int m0 = blockIdx.y * MT;
  const int nvec = n < N ? K / VN : 0, v0 = split * 32 + lane, step = ks * 32;
  const float* wrow = W + (size_t)n * K;
  Vec16<float> ahead[AHEAD][R];
  if (n_active == nullptr) RSD_PDL_WAIT();   // outside a decode pass W may be an earlier kernel's output
  const bool idle = n_active != nullptr && ld_cg(n_active) == 0;
  auto weights = [&](Vec16<float> (&w)[R], int v) {
    float g[VN];                             // (a caller's gains may start anywhere)
#pragma unroll
    for (int j = 0; j < VN; ++j) g[j] = gain[(size_t)v * VN + j];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      w[r].load_stream(wrow + (size_t)r * N * K + (size_t)v * VN);
#pragma unroll
      for (int j = 0; j < VN; ++j) w[r].v[j] *= g[j];
    }
  };
#pragma unroll
  for (int i = 0; i < AHEAD; ++i)
    if (v0 + i * step < nvec) weights(ahead[i], v0 + i * step);
  RSD_PDL_WAIT();
  if (idle) return;
  float acc[R + 1][MT];                      // the last: sums of squares
#pragma unroll
  for (int r = 0; r <= R; ++r)
#pragma unroll
    for (int m = 0; m < MT; ++m) acc[r][m] = 0.f;
  auto fold = [&](const Vec16<float> (&w)[R], int v) {
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      if (m0 + m < M) {
        Vec16<float> xv;
        xv.load(X + (size_t)(m0 + m) * K + (size_t)v * VN);
#pragma unroll
        for (int j = 0; j < VN; ++j) {
#pragma unroll
          for (int r = 0; r < R; ++r) acc[r][m] = fmaf(w[r].v[j], xv.v[j], acc[r][m]);
          acc[R][m] = fmaf(xv.v[j], xv.v[j], acc[R][m]);
        }
      }
    }
  };
#pragma unroll
  for (int i = 0; i < AHEAD; ++i)
    if (v0 + i * step < nvec) fold(ahead[i], v0 + i * step);
  for (int v = v0 + AHEAD * step; v < nvec; v += step) {
    Vec16<float> w[R];
    weights(w, v);
    fold(w, v);
  }
#pragma unroll
  for (int r = 0; r <= R; ++r)
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const float t = warp_sum(acc[r][m]);
      if (lane == 0) part[warp][r][m] = t;
    }
  __syncthreads();
  const int oc = threadIdx.x / MT, om = threadIdx.x % MT, on = blockIdx.x * nb + oc;
  if (!(threadIdx.x < nb * MT && on < N && m0 + om < M)) return;
  float sum[R + 1];
#pragma unroll
  for (int r = 0; r <= R; ++r) {
    sum[r] = 0.f;
    for (int sidx = 0; sidx < ks; ++sidx) sum[r] += part[oc * ks + sidx][r][om];
  }
  const float inv = rsqrtf(sum[R] / (float)K + eps);
  Y[(size_t)(m0 + om) * N + on] = GU ? swiglu(sum[0] * inv, sum[R - 1] * inv) : sum[0] * inv;
}

// fp32 products of more rows (prefill, scoring and catch-up of fp32 models): 32 rows of x by 32 of W a block, 32 values of K a stage, four
// stages of 16-byte cp.async copies; four groups of 64 threads take eight of a stage's 32 values of K each, 4 x 4 results a thread, and
// their sums meet at the end.  (Eight rows at a time, as above, the weights come from L2 once per eight rows and every one is used eight
// times per load.)  Bound by shared memory (two reads of 16 bytes per 16 multiply-adds, the copies, the sums kept there), with few blocks by
// the latency of a stage, 0.4 us (tiles of 64 columns with 4 x 4 or 4 x 8 results a thread took 1.5 and 1.9 times as long a stage).  Two products
// at a time: 256 x 512 x 512, 256 x 512 x 1376 and 256 x 1024 x 4096 take 15.7, 37.9 and 112 us, with scalar ones and sums of less depth
// 18.9, 47.0 and 154; with many blocks, 256 x 2752 x 512 and 1024 x 4096 x 1024, the depth of the sums costs 35.5 -> 38.9 and 354 -> 387.
constexpr int kSgM = 32, kSgN = 32, kSgK = 32, kSgLd = kSgK + 4, kSgStages = 4, kSgGroups = 4;   // rows 16 bytes apart modulo 128: no bank conflicts
constexpr int kSgStage = (kSgM + kSgN) * kSgLd, kSgThreads = 64 * kSgGroups;
static_assert((kSgGroups - 1) * kSgM * kSgN <= kSgStages * kSgStage, "the groups' sums take the place of the stages");
static_assert(kSgGroups == 4 && kSgK == 32, "the order of the sums below");

// Two fp32 products or sums at once, rounded as the scalar ones.
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float add_halves(uint64_t a) { return __uint_as_float((uint32_t)a) + __uint_as_float((uint32_t)(a >> 32)); }

__global__ void __launch_bounds__(kSgThreads, 2)
sgemm_kernel(const float* __restrict__ W, const float* __restrict__ X, float* Y, int M, int N, int K, int accumulate) {
  RSD_PDL_SYNC();
  extern __shared__ __align__(16) float sg_smem[];
  const int n0 = blockIdx.x * kSgN, m0 = blockIdx.y * kSgM, grp = threadIdx.x / 64, tid = threadIdx.x % 64;
  const int steps = (K + kSgK - 1) / kSgK;
  auto fetch = [&](int step) {
    if (step < steps) {
      float* dst = sg_smem + (step % kSgStages) * kSgStage;
      for (int idx = threadIdx.x; idx < (kSgM + kSgN) * kSgK / 4; idx += kSgThreads) {
        const int r = idx / (kSgK / 4), c = idx % (kSgK / 4) * 4, k = step * kSgK + c;
        const bool is_x = r < kSgM;
        const int row = is_x ? m0 + r : n0 + r - kSgM;
        const bool in = k < K && row < (is_x ? M : N);
        const float* src = (is_x ? X : W) + (in ? (size_t)row * K + k : 0);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + r * kSgLd + c)),
                     "l"(src), "r"(in ? 16 : 0) : "memory");          // beyond an edge: zeros
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int i = 0; i < kSgStages - 1; ++i) fetch(i);
  const int tn = tid & 7, tm = tid >> 3;         // rows tm + 8 i of x, tn + 8 j of W
  // Sums in a tree: two chains of four products a stage, pairs of stages, chains of four pairs, of four of those, and of these.  Along K it is
  // then never deeper than a lane's chain, the warp's tree and the K splits of the kernel above (relative error against fp64, that kernel / this
  // one, at K = 256, 512, 1376, 4096: 0.81 / 0.79, 0.85 / 0.83, 0.96 / 0.91, 1.10 / 0.99e-7).  The last two sums, touched every eighth and
  // thirty-second stage, lie in shared memory: two blocks an SM instead of one.
  float hold[4][4], eight[4][4];
  float *acc = sg_smem + kSgStages * kSgStage + threadIdx.x, *top = acc + 16 * kSgThreads;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[(4 * i + j) * kSgThreads] = top[(4 * i + j) * kSgThreads] = 0.f;
  for (int step = 0; step < steps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSgStages - 2) : "memory");
    __syncthreads();                             // the stage is there for all, and the one before it has been read by all
    fetch(step + kSgStages - 1);
    const float* xs = sg_smem + (step % kSgStages) * kSgStage;
    const float* ws = xs + kSgM * kSgLd;
    uint64_t part[4][4];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int kk = grp * (kSgK / kSgGroups) + 4 * k;
      ulonglong2 a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(xs + (tm + 8 * i) * kSgLd + kk);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const ulonglong2*>(ws + (tn + 8 * j) * kSgLd + kk);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          part[i][j] = k == 0 ? mul2(a[i].x, b[j].x) : fma2(a[i].x, b[j].x, part[i][j]);
          part[i][j] = fma2(a[i].y, b[j].y, part[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = add_halves(part[i][j]);
        if ((step & 1) == 0) {
          hold[i][j] = p;
        } else if ((step & 7) == 1) {
          eight[i][j] = hold[i][j] + p;
        } else {
          eight[i][j] += hold[i][j] + p;
          if ((step & 7) == 7) {
            float& u = acc[(4 * i + j) * kSgThreads];
            const float v = u + eight[i][j];
            u = (step & 31) == 31 ? 0.f : v;
            if ((step & 31) == 31) top[(4 * i + j) * kSgThreads] += v;
          }
        }
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float rest = (steps & 6 ? eight[i][j] : 0.f) + (steps & 1 ? hold[i][j] : 0.f);     // of the stages after the last eight
      eight[i][j] = top[(4 * i + j) * kSgThreads] + (acc[(4 * i + j) * kSgThreads] + rest);
    }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if (grp > 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sg_smem[((grp - 1) * kSgM + tm + 8 * i) * kSgN + tn + 8 * j] = eight[i][j];
  }
  __syncthreads();
  if (grp > 0) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + tm + 8 * i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tn + 8 * j;
      const float* other = sg_smem + (tm + 8 * i) * kSgN + tn + 8 * j;
      const float v = (eight[i][j] + other[0]) + (other[kSgM * kSgN] + other[2 * kSgM * kSgN]);
      if (m < M && n < N) {
        float* y = Y + (size_t)m * N + n;
        *y = accumulate ? *y + v : v;
      }
    }
  }
}

// Both take as long along K, so that rows times columns decide.  us, eight rows at a time / tiled: 128 x 256 x 256 5.6 / 6.3, 64 x 512 x 1376
// 24.2 / 25.6, 72 x 512 x 1376 25.2 / 25.7, 80 x 512 x 1376 29.8 / 25.7, 160 x 256 x 688 18.2 / 13.9, 17 x 2752 x 512 13.7 / 14.7, 20 x 2752 x 512
// 15.5 / 14.7, 48 x 1024 x 1024 24.1 / 24.8, 96 x 512 x 256 9.2 / 6.3, 256 x 2752 x 512 154 / 39.
static bool sgemm_pays(int M, int N) { return M > 16 && (long)M * N >= 40000; }

// K splits over the warps of a block.
static int simt_splits(int dtype, int M, int N, int K) {
  // Pick the split so that the grid covers the 148 SMs a few times over, as long as every lane has two vectors, or one (fp32) where
  // there are up to four rows or few blocks.  More rows are more blocks, each with its reductions: splitting them as finely, and
  // holding weights ahead in registers where no wait is to be bridged, cost 256 x 512 x 1376 146 us instead of 84 and 60 x 512 x
  // 256 12 instead of 5.6; few blocks left whole, 8 x 512 x 256 4.6 us, halved 3.4.
  int ks = 1;
  const int mt = M <= 4 ? 4 : 8;
  const long m_blocks = (M + mt - 1) / mt;
  auto lanes_full = [&](int k) {
    const long blocks = N * m_blocks * (k / 2) / 8;       // before the step to k
    return K / k >= (dtype != 1 && (M <= 4 || blocks < 148 || (k == 2 && blocks < 296)) ? 128 : 256);
  };
  while (ks < 8 && (long)N * ks / 8 < 148L * 4 && lanes_full(2 * ks)) ks *= 2;
  return ks;
}

// y = rmsnorm(x) W^T, or silu(g) * u with [g | u] = rmsnorm(x) W^T and W of 2 N rows.
cudaError_t launch_gemv_norm(const float* W, const float* gain, const float* x, float* y, int M, int N, int K, float eps, bool gate_up,
                             const int32_t* n_active, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const int ks = simt_splits(0, M, N, K), mt = M <= 4 ? 4 : 8;
  const dim3 grid((N + (8 / ks) - 1) / (8 / ks), (unsigned)((M + mt - 1) / mt));
#define RSD_GN(MT, GU) RSD_LAUNCH((gemv_norm_kernel<MT, GU ? 2 : kGemvAhead, GU>), grid, 256, 0, s, W, gain, x, y, M, N, K, ks, eps, n_active)
  if (mt == 4) { if (gate_up) RSD_GN(4, true); else RSD_GN(4, false); }
  else { if (gate_up) RSD_GN(8, true); else RSD_GN(8, false); }
#undef RSD_GN
  return launched(1);
}

cudaError_t launch_gemm_simt(int dtype, const void* W, const void* x, const void* x_lo, float* y, int M, int N, int K,
                             int accumulate, const int32_t* n_active, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (dtype != 1 && n_active == nullptr && sgemm_pays(M, N)) {
    static OncePerDevice configured;
    constexpr size_t smem = (kSgStages * kSgStage + 2 * 16 * kSgThreads) * sizeof(float);
    const cudaError_t set = allow_smem(configured, sgemm_kernel, smem);
    if (set != cudaSuccess) return set;
    RSD_LAUNCH((sgemm_kernel), dim3((N + kSgN - 1) / kSgN, (M + kSgM - 1) / kSgM), kSgThreads, smem, s, (const float*)W, (const float*)x, y, M, N, K, accumulate);
    return launched(1);
  }
  const int ks = simt_splits(dtype, M, N, K), mt = M <= 4 ? 4 : 8;
  const long m_blocks = (M + mt - 1) / mt;
  const bool ahead = M <= 4 || n_active != nullptr;
  dim3 grid((N + (8 / ks) - 1) / (8 / ks), (unsigned)m_blocks);
#define RSD_GEMV(WT, MT, AHEAD) RSD_LAUNCH((gemv_splitk_kernel<WT, MT, AHEAD>), grid, 256, 0, s, (const WT*)W, (const WT*)x, (const WT*)x_lo, y, M, N, K, ks, accumulate, n_active)
#define RSD_GEMV_M(WT) do { if (mt == 4) RSD_GEMV(WT, 4, kGemvAhead); else if (ahead) RSD_GEMV(WT, 8, kGemvAhead); else RSD_GEMV(WT, 8, 0); } while (0)
  if (dtype == 1) RSD_GEMV_M(__nv_bfloat16);
  else { x_lo = nullptr; RSD_GEMV_M(float); }
#undef RSD_GEMV_M
#undef RSD_GEMV
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// Rotary table: table[pos, i] = (cos, sin)(pos * theta^(-2i/hd)), evaluated in fp64
// ---------------------------------------------------------------------------------------------
__global__ void rope_table_kernel(float2* table, int n_pos, int half, double theta, double hd) {
  RSD_PDL_SYNC();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_pos * half) return;
  const int pos = idx / half, i = idx % half;
  const double ang = (double)pos * pow(theta, -2.0 * (double)i / hd);
  double sn, cs;
  sincos(ang, &sn, &cs);
  table[idx] = make_float2((float)cs, (float)sn);
}

cudaError_t launch_rope_table(float2* table, int n_pos, int hd, float theta, cudaStream_t s) {
  const int n = n_pos * (hd / 2);
  if (n <= 0) return cudaSuccess;
  RSD_LAUNCH((rope_table_kernel), (n + 255) / 256, 256, 0, s, table, n_pos, hd / 2, (double)theta, (double)hd);
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// RoPE on q and k, KV page write.  One block per token slot; threads walk the (head, pair) grid.
// Pair (i, i + hd/2) of a head turns by the angle of (position, i).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float split_sum(const float* direct, const float* partials, int splits,
                                           size_t idx, size_t stride) {
  if (splits <= 1) return direct[idx];
  // loads go out twelve at a time (tail predicated) so their latencies overlap; the sums stay in split order
  float v = 0.f;
  for (int s0 = 0; s0 < splits; s0 += 12) {
    float t[12];
#pragma unroll
    for (int u = 0; u < 12; ++u) t[u] = s0 + u < splits ? ld_cg(partials + (size_t)(s0 + u) * stride + idx) : 0.f;
#pragma unroll
    for (int u = 0; u < 12; ++u) v += t[u];
  }
  return v;
}

// Bound by latency like reduce_norm: lists, page and angle are fetched under the wait, and with K-split partial sums
// kSumGroups groups of 64 threads share them out.
template <typename KT>
__global__ void __launch_bounds__(64 * kSumGroups)
rope_kv_kernel(const float* qkv, const float* partials, int splits, PassView p, float* q_out, KT* pool, const int32_t* page_table,
               int max_pages, const float2* __restrict__ rope, int H, int KV, int hd, int pf) {
  RSD_PDL_TRIGGER();
  __shared__ float s_part[kSumGroups - 1][128];
  if (p.n_active == nullptr) RSD_PDL_WAIT();   // a decode pass's lists may be read ahead of the wait, others not
  const int t = blockIdx.x;
  const bool idle = p.n_active != nullptr && ld_cg(p.n_active) == 0;
  const int row = ld_cg(p.tok_row + t), pos = ld_cg(p.tok_pos + t);
  if (idle || row < 0) { RSD_PDL_WAIT(); return; }
  // one block per (token, head): query and key heads are rotated, value heads copied; a pair (i, i + hd/2) per thread
  const int head = blockIdx.y, half = hd / 2, i = threadIdx.x, grp = threadIdx.y;
  const int width = (H + 2 * KV) * hd;
  const size_t src = (size_t)t * width + (size_t)head * hd + i;   // of this thread's pair in qkv / a partial
  const size_t sstride = (size_t)gridDim.x * width;               // one partial array = [T][width]
  const int page = ld_cg(page_table + (size_t)row * max_pages + pos / kPageTokens);
  const int slot = pos % kPageTokens;
  float2 cs = make_float2(1.f, 0.f);
  if (i < half && head < H + KV && grp == 0) cs = rope[(size_t)pos * half + i];
  RSD_PDL_WAIT();
  float a = 0.f, b = 0.f;
  if (i < half) {
    if (splits <= 1) {
      a = qkv[src]; b = qkv[src + half];
    } else {
      const int per = (splits + kSumGroups - 1) / kSumGroups, s_end = min(splits, (grp + 1) * per);
      for (int s0 = grp * per; s0 < s_end; s0 += kSumAhead) {
        float ta[kSumAhead], tb[kSumAhead];
#pragma unroll
        for (int u = 0; u < kSumAhead; ++u)
          if (s0 + u < s_end) {
            ta[u] = ld_cg(partials + (size_t)(s0 + u) * sstride + src);
            tb[u] = ld_cg(partials + (size_t)(s0 + u) * sstride + src + half);
          }
#pragma unroll
        for (int u = 0; u < kSumAhead; ++u)
          if (s0 + u < s_end) { a += ta[u]; b += tb[u]; }
      }
      if (grp > 0) { s_part[grp - 1][i] = a; s_part[grp - 1][i + 64] = b; }
    }
  }
  if (splits > 1) __syncthreads();
  if (grp > 0 || i >= half) return;
  if (splits > 1) {
#pragma unroll
    for (int u = 0; u < kSumGroups - 1; ++u) { a += s_part[u][i]; b += s_part[u][i + 64]; }
  }
  // page = K block [KV][16][hd] followed by V block [KV][hd][16] (V transposed within the page)
  // (pf = 4: two more blocks hold the low halves of the keys and of the values)
  const size_t block = (size_t)KV * kPageTokens * hd;
  KT* kbase = pool + (size_t)page * pf * block;
  KT* dst;                                     // where the pair's two elements go, `gap` elements apart
  size_t gap;
  if (head < H + KV) {
    const float ra = rotate_lo(a, b, cs), rb = rotate_hi(a, b, cs);
    a = ra; b = rb;
    if (head < H) {
      float* q = q_out + ((size_t)t * H + head) * hd + i;
      q[0] = a;
      q[half] = b;
      return;
    }
    dst = kbase + ((size_t)(head - H) * kPageTokens + slot) * hd + i;
    gap = half;
  } else {
    dst = kbase + block + ((size_t)(head - H - KV) * hd + i) * kPageTokens + slot;
    gap = (size_t)half * kPageTokens;
  }
  const KT ka = from_f32<KT>(a), kb = from_f32<KT>(b);
  dst[0] = ka;
  dst[gap] = kb;
  if (pf == 4) {
    dst[2 * block] = from_f32<KT>(a - to_f32(ka));
    dst[2 * block + gap] = from_f32<KT>(b - to_f32(kb));
  }
}

// The same for the long passes (prefill, scoring, sync, catch-up: thousands of tokens, no K-split sums): a block takes
// kRopeTokens consecutive list entries.  Their rows, positions and pages are looked up once into shared memory, so the
// data loads of all entries go out together instead of after a chain of three dependent loads per (token, head)
// block; and when the entries are consecutive positions of one row inside one page (the rule in a long pass), a thread
// writes the eight transposed value elements of a (head, dim) as ONE 16-byte store instead of eight 2-byte ones.
// Bound by DRAM: a token's fp32 qkv row in, its fp32 queries and 16-bit keys and values out.
constexpr int kRopeTokens = 8;

// Four neighbouring cache elements (and their low halves) as one store.
template <typename KT> __device__ __forceinline__ void store_cache4(KT* hi, KT* lo, const float* v) {
  __align__(16) KT h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { h[i] = from_f32<KT>(v[i]); l[i] = from_f32<KT>(v[i] - to_f32(h[i])); }
  if (sizeof(KT) == 2) {
    *reinterpret_cast<uint2*>(hi) = *reinterpret_cast<const uint2*>(h);
    if (lo != nullptr) *reinterpret_cast<uint2*>(lo) = *reinterpret_cast<const uint2*>(l);
  } else {
    *reinterpret_cast<uint4*>(hi) = *reinterpret_cast<const uint4*>(h);
  }
}

template <typename KT>
__global__ void __launch_bounds__(256)
rope_kv_long_kernel(const float* __restrict__ qkv, PassView p, float* __restrict__ q_out, KT* pool,
                    const int32_t* __restrict__ page_table, int max_pages, const float2* __restrict__ rope, int H, int KV,
                    int hd, int pf) {
  RSD_PDL_SYNC();
  __shared__ int s_row[kRopeTokens], s_pos[kRopeTokens], s_page[kRopeTokens];
  __shared__ int s_run;            // 1: the entries are eight consecutive positions of one row within one page
  const int t0 = blockIdx.x * kRopeTokens;
  const int n_tok = min(kRopeTokens, p.T - t0);
  if (threadIdx.x < kRopeTokens) {
    const int i = threadIdx.x;
    int row = -1, pos = 0, page = 0;
    if (i < n_tok) {
      row = p.tok_row[t0 + i];
      pos = p.tok_pos[t0 + i];
      if (row >= 0) page = page_table[(size_t)row * max_pages + pos / kPageTokens];
    }
    s_row[i] = row; s_pos[i] = pos; s_page[i] = page;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = n_tok == kRopeTokens && s_row[0] >= 0 && (s_pos[0] % kRopeTokens) == 0;
    for (int i = 1; i < kRopeTokens && run; ++i) run = s_row[i] == s_row[0] && s_pos[i] == s_pos[0] + i;
    s_run = run;
  }
  __syncthreads();
  const int half = hd / 2;
  const int width = (H + 2 * KV) * hd;
  const size_t block = (size_t)KV * kPageTokens * hd;
  // queries and keys: a thread takes four neighbouring pairs of a head for all tokens of the block, all their loads in
  // flight together
  const int per_head = half / 4;                // 8 or 16
  for (int e = threadIdx.x; e < (H + KV) * per_head; e += blockDim.x) {
    const int head = e / per_head, i = (e % per_head) * 4;
    const float* src = qkv + (size_t)t0 * width + head * hd + i;
#pragma unroll 4
    for (int tk = 0; tk < n_tok; ++tk) {
      if (s_row[tk] < 0) continue;
      const float4 a = *reinterpret_cast<const float4*>(src + (size_t)tk * width);
      const float4 b = *reinterpret_cast<const float4*>(src + (size_t)tk * width + half);
      const float4 c01 = *reinterpret_cast<const float4*>(rope + (size_t)s_pos[tk] * half + i);
      const float4 c23 = *reinterpret_cast<const float4*>(rope + (size_t)s_pos[tk] * half + i + 2);
      const float2 c[4] = {make_float2(c01.x, c01.y), make_float2(c01.z, c01.w), make_float2(c23.x, c23.y), make_float2(c23.z, c23.w)};
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
      float ra[4], rb[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) { ra[k] = rotate_lo(av[k], bv[k], c[k]); rb[k] = rotate_hi(av[k], bv[k], c[k]); }
      if (head < H) {
        float* q = q_out + ((size_t)(t0 + tk) * H + head) * hd + i;
        *reinterpret_cast<float4*>(q) = make_float4(ra[0], ra[1], ra[2], ra[3]);
        *reinterpret_cast<float4*>(q + half) = make_float4(rb[0], rb[1], rb[2], rb[3]);
      } else {
        KT* k = pool + (size_t)s_page[tk] * pf * block + ((size_t)(head - H) * kPageTokens + s_pos[tk] % kPageTokens) * hd + i;
        store_cache4<KT>(k, pf == 4 ? k + 2 * block : nullptr, ra);
        store_cache4<KT>(k + half, pf == 4 ? k + 2 * block + half : nullptr, rb);
      }
    }
  }
  // values, transposed inside the page: [KV][hd][16 tokens]
  if (s_run && sizeof(KT) == 2) {
    const int slot0 = s_pos[0] % kPageTokens;                     // 0 or 8: the 16-byte store is aligned
    KT* vbase = pool + (size_t)s_page[0] * pf * block + block;
    for (int e = threadIdx.x; e < KV * hd; e += blockDim.x) {
      __align__(16) KT hi8[kRopeTokens];
      __align__(16) KT lo8[kRopeTokens];
#pragma unroll
      for (int tk = 0; tk < kRopeTokens; ++tk) {
        const float v = qkv[(size_t)(t0 + tk) * width + (size_t)(H + KV) * hd + e];
        hi8[tk] = from_f32<KT>(v);
        lo8[tk] = from_f32<KT>(v - to_f32(hi8[tk]));
      }
      *reinterpret_cast<uint4*>(vbase + (size_t)e * kPageTokens + slot0) = *reinterpret_cast<const uint4*>(hi8);
      if (pf == 4) *reinterpret_cast<uint4*>(vbase + 2 * block + (size_t)e * kPageTokens + slot0) = *reinterpret_cast<const uint4*>(lo8);
    }
  } else {
    for (int idx = threadIdx.x; idx < n_tok * KV * hd; idx += blockDim.x) {
      const int tk = idx / (KV * hd), e = idx % (KV * hd);
      if (s_row[tk] < 0) continue;
      const float v = qkv[(size_t)(t0 + tk) * width + (size_t)(H + KV) * hd + e];
      KT* vbase = pool + (size_t)s_page[tk] * pf * block + block;
      const int slot = s_pos[tk] % kPageTokens;
      const KT vh = from_f32<KT>(v);
      vbase[(size_t)e * kPageTokens + slot] = vh;
      if (pf == 4) vbase[2 * block + (size_t)e * kPageTokens + slot] = from_f32<KT>(v - to_f32(vh));
    }
  }
}

cudaError_t launch_rope_kv(int kv_dtype, const float* qkv, SplitSum pending, PassView p, float* q_out, KvView kv,
                           const float2* rope, int H, int KV, int hd, cudaStream_t s) {
  if (p.T <= 0) return cudaSuccess;
  const int pf = 2 + 2 * kv.v_extra;
  if (pending.splits <= 1 && p.n_active == nullptr && p.T >= 64 && ((uintptr_t)kv.pool_layer & 15) == 0) {
    // long pass: eight list entries per block, keys and values in vectors (a caller's pool that starts off a 16-byte boundary: element by element below)
    const int blocks = (p.T + kRopeTokens - 1) / kRopeTokens;
    if (kv_dtype == 2 || kv_dtype == 3)
      RSD_LAUNCH((rope_kv_long_kernel<__half>), blocks, 256, 0, s, qkv, p, q_out, (__half*)kv.pool_layer, kv.page_table, kv.max_pages, rope, H, KV, hd, pf);
    else if (kv_dtype == 1)
      RSD_LAUNCH((rope_kv_long_kernel<__nv_bfloat16>), blocks, 256, 0, s, qkv, p, q_out, (__nv_bfloat16*)kv.pool_layer, kv.page_table, kv.max_pages, rope, H, KV, hd, pf);
    else
      RSD_LAUNCH((rope_kv_long_kernel<float>), blocks, 256, 0, s, qkv, p, q_out, (float*)kv.pool_layer, kv.page_table, kv.max_pages, rope, H, KV, hd, pf);
    return launched(1);
  }
  if (kv_dtype == 2 || kv_dtype == 3)
    RSD_LAUNCH((rope_kv_kernel<__half>), dim3(p.T, H + 2 * KV), dim3(64, pending.splits > 1 ? kSumGroups : 1), 0, s, qkv, pending.partials, pending.splits, p, q_out, (__half*)kv.pool_layer, kv.page_table, kv.max_pages, rope, H, KV, hd, pf);
  else if (kv_dtype == 1)
    RSD_LAUNCH((rope_kv_kernel<__nv_bfloat16>), dim3(p.T, H + 2 * KV), dim3(64, pending.splits > 1 ? kSumGroups : 1), 0, s, qkv, pending.partials, pending.splits, p, q_out, (__nv_bfloat16*)kv.pool_layer, kv.page_table, kv.max_pages, rope, H, KV, hd, pf);
  else
    RSD_LAUNCH((rope_kv_kernel<float>), dim3(p.T, H + 2 * KV), dim3(64, pending.splits > 1 ? kSumGroups : 1), 0, s, qkv, pending.partials, pending.splits, p, q_out, (float*)kv.pool_layer, kv.page_table, kv.max_pages, rope, H, KV, hd, pf);
  return launched(1);
}

// Stand-alone rotary kernel on [T, n_heads, hd] fp32 (angles in fp64).
__global__ void rope_only_kernel(float* v, const int32_t* pos, int n_heads, int hd, double theta) {
  RSD_PDL_SYNC();
  const int t = blockIdx.x, half = hd / 2;
  const int p = pos[t];
  for (int idx = threadIdx.x; idx < n_heads * half; idx += blockDim.x) {
    const int head = idx / half, i = idx % half;
    double sn, cs;
    sincos((double)p * pow(theta, -2.0 * (double)i / (double)hd), &sn, &cs);
    float* h = v + ((size_t)t * n_heads + head) * hd;
    const float a = h[i], b = h[i + half];
    h[i] = a * (float)cs - b * (float)sn;
    h[i + half] = b * (float)cs + a * (float)sn;
  }
}

cudaError_t launch_rope_only(float* v, const int32_t* pos, int T, int n_heads, int hd, float theta, cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  RSD_LAUNCH((rope_only_kernel), T, 128, 0, s, v, pos, n_heads, hd, (double)theta);
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// Generic causal attention over paged KV (fp32 caches, groups wider than eight heads): one block of four to sixteen
// warps per (slot, query head), the row's pages dealt round the warps; query head j reads KV head j / (H / KV).
// Bound by latency: the caches it serves are small, the chain of dependent steps is not.  A page is therefore one
// flat piece of work for a warp: lane = (token, half of the head dim), so that all 16 scores come out of ONE shuffle
// instead of sixteen warp sums, every load of the page's keys and values goes out before the first use, and the next
// page's id is fetched a page ahead.  The warps' partial (max, sum, O) meet in shared memory in warp order.
// (One warp walking all pages of a head with a warp sum per token: 50 us a launch at 4 rows x 64..190 cached tokens,
// growing with the context; this form: 4.5 us.)
// ---------------------------------------------------------------------------------------------
constexpr int kGenericWarps = 16;

// VEC: 16-byte loads; a caller's pool may start anywhere, and one off a 16-byte boundary is read element by element.
// FUSE (a decode pass of an fp32 model; every row's only new position is its last): q is the qkv product [T][(H + 2 KV) HD]; the kernel
// rotates by the table, keeps the new key and value in shared memory, and the first block of a group writes them to the cache.  Every page
// is then older than the pass but for that one slot, so a warp's first page is on its way before the wait.
template <typename KT, typename OT, int HD, bool VEC, bool FUSE>
__global__ void __launch_bounds__(32 * kGenericWarps)
attn_generic_kernel(const float* q, PassView p, KT* pool, const int32_t* page_table, int max_pages, OT* out, OT* out_lo,
                    int H, int KV, int pf, const float2* __restrict__ rope) {
  RSD_PDL_TRIGGER();
  constexpr int DPL = HD / 32;            // output dims of a lane
  constexpr int VN = 16 / sizeof(KT);     // elements of a 16-byte load
  constexpr int NK = HD / 2 / VN;         // key loads of a lane
  constexpr int NV = kPageTokens / VN;    // value loads of a dim
  __shared__ __align__(16) float s_q[HD];
  __shared__ float s_m[kGenericWarps], s_l[kGenericWarps], s_o[kGenericWarps][HD];
  __shared__ __align__(16) float s_kv[FUSE ? 2 : 1][HD];    // the new token's key and value
  const int t = blockIdx.x / H, h = blockIdx.x % H;
  if (p.n_active == nullptr) RSD_PDL_WAIT();   // a decode pass's lists may be read ahead of the wait, others not
  const bool idle = p.n_active != nullptr && ld_cg(p.n_active) == 0;
  const int row = ld_cg(p.tok_row + t), pos = ld_cg(p.tok_pos + t);
  if (idle || row < 0) { RSD_PDL_WAIT(); return; }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  const int tok = lane & 15, hf = lane >> 4;
  const int g = h / (H / KV);
  const float scale = rsqrtf((float)HD);
  const int32_t* pt = page_table + (size_t)row * max_pages;
  const int n_pages = pos / kPageTokens + 1;
  const size_t block = (size_t)KV * kPageTokens * HD;
  int page = warp < n_pages ? ld_cg(pt + warp) : 0;
  uint4 kr[NK], vr[DPL * NV];
  auto keys = [&](int id) { return pool + (size_t)id * pf * block + (size_t)g * kPageTokens * HD + tok * HD + hf * (HD / 2); };
  auto values = [&](int id) { return pool + (size_t)id * pf * block + block + (size_t)g * kPageTokens * HD + lane * DPL * kPageTokens; };
  float2 cs = make_float2(1.f, 0.f);
  int new_page = 0;
  if (FUSE) {
    if (VEC && warp < n_pages) {
#pragma unroll
      for (int i = 0; i < NK; ++i) kr[i] = __ldcg(reinterpret_cast<const uint4*>(keys(page) + i * VN));
#pragma unroll
      for (int i = 0; i < DPL * NV; ++i) vr[i] = __ldcg(reinterpret_cast<const uint4*>(values(page) + i * VN));
    }
    cs = rope[(size_t)pos * (HD / 2) + threadIdx.x % (HD / 2)];        // HD divides the block
    new_page = ld_cg(pt + n_pages - 1);
  }
  RSD_PDL_WAIT();
  if (FUSE) {
    // HD threads each for the query, the key and the value; dim i < HD / 2 turns with i + HD / 2
    const int dim = threadIdx.x % HD, pair = dim < HD / 2 ? dim + HD / 2 : dim - HD / 2;
    for (int w = threadIdx.x / HD; w < 3; w += blockDim.x / HD) {
      const float* src = q + (size_t)t * (H + 2 * KV) * HD + (size_t)(w == 0 ? h : H + (w - 1) * KV + g) * HD;
      float a = src[dim];
      if (w < 2) {
        const float b = src[pair];
        a = dim < HD / 2 ? rotate_lo(a, b, cs) : rotate_hi(b, a, cs);
      }
      if (w == 0) s_q[dim] = a * scale;
      else s_kv[FUSE ? w - 1 : 0][dim] = a;
      if (w > 0 && h % (H / KV) == 0) {
        const int slot = pos % kPageTokens;
        KT* at = pool + (size_t)new_page * pf * block + (w == 1 ? ((size_t)g * kPageTokens + slot) * HD + dim : block + ((size_t)g * HD + dim) * kPageTokens + slot);
        *at = from_f32<KT>(a);
      }
    }
  } else if (threadIdx.x < HD) {
    s_q[threadIdx.x] = q[((size_t)t * H + h) * HD + threadIdx.x] * scale;
  }
  __syncthreads();
  float m = -INFINITY, l = 0.f, acc[DPL];
#pragma unroll
  for (int i = 0; i < DPL; ++i) acc[i] = 0.f;
  for (int pg = warp; pg < n_pages; pg += n_warps) {
    const KT *kb = keys(page), *vb = values(page);
    if (pg + n_warps < n_pages) page = ld_cg(pt + pg + n_warps);
    const int n = min(kPageTokens, pos + 1 - pg * kPageTokens);
    const bool has_new = FUSE && pg == n_pages - 1;
    if (FUSE && VEC && pg == warp) {                       // on its way since before the wait
    } else if (VEC) {
#pragma unroll
      for (int i = 0; i < NK; ++i) kr[i] = *reinterpret_cast<const uint4*>(kb + i * VN);
#pragma unroll
      for (int i = 0; i < DPL * NV; ++i) vr[i] = *reinterpret_cast<const uint4*>(vb + i * VN);
    } else {
#pragma unroll
      for (int i = 0; i < NK * VN; ++i) reinterpret_cast<KT*>(kr)[i] = kb[i];
#pragma unroll
      for (int i = 0; i < DPL * NV * VN; ++i) reinterpret_cast<KT*>(vr)[i] = vb[i];
    }
    if (has_new && tok == n - 1) {
#pragma unroll
      for (int i = 0; i < NK; ++i) kr[i] = *reinterpret_cast<const uint4*>(&s_kv[0][hf * (HD / 2) + i * VN]);
    }
    float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < NK; ++i) {
      const KT* e = reinterpret_cast<const KT*>(&kr[i]);
#pragma unroll
      for (int j = 0; j < VN; ++j) {
        float kk = to_f32(e[j]);
        if (pf == 4) kk += to_f32(kb[2 * block + i * VN + j]);
        part[j & 3] = fmaf(s_q[hf * (HD / 2) + i * VN + j], kk, part[j & 3]);
      }
    }
    float sc = (part[0] + part[1]) + (part[2] + part[3]);
    sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 16);
    if (tok >= n) sc = -INFINITY;
    float mx = sc;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    mx = fmaxf(m, mx);                                     // finite: token 0 of a walked page is always valid
    const float corr = __expf(m - mx), pr = __expf(sc - mx);
    l = l * corr + (hf == 0 ? pr : 0.f);                   // this lane's token only; the lanes meet after the loop
#pragma unroll
    for (int i = 0; i < DPL; ++i) acc[i] *= corr;
#pragma unroll
    for (int j = 0; j < kPageTokens; ++j) {
      const float pj = __shfl_sync(0xFFFFFFFFu, pr, j);
      if (j < n) {                                         // slots beyond the context hold anything, NaN included
#pragma unroll
        for (int i = 0; i < DPL; ++i) {
          float vv = to_f32(reinterpret_cast<const KT*>(&vr[i * NV + j / VN])[j % VN]);
          if (FUSE && has_new && j == n - 1) vv = s_kv[FUSE ? 1 : 0][lane * DPL + i];
          if (pf == 4) vv += to_f32(vb[2 * block + i * kPageTokens + j]);
          acc[i] = fmaf(pj, vv, acc[i]);
        }
      }
    }
    m = mx;
  }
  l = warp_sum(l);
  if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
#pragma unroll
  for (int i = 0; i < DPL; ++i) s_o[warp][lane * DPL + i] = acc[i];
  __syncthreads();
  if (threadIdx.x < HD) {
    float M = s_m[0], L = 0.f, O = 0.f;
    for (int w = 1; w < n_warps; ++w) M = fmaxf(M, s_m[w]);
    for (int w = 0; w < n_warps; ++w) {
      const float e = __expf(s_m[w] - M);                  // 0 for a warp without pages
      L += s_l[w] * e;
      O += s_o[w][threadIdx.x] * e;
    }
    store_operand<OT>(out, out_lo, ((size_t)t * H + h) * HD + threadIdx.x, O / L);
  }
}

cudaError_t launch_attn_generic(int kv_dtype, const float* q, PassView p, KvView kv, void* out, void* out_lo,
                                int out_dtype, int H, int KV, int hd, cudaStream_t s, const float2* rope) {
  if (p.T <= 0) return cudaSuccess;
  if (rope != nullptr && (kv_dtype != 0 || out_dtype != 0 || p.n_active == nullptr)) return cudaErrorInvalidValue;
  const int blocks = p.T * H;
  // few (slot, head) pairs: sixteen warps, so that 256 cached tokens are one round; once the pairs alone fill the SMs,
  // four warps a block waste fewer on short contexts
  const int threads = 32 * (blocks <= 148 ? kGenericWarps : (blocks <= 148 * 4 ? 8 : 4));
#define RSD_ATTN_K(KT, OT, HD, VEC, FUSE)                                                                               \
  RSD_LAUNCH((attn_generic_kernel<KT, OT, HD, VEC, FUSE>), blocks, threads, 0, s, q, p, (KT*)kv.pool_layer, kv.page_table, kv.max_pages, (OT*)out, (OT*)out_lo, H, KV, 2 + 2 * kv.v_extra, rope)
#define RSD_ATTN_F(KT, OT, HD, FUSE) do { if (((uintptr_t)kv.pool_layer & 15) == 0) RSD_ATTN_K(KT, OT, HD, true, FUSE); else RSD_ATTN_K(KT, OT, HD, false, FUSE); } while (0)
#define RSD_ATTN(KT, OT, HD) RSD_ATTN_F(KT, OT, HD, false)
#define RSD_ATTN_HD(KT, OT) do { if (hd == 128) RSD_ATTN(KT, OT, 128); else RSD_ATTN(KT, OT, 64); } while (0)
  using bf = __nv_bfloat16;
  if (kv_dtype == 2) { if (out_dtype == 1) RSD_ATTN_HD(__half, bf); else RSD_ATTN_HD(__half, float); }
  else if (kv_dtype == 1) { if (out_dtype == 1) RSD_ATTN_HD(bf, bf); else RSD_ATTN_HD(bf, float); }
  else if (rope != nullptr) { if (hd == 128) RSD_ATTN_F(float, float, 128, true); else RSD_ATTN_F(float, float, 64, true); }
  else RSD_ATTN_HD(float, float);
#undef RSD_ATTN_HD
#undef RSD_ATTN
#undef RSD_ATTN_F
#undef RSD_ATTN_K
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// SwiGLU: out[t, f] = silu(gu[t, f]) * gu[t, F + f]
// ---------------------------------------------------------------------------------------------
template <typename OT>
__global__ void swiglu_kernel(const float* gu, const float* partials, int splits, OT* out, OT* out_lo, int T, int F, const int32_t* n_active) {
  RSD_PDL_SYNC_UNLESS_IDLE(n_active);
  const size_t n = (size_t)T * F;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t t = i / F, f = i % F;
    const size_t sstride = (size_t)T * 2 * F;
    const float a = split_sum(gu, partials, splits, t * 2 * F + f, sstride);
    const float b = split_sum(gu, partials, splits, t * 2 * F + F + f, sstride);
    store_operand<OT>(out, out_lo, i, swiglu(a, b));
  }
}

cudaError_t launch_swiglu(int dtype, const float* gu, SplitSum pending, void* out, void* out_lo, int T, int F,
                          const int32_t* n_active, cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  const size_t n = (size_t)T * F;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 148 * 8) blocks = 148 * 8;
  if (dtype == 1) RSD_LAUNCH((swiglu_kernel<__nv_bfloat16>), blocks, 256, 0, s, gu, pending.partials, pending.splits, (__nv_bfloat16*)out, (__nv_bfloat16*)out_lo, T, F, n_active);
  else RSD_LAUNCH((swiglu_kernel<float>), blocks, 256, 0, s, gu, pending.partials, pending.splits, (float*)out, nullptr, T, F, n_active);
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// Sampling: greedy argmax, or Gumbel-max with Philox noise keyed by (seed; vocab id / 4, position
// of the generated token, row, model id).  One block per slot; ties go to the lowest id.
// ---------------------------------------------------------------------------------------------
// Grid (slots, chunks): every warp takes `steps` runs of 128 ids of a slot and folds its best candidate into best[slot] with
// an atomic maximum (order-independent, hence deterministic).
// Exact noise for every id -- ten Philox rounds per four ids and two logarithms per id -- kept the ALUs busy for 66 us at
// 151936 ids x 128 rows, four times what the logits' 78 MB take.  So with many ids in all (launch_sample draws the line) a warp
// first publishes the exact score of its largest logit; then a score is first taken with fast logarithms, and only ids within
// kScoreMargin of the best so far (this warp's, or what others have published) get exact ones; and as the noise lies below
// 16.64, ids whose logits stay kNoiseMax below that best draw none at all.  The winner is the same.
// DIRECT: few ids in all, exact noise for each of them.
constexpr int kSampleThreads = 256, kSampleBlocks = 4;   // ... and blocks per SM
constexpr int kSampleSteps = 8;             // runs of 128 ids that a warp holds in registers at most
template <bool DIRECT>
__global__ void __launch_bounds__(kSampleThreads, kSampleBlocks) sample_kernel(SampleArgs a, int steps) {
  RSD_PDL_TRIGGER();
  if (a.n_active == nullptr) RSD_PDL_WAIT();   // a decode pass's lists may be read ahead of the wait, others not
  const bool idle = a.n_active != nullptr && ld_cg(a.n_active) == 0;
  const int slot = blockIdx.x;
  const int row = ld_cg(a.slot_row + slot);
  const uint32_t position = (uint32_t)(ld_cg(a.slot_pos + slot) + 1);
  RSD_PDL_WAIT();
  if (idle || row < 0) return;
  const float* lg = a.logits + (size_t)slot * a.V;
  const uint2 key = make_uint2((uint32_t)(a.seed & 0xFFFFFFFFull), (uint32_t)(a.seed >> 32));
  const bool noisy = a.temperature > 0.f;
  const float inv_t = noisy ? 1.f / a.temperature : 1.f;
  const int lane = threadIdx.x & 31, n_v4 = (a.v_limit + 3) / 4;
  const int v4_0 = ((blockIdx.y * (kSampleThreads / 32) + (threadIdx.x >> 5)) * steps) * 32 + lane;
  const bool vec = (a.V & 3) == 0 && ((uintptr_t)a.logits & 15) == 0;
  const float out = __int_as_float(0x7FC00000);        // NaN: an id out of the race never wins a comparison
  float x[kSampleSteps][4];
#pragma unroll
  for (int k = 0; k < kSampleSteps; ++k) {
    const int v4 = v4_0 + k * 32;
#pragma unroll
    for (int j = 0; j < 4; ++j) x[k][j] = out;
    if (k < steps && vec && v4 * 4 + 3 < a.v_limit) {
      const float4 t = *reinterpret_cast<const float4*>(lg + v4 * 4);
      x[k][0] = t.x; x[k][1] = t.y; x[k][2] = t.z; x[k][3] = t.w;
    } else if (k < steps && v4 < n_v4) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (v4 * 4 + j < a.v_limit) x[k][j] = lg[v4 * 4 + j];
    }
  }
  auto noise_bits = [&](int v4, uint32_t (&w)[4]) {
    const uint4 r = philox4x32_10(make_uint4((uint32_t)v4, position, (uint32_t)row, (uint32_t)a.model_id), key);
    w[0] = r.x; w[1] = r.y; w[2] = r.z; w[3] = r.w;
  };
  auto exact = [&](float logit, uint32_t bits) { return fmaf(logit, inv_t, -logf(-logf(uniform_from_bits(bits)))); };
  float bs = -INFINITY;
  int bi = 0x7FFFFFFF;
  if (DIRECT && noisy) {
#pragma unroll
    for (int k = 0; k < kSampleSteps; ++k) {
      if (k >= steps) break;
      uint32_t w[4];
      noise_bits(v4_0 + k * 32, w);
#pragma unroll
      for (int j = 0; j < 4; ++j) better(bs, bi, exact(x[k][j], w[j]), (v4_0 + k * 32) * 4 + j);
    }
  } else {
    // this lane's largest logit, then the warp's
    float tx = -INFINITY;
    int ti = 0x7FFFFFFF;
#pragma unroll
    for (int k = 0; k < kSampleSteps; ++k)
#pragma unroll
      for (int j = 0; j < 4; ++j) better(tx, ti, x[k][j], (v4_0 + k * 32) * 4 + j);
    if (!noisy) {
      bs = tx; bi = ti;
    } else {
      float wx = tx;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) wx = fmaxf(wx, __shfl_xor_sync(0xFFFFFFFFu, wx, o));
      float run = -INFINITY;
      if (tx == wx && ti != 0x7FFFFFFF) {                // one lane, or a few that tie
        uint32_t w[4];
        noise_bits(ti >> 2, w);
        const int j = ti & 3;
        bs = exact(tx, j == 0 ? w[0] : j == 1 ? w[1] : j == 2 ? w[2] : w[3]);
        bi = ti;
        const unsigned long long mine = pack_best(bs, bi), seen = atomicMax(a.best + slot, mine);
        run = unpack_score(seen > mine ? seen : mine);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) run = fmaxf(run, __shfl_xor_sync(0xFFFFFFFFu, run, o));
#pragma unroll
      for (int k = 0; k < kSampleSteps; ++k) {
        if (k >= steps) break;
        const int v4 = v4_0 + k * 32;
        const float top = fmaxf(fmaxf(x[k][0], x[k][1]), fmaxf(x[k][2], x[k][3])) * inv_t;
        if (!__any_sync(0xFFFFFFFFu, top >= run - kNoiseMax || run == -INFINITY)) continue;
        uint32_t w[4];
        noise_bits(v4, w);
        float sc[4], wm = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          sc[j] = fmaf(x[k][j], inv_t, fast_gumbel(uniform_from_bits(w[j])));
          wm = fmaxf(wm, sc[j]);
        }
        const float need = score_needed(run);
        if (!__any_sync(0xFFFFFFFFu, wm >= need)) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (sc[j] >= need) better(bs, bi, exact(x[k][j], w[j]), v4 * 4 + j);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xFFFFFFFFu, wm, o));
        run = fmaxf(run, wm);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float os = __shfl_xor_sync(0xFFFFFFFFu, bs, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
    better(bs, bi, os, oi);
  }
  if (DIRECT && (noisy || gridDim.y > 1)) {
    // one atomic per block: with few slots the warps' own would queue up at a few addresses
    __shared__ unsigned long long s_best[kSampleThreads / 32];
    if (lane == 0) s_best[threadIdx.x >> 5] = bi != 0x7FFFFFFF ? pack_best(bs, bi) : 0ull;
    __syncthreads();
    if (threadIdx.x != 0) return;
    unsigned long long top = s_best[0];
#pragma unroll
    for (int w = 1; w < kSampleThreads / 32; ++w) top = s_best[w] > top ? s_best[w] : top;
    if (top != 0ull) atomicMax(a.best + slot, top);
    return;
  }
  if (lane == 0 && bi != 0x7FFFFFFF) atomicMax(a.best + slot, pack_best(bs, bi));
}

// token[slot] = id held in best[slot]; best is cleared for the next use.
__global__ void sample_finalize_kernel(unsigned long long* best, const int32_t* slot_row, int32_t* token, int n) {
  RSD_PDL_SYNC();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (slot_row[i] >= 0) token[i] = (int32_t)(0xFFFFFFFFu - (uint32_t)(best[i] & 0xFFFFFFFFull));
  best[i] = 0ull;
}

cudaError_t launch_sample_finalize(unsigned long long* best, const int32_t* slot_row, int32_t* token, int n, cudaStream_t s) {
  RSD_LAUNCH((sample_finalize_kernel), (n + 255) / 256, 256, 0, s, best, slot_row, token, n);
  return launched(1);
}

// Leaves the winners packed in a.best (which must be zero on entry); when a.token is given a second
// kernel unpacks them into a.token and clears a.best.
cudaError_t launch_sample(const SampleArgs& a, cudaStream_t s) {
  if (a.n_slots <= 0) return cudaSuccess;
  // Runs of 128 ids per warp: the fewest that leave one wave of kSampleBlocks blocks per SM (8 x 151936 ids, greedy, the call's
  // other two nodes included: 600 blocks 10.4 us, 400 blocks 8.3).  Up to 1.5 million ids exact noise for all of them takes less
  // than the shortcuts' two dependent rounds: shortcuts / all, 8 x 151936 ids 15.2 / 11.3 us, 3 x 151936 12.5 / 9.4, 8 x 1024
  // 8.3 / 6.3; beyond it more, 32 x 151936 peaked logits 18.7 / 24.7.
  const int runs = (a.v_limit + 127) / 128, warps = kSampleThreads / 32;
  int steps = 1;
  while (steps < kSampleSteps && (long)a.n_slots * ((runs + warps * steps - 1) / (warps * steps)) > 148L * kSampleBlocks) ++steps;
  const dim3 grid(a.n_slots, (runs + warps * steps - 1) / (warps * steps));
  if ((long)a.n_slots * a.v_limit <= 1500000) RSD_LAUNCH((sample_kernel<true>), grid, kSampleThreads, 0, s, a, steps);
  else RSD_LAUNCH((sample_kernel<false>), grid, kSampleThreads, 0, s, a, steps);
  if (a.token == nullptr) return launched(1);
  const cudaError_t e = launched(1);
  return e != cudaSuccess ? e : launch_sample_finalize(a.best, a.slot_row, a.token, a.n_slots, s);
}

__global__ void philox_kernel(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int n) {
  RSD_PDL_SYNC();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 r = philox4x32_10(make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]),
                                make_uint2(key[0], key[1]));
  out[4 * i] = r.x; out[4 * i + 1] = r.y; out[4 * i + 2] = r.z; out[4 * i + 3] = r.w;
}

cudaError_t launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  RSD_LAUNCH((philox_kernel), (n + 255) / 256, 256, 0, s, ctr, key, out, n);
  return launched(1);
}

// ---------------------------------------------------------------------------------------------
// PRM step scoring head: gathers the hidden state of each row's last step token, applies the final
// RMSNorm, projects to a scalar and squashes it (Appendix B.3; score in [0,1], Section 3 "Models").
// ---------------------------------------------------------------------------------------------
template <typename WT>
__global__ void reward_kernel(const float* __restrict__ x, const WT* __restrict__ final_norm, const WT* __restrict__ w_r,
                              int head_kind, const int32_t* __restrict__ last_idx, int t0, int T, int d, float eps,
                              float* __restrict__ reward) {
  RSD_PDL_SYNC();
  __shared__ float red[33];
  const int row = blockIdx.x;
  const int idx = last_idx[row];
  if (idx < t0 || idx >= t0 + T) return;
  const float* xr = x + (size_t)(idx - t0) * d;
  float ss = 0.f, dot = 0.f;
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    const float v = xr[i];
    ss += v * v;
    dot += v * to_f32(final_norm[i]) * to_f32(w_r[i]);
  }
  ss = block_sum(ss, red);
  dot = block_sum(dot, red);
  if (threadIdx.x == 0) {
    const float a = dot * rsqrtf(ss / (float)d + eps);
    reward[row] = head_kind == 2 ? a : 1.f / (1.f + expf(-a));
  }
}

cudaError_t launch_reward(int dtype, const float* x, const void* final_norm, const void* w_r, int head_kind,
                          const int32_t* last_idx, int t0, int T, int d, float eps, float* reward, int n_rows,
                          cudaStream_t s) {
  if (n_rows <= 0) return cudaSuccess;
  if (dtype == 1)
    RSD_LAUNCH((reward_kernel<__nv_bfloat16>), n_rows, 256, 0, s, x, (const __nv_bfloat16*)final_norm, (const __nv_bfloat16*)w_r, head_kind, last_idx, t0, T, d, eps, reward);
  else
    RSD_LAUNCH((reward_kernel<float>), n_rows, 256, 0, s, x, (const float*)final_norm, (const float*)w_r, head_kind, last_idx, t0, T, d, eps, reward);
  return launched(1);
}

}  // namespace rsd
