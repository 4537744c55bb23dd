// What the two tcgen05 chunk-attention kernels share: page boxes, shared-memory descriptors of the page tiles, tensor-memory
// loads and stores, the copy of a partly cached value page, output stores.
#pragma once

#include "common.cuh"
#include "kernels.cuh"
#include "tc_ptx.cuh"

namespace rsd {
namespace chunk {

using namespace tc;

constexpr int kHd = 128;
constexpr int kBlockBytes = 4096;                   // keys (or values) of one page and KV head
constexpr uint32_t kProbeLimit = 1u << 18;          // polls of a bounded wait (a healthy wait ends within microseconds)
// PROBE (reached only through the wait-probe entry): the fetch warp issues NO copy, so that the first tile never comes; the MMA
// warp's wait, cut to this many polls, runs out, and the kernel must take its failure path -- error flag raised, softmax warps
// released, tensor memory freed, clean return -- with nothing in flight.
constexpr uint32_t kProbePolls = 4096;

// Writes of this thread to shared memory become visible to the tensor cores.
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The box of a tensor map whose first block coordinate is `blk` (all inner coordinates 0).
__device__ __forceinline__ void tma_load_block_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int blk) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(0), "r"(blk) : "memory");
}
__device__ __forceinline__ void tma_load_block_5d(void* dst, const CUtensorMap* map, uint64_t* bar, int blk) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %3, %3, %3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(0), "r"(blk) : "memory");
}

// Shared-memory matrix descriptors of K-major operands (leading byte offset unused, version 1).  A later k-step or
// half of the same tile is the descriptor plus its byte offset / 16: shared-memory addresses fit the 14-bit field.
// 128-byte swizzle: rows of 128 bytes, groups of 8 rows `sbo` bytes apart.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// 32-byte swizzle: rows of 32 bytes (one K = 16 step), groups of 8 rows 256 bytes apart.
__device__ __forceinline__ uint64_t desc_sw32(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (1ull << 16) | ((uint64_t)(256 >> 4) << 32) | (1ull << 46) | (6ull << 61);
}

// D (tensor memory) (+)= A (tensor memory: 128 lanes x 8 columns of fp16 pairs, one K = 16 step) * B (shared memory)
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
// ... from a converged warp, by the lane with on != 0.
__device__ __forceinline__ void umma_f16_ts_if(uint32_t on, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc), "r"(on) : "memory");
}
// 16 (32) registers of this thread into 16 (32) consecutive columns of its tensor-memory lane.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  tmem_st16(taddr, r);
  tmem_st16(taddr + 16, r + 16);
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);         // .x (the low 16 bits) = lo: the element with the even index
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 32 consecutive columns of this warp's tensor-memory lanes, one per register.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Bounded wait that leaves the issue slots to the warps with work: a short spin (most waits end within a few hundred
// cycles), then suspended polls.
__device__ __forceinline__ bool wait_sleep(uint64_t* bar, uint32_t parity, volatile uint32_t* stop) {
  for (int i = 0; i < 64; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  for (uint32_t i = 0; i < (1u << 19); ++i) {
    if (mbar_try_wait_sleep(bar, parity, 1000)) return true;
    if (*stop) return false;
  }
  return false;
}

// ... by a whole warp, with one answer for all lanes: what follows (tensor-memory loads and stores, votes) takes the warp together,
// and a barrier that completes or a stop that is raised between two lanes' polls would part it.
__device__ __forceinline__ bool wait_sleep_warp(uint64_t* bar, uint32_t parity, volatile uint32_t* stop) {
  const bool ok = wait_sleep(bar, parity, stop);
  return __all_sync(0xFFFFFFFFu, ok) != 0;
}

template <typename OT> __device__ __forceinline__ void store16(OT* hi, OT* lo, size_t o, const float* v);
template <> __device__ __forceinline__ void store16<float>(float* hi, float*, size_t o, const float* v) {
#pragma unroll
  for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(hi + o + 4 * i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}
template <> __device__ __forceinline__ void store16<__half>(__half* hi, __half*, size_t o, const float* v) {
  __align__(16) __half2 h[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) h[i] = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
  *reinterpret_cast<uint4*>(hi + o) = *reinterpret_cast<const uint4*>(h);
  *reinterpret_cast<uint4*>(hi + o + 8) = *reinterpret_cast<const uint4*>(h + 4);
}
template <> __device__ __forceinline__ void store16<__nv_bfloat16>(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t o, const float* v) {
  __align__(16) __nv_bfloat16 h[16];
  __align__(16) __nv_bfloat16 l[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    h[i] = __float2bfloat16_rn(v[i]);
    l[i] = __float2bfloat16_rn(v[i] - __bfloat162float(h[i]));
  }
  *reinterpret_cast<uint4*>(hi + o) = *reinterpret_cast<const uint4*>(h);
  *reinterpret_cast<uint4*>(hi + o + 8) = *reinterpret_cast<const uint4*>(h + 8);
  if (lo != nullptr) {
    *reinterpret_cast<uint4*>(lo + o) = *reinterpret_cast<const uint4*>(l);
    *reinterpret_cast<uint4*>(lo + o + 8) = *reinterpret_cast<const uint4*>(l + 8);
  }
}

// The values of a partly cached page (global: [128 dims][16 tokens]) into a page buffer of the value tile (rows of
// 32 bytes under the 32-byte swizzle: the 16-byte halves of a row trade places when bit 2 of the row is set), the
// tokens from `cached` on zeroed: their memory may hold anything, and 0 * NaN would poison the product.  One warp.
static __device__ __noinline__ void copy_partial_values(const __half* __restrict__ src, uint8_t* dst, int cached, int lane) {
#pragma unroll 1
  for (int j = 0; j < 8; ++j) {
    const int d = lane + 32 * (j >> 1), c = j & 1;
    __align__(16) __half hv[8];
    *reinterpret_cast<uint4*>(hv) = *reinterpret_cast<const uint4*>(src + (size_t)d * kPageTokens + c * 8);
#pragma unroll
    for (int x = 0; x < 8; ++x)
      if (c * 8 + x >= cached) hv[x] = __float2half_rn(0.f);
    *reinterpret_cast<uint4*>(dst + d * 32 + ((c ^ ((d >> 2) & 1)) << 4)) = *reinterpret_cast<const uint4*>(hv);
  }
  fence_async_smem();
}

// 128 consecutive columns of this warp's tensor-memory lanes, one per register, behind one wait.
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld128(uint32_t taddr, float* v) {
  uint32_t r[128];
#pragma unroll
  for (int c = 0; c < 128; c += 32) tmem_ld32_async(taddr + c, r + c);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 128; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace chunk
}  // namespace rsd
