// A whole decode phase of a small model over up to eight rows in one launch (sm_100a): every iteration's embedding, layers, head,
// sampling and row update, until no row is left.
//
// A model of a few dozen MB takes an iteration of 15 to 25 dependent steps, each of which is over in a microsecond once its input is
// there.  As kernels they cost 2 to 5 us each, whatever they do (launch, wait, first loads, drain); here they are phases of
// one cooperative launch, a CTA per SM, and a phase costs the way of its input through L2 and a few hundred instructions.  An iteration, us, kernels of
// a graph / here: bf16, 2 x 512 and 3 x 768 columns, 8 rows 42 / 32 and 67 / 54, 1 row 39 / 31 and 57 / 52; fp32, 2 x 256 and 4 x 512 columns,
// 4 rows 37 / 29 and 85 / 66, 8 rows 55 / 38 and 124 / 93; a phase has 10 us more to start.
//   weights    the CTA's weight rows of all phases, layers and iterations, in order, come by TMA into a ring of 16 KB stages, requested as soon as
//              the stages are free.  Weights depend on nothing, so they are in shared memory before the phase that needs them.
//   exchange   there is no barrier between phases.  A result goes to L2 as words that can never be kEmpty, into slots that are kEmpty
//              until then, and who needs it polls the words themselves (kernel boundary 2.2-2.7 us; barrier by a counter and a load behind it 1.8-2.2;
//              this 0.9-1.3 for 512-1536 columns, 148 CTAs).  Slots are written once an iteration and there are two sets of them:
//              an iteration fills one and empties the other.  Everybody sends the ids that it has sampled to everybody else: who has them all
//              knows that the set of this iteration has been read, and may empty it in the next.  The ids are also what orders everything that is not
//              polled itself: a CTA's ids are a release (behind a barrier, a fence by the lanes that send them), whoever has polled them acquires (a fence by the lanes
//              that polled, ahead of a barrier).  So the slots that a CTA has emptied are empty for all who poll them in the iteration after, and the keys and
//              values that it has put into pages are there for the CTAs that read them from then on (fp32: the other heads of the group).
//   products   units of sixteen weight rows (two groups of eight) and all of K; which rows meet in a unit is what its epilogue needs together: the
//              dims that rotate with one another, gate and up rows of the same features, sixteen features of the residual stream.
//              bf16: hi + lo operand pairs, eight rows of each as the 16 rows of an mma.sync tile (as in gemm_rows.cu; tcgen05 has no tile this
//              narrow), the warps share K, chains of at most eight MMAs; operands are exchanged in the order of the MMA's registers.  fp32: a warp
//              takes one row of each group, the operand sits in shared memory.
//   attention  a (slot, KV head) pair per CTA (bf16; fp32: a (slot, head) pair), as in attn_decode.cu and attn_generic_kernel; the new key
//              and value come with the queries and go into the page from here.
// The residual stream never leaves the CTA that owns its features.
// What bounds it: per step 1 us of exchange, 0.2-0.9 us of products, 0.5 us in which the warps' parts meet, 0.3 us of epilogue; instructions count,
// and so does every register spilled (above).
// Every wait is bounded; a wait that expires raises the error flag, every CTA then leaves within its own bounds.
#include <cuda.h>

#include <algorithm>
#include <memory>
#include <new>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "sampling.cuh"
#include "tc_ptx.cuh"

namespace rsd {

namespace {

using namespace tc;

constexpr int kWarps = 8, kWorkers = 32 * kWarps, kBlock = kWorkers;    // (a ninth warp would leave 168 registers a thread, and spills that the little L1 beside the shared memory does not hold)
constexpr int kMaxSteps = 128;                 // of a CTA in an iteration
constexpr int kRows = 8;                       // slots at most
constexpr int kStage = 16384;                  // two boxes of eight weight rows: 512 bf16 or 256 fp32 columns
constexpr int kSlabs = 4;                      // stages of a unit at most (bf16), i.e. K <= 2048
constexpr int kMaxK = 2048;
constexpr uint32_t kEmpty = 0xFFFFFFFFu;       // a NaN that no conversion or sum gives
constexpr uint32_t kPolls = 1u << 21;          // of L2, half a microsecond or more each
constexpr int kOwn = 4;                        // units of the residual stream that a CTA owns at most
constexpr int kSharers = 4;                    // callers that share the SMs at most; more take turns

struct alignas(128) ResidentLayer {
  CUtensorMap w[4];                            // qkv, wo, gate/up, down
  const void *norm1, *norm2;
  char* kv;
};

struct alignas(128) ResidentParams {
  CUtensorMap head;
  int L, d, H, KV, hd, F, V, v_limit, max_pages, model_id;
  float eps, temperature;
  uint64_t seed;
  const void *embed, *final_norm;
  const float2* rope;
  const int32_t* page_table;
  uint32_t* slots;                             // two sets of exchange slots
  uint32_t set_words, at_x, at_y, at_q, at_a, at_f, at_s;   // words of a set; where its parts begin
  int* err;
  float* dbg_logits;                           // null, or [rows][C][V]
};

enum Phase { kQkv, kAttn, kWo, kGateUp, kDown, kHead };

// ---- exchange ------------------------------------------------------------------------------------------
__device__ __forceinline__ void ld4_if(bool on, uint4& v, const uint32_t* p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %4, 0;\n\t@q ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%5];\n\t}"
               : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "r"((uint32_t)on), "l"(p) : "memory");
}
__device__ __forceinline__ void ld2_if(bool on, uint2& v, const uint32_t* p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%3];\n\t}"
               : "+r"(v.x), "+r"(v.y) : "r"((uint32_t)on), "l"(p) : "memory");
}
__device__ __forceinline__ void ld1_if(bool on, uint32_t& v, const uint32_t* p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q ld.relaxed.gpu.global.u32 %0, [%2];\n\t}"
               : "+r"(v) : "r"((uint32_t)on), "l"(p) : "memory");
}
__device__ __forceinline__ void st_word(uint32_t* p, uint32_t a) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(a) : "memory"); }
__device__ __forceinline__ void st_word(uint32_t* p, uint2 a) { asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(a.x), "r"(a.y) : "memory"); }
__device__ __forceinline__ void st_word(uint32_t* p, uint4 a) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w) : "memory");
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ bool full(uint32_t v) { return v != kEmpty; }
__device__ __forceinline__ bool full(uint4 v) { return v.x != kEmpty && v.y != kEmpty && v.z != kEmpty && v.w != kEmpty; }
// an fp32 result as a word: arithmetic gives one NaN, moves may pass any
__device__ __forceinline__ uint32_t word_of(float v) { const uint32_t b = __float_as_uint(v); return b == kEmpty ? 0x7FFFFFFFu : b; }
__device__ __forceinline__ uint32_t pack_bf(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}
// two neighbouring operand values as (hi, hi) and (lo, lo) words
__device__ __forceinline__ uint2 operand_words(float a, float b) {
  __nv_bfloat16 h[2], l[2];
  store_operand<__nv_bfloat16>(h, l, 0, a);
  store_operand<__nv_bfloat16>(h, l, 1, b);
  return make_uint2(pack_bf(h[0], h[1]), pack_bf(l[0], l[1]));
}

// The state of a worker thread that the waits share.
struct Wait {
  int* err;
  bool dead;                                   // a wait has expired here or another CTA has raised the flag
  __device__ __forceinline__ bool give_up(uint32_t polls) {
    if (polls >= kPolls) { atomicCAS(err, 0, -5); dead = true; }
    else if ((polls & 1023u) == 1023u && *(volatile int*)err != 0) dead = true;
    return dead;
  }
};

// N vectors of this lane, those of `need`, until none of them has an empty word; the whole warp stays together.
template <int N, typename V, typename Load>
__device__ __forceinline__ void poll(V (&v)[N], uint32_t need, Wait& w, Load load) {
  for (uint32_t polls = 0; !w.dead; ++polls) {
#pragma unroll
    for (int i = 0; i < N; ++i) load((need >> i) & 1u, v[i], i);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (full(v[i])) need &= ~(1u << i);
    if (!__any_sync(0xFFFFFFFFu, need != 0)) return;
    w.give_up(polls);
    w.dead = __any_sync(0xFFFFFFFFu, w.dead);
  }
}

// Barrier of the workers; true if any of them brings `flag`, for all alike.
__device__ __forceinline__ bool sync_or(bool flag) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, 256, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)flag) : "memory");
  return r != 0;
}

// ---- weight ring -----------------------------------------------------------------------------------------
struct Ring {
  int n, s;
  uint32_t phase;
  __device__ __forceinline__ void step() { if (++s == n) { s = 0; phase ^= 1u; } }
};

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// Unit u of a phase: the first rows of its two groups.
__device__ __forceinline__ void unit_rows(Phase ph, int u, int hd, int F, int& r0, int& r1) {
  if (ph == kQkv) {                            // eight dims of a head and those that they turn with
    const int per = hd / 16;
    r0 = (u / per) * hd + (u % per) * 8;
    r1 = r0 + hd / 2;
  } else if (ph == kGateUp) {
    r0 = u * 8;
    r1 = F + r0;
  } else {
    r0 = u * 16;
    r1 = r0 + 8;
  }
}

// What this CTA does in an iteration, in order: units u0, u0 + grid, ... below n_units of a product, or pairs of the attention.
struct Step {
  int ph, l, u0, n_units, K;
  uint32_t src, dst;                           // words of a set: the operand, the first result
  const void *gain, *next;                     // norm ahead of the product (fp32; bf16: of the embedding), norm behind it (bf16)
  const CUtensorMap* map;
  char* kv;
};

template <bool F32> struct StageK { static constexpr int value = F32 ? 256 : 512; };

// bf16: the warp's eight columns of 64 in each stage; K % 64 == 0.
__device__ __forceinline__ void ldmatrix4(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_top(float& d0, float& d1, uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {
  float x, y;                                  // rows 8..15 are padding (attn_decode.cu)
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%8,%5,%8}, {%6,%7}, {%0,%1,%9,%9};"
               : "+f"(d0), "+f"(d1), "=f"(x), "=f"(y) : "r"(a0), "r"(a2), "r"(b0), "r"(b1), "r"(0u), "f"(0.f));
}
__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
  const __half2 v = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void pack_h2_split(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __half ah = __float2half_rn(a), bh = __float2half_rn(b);
  hi = pack_h2(__half2float(ah), __half2float(bh));
  lo = pack_h2(a - __half2float(ah), b - __half2float(bh));
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Every line of 128 bytes that others poll is written by one store of one warp: a line that several stores complete is taken away from its readers by
// each of them, half a microsecond a time (the ids of 148 CTAs, sixteen to a line: 7 us).  Hence, in words, with lane = 4 row + t:
//   X, Y (residual stream) [unit of 16 columns][lane][4]: bf16 the MMA's (hi, lo) of columns 2t, 2t + 1 and 2t + 8, 2t + 9, fp32 those four columns;
//                          bf16 has the sums of squares behind it, [unit][32], eight in use
//   Q (queries, keys, values) [unit][lane][4]: columns 2t, 2t + 1 of the unit's two groups, fp32
//   A (attention) bf16 [32 columns][row][32], the MMA's words of two units; fp32 [row][column]
//   F (SwiGLU) [unit of 8][lane][2]: columns 2t, 2t + 1, bf16 (hi, lo)
//   ids [CTA][32]: (score, id + 1) of eight rows
__device__ __forceinline__ uint32_t attn_word(int f, int m) {               // bf16: of columns f, f + 1
  const int p = (f & 15) / 2;
  return (uint32_t)(((f >> 5) * kRows + m) * 32 + ((f >> 4) & 1) * 16 + (p & 3) * 4 + (p >> 2) * 2);
}

__device__ __forceinline__ float gumbel(uint32_t bits) { return -logf(-logf(uniform_from_bits(bits))); }

// Shared memory behind the ring.
template <bool F32, bool EXT> struct ResidentCfg {
  static constexpr int kPageBytes = (EXT ? 4 : 2) * kPageTokens * 128 * 2;
  static constexpr int kBufs = EXT ? 1 : 2;
  // fp32: the operand rows; bf16: pages, kBufs a warp, whose place the warp's outputs take
  static constexpr int kBuffer = F32 ? kRows * kMaxK * 4 : kWarps * kBufs * kPageBytes;
  static constexpr int kStages = F32 ? 8 : 4;
  static_assert(kStages * (F32 ? 256 : 512) >= kMaxK, "the stages of a unit: they are requested behind the barrier of the unit before");
  static_assert(F32 || 8 * (128 + 8) * 4 <= kBufs * kPageBytes, "a warp's outputs");
  static constexpr size_t kSmem = 1024 + (size_t)kStages * kStage + kBuffer;
  static_assert(kSmem + 34 * 1024 <= 227 * 1024, "shared memory of one CTA");
};

template <bool F32, bool EXT, int MT>          // MT: rows of an fp32 product, 4 or 8
__global__ void __launch_bounds__(kBlock, 1)
decode_resident_kernel(const __grid_constant__ ResidentParams P, const ResidentLayer* __restrict__ layers, const __grid_constant__ RowState st,
                       int which, int phase, int n_slots, const __grid_constant__ LoopParams lp) {
  using Cfg = ResidentCfg<F32, EXT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* buffer = smem + (size_t)Cfg::kStages * kStage;
  __shared__ uint64_t bar_full[Cfg::kStages];
  __shared__ float red[2][F32 ? 1 : kWarps][2][kRows][8];
  __shared__ __align__(16) float s_ssq[kRows][kWarps];
  __shared__ float4 own[kOwn][32];             // residual stream of the CTA's features (bf16: as the epilogue's lanes hold it)
  __shared__ int s_row[kRows], s_pos[kRows], s_tok[kRows], s_flen[kRows], s_on[kRows], s_active, s_left, s_iter, s_n_steps;
  __shared__ float s_noise[kWarps][32][4];
  __shared__ float2 s_rope[kRows][64];         // the angles of the rows' positions
  __shared__ unsigned long long s_best[kWarps][kRows], s_top[kWarps][kRows];
  __shared__ Step s_steps[kMaxSteps];
  __shared__ int s_feed[4];                    // of the weight stream: step, unit, column, stages requested so far
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int grid = gridDim.x, d = P.d, hd = P.hd, n_qkv = (P.H + 2 * P.KV) * P.hd, hq = P.H * P.hd;
  const uint32_t x_words = (uint32_t)(d * kRows + d / 16 * 32);
  if (threadIdx.x == 0) {
    for (int i = 0; i < Cfg::kStages; ++i) mbar_init(&bar_full[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_left = st.n_active[0];
    s_iter = st.iter[0];
  }
  if (warp == 1) {
    const int m = lane & 7, row = m < n_slots ? st.pass_tok_row[m] : -1;
    if (lane < kRows) {
      s_row[m] = row;
      s_pos[m] = row >= 0 ? st.pass_tok_pos[m] : 0;
      s_tok[m] = row >= 0 ? st.pass_tok_id[m] : 0;
      s_flen[m] = row >= 0 ? st.forced_len[phase][row] : 0;
    }
    const unsigned on = __ballot_sync(0xFFFFFFFFu, row >= 0 && lane < kRows);
    if (lane == 0) s_active = (int)on;
  }
  if (warp == 2) {
    // The list of steps.  Units go round the CTAs, the phases' first ones where the phase before has its last, so that the CTAs of a phase are
    // waiting while those of the phase ahead of it work; wo and down have the same owners.
    int n = 0;
    for (int base = 0; base <= 5 * P.L; base += 32) {
      const int i = base + lane, l = i / 5;
      Step s{};
      s.ph = i == 5 * P.L ? kHead : i % 5;
      s.l = l;
      int off = 0;
      if (i < 5 * P.L) {
        const ResidentLayer* Ly = layers + l;
        s.kv = Ly->kv;
        if (s.ph == kQkv) { s.n_units = n_qkv / 16; s.K = d; s.src = P.at_x + l * x_words; s.dst = P.at_q + (uint32_t)(l * kRows * n_qkv); s.gain = Ly->norm1; s.map = &Ly->w[0]; }
        else if (s.ph == kAttn) { s.n_units = n_slots * (F32 ? P.H : P.KV); off = n_qkv / 16 + d / 16; s.src = P.at_q + (uint32_t)(l * kRows * n_qkv); s.dst = P.at_a + (uint32_t)(l * kRows * hq); }
        else if (s.ph == kWo) { s.n_units = d / 16; off = n_qkv / 16; s.K = hq; s.src = P.at_a + (uint32_t)(l * kRows * hq); s.dst = P.at_y + l * x_words; s.next = Ly->norm2; s.map = &Ly->w[1]; }
        else if (s.ph == kGateUp) { s.n_units = P.F / 8; s.K = d; s.src = P.at_y + l * x_words; s.dst = P.at_f + (uint32_t)(l * kRows * P.F); s.gain = Ly->norm2; s.map = &Ly->w[2]; }
        else { s.n_units = d / 16; off = n_qkv / 16; s.K = P.F; s.src = P.at_f + (uint32_t)(l * kRows * P.F); s.dst = P.at_x + (l + 1) * x_words; s.next = l + 1 < P.L ? layers[l + 1].norm1 : P.final_norm; s.map = &Ly->w[3]; }
      } else {
        s.n_units = (P.V + 15) / 16; s.K = d; s.src = P.at_x + P.L * x_words; s.gain = P.final_norm; s.map = &P.head;
      }
      s.u0 = ((int)blockIdx.x - off % grid + grid) % grid;
      const bool has = i <= 5 * P.L && s.u0 < s.n_units;
      const unsigned b = __ballot_sync(0xFFFFFFFFu, has);
      if (has) s_steps[n + __popc(b & ((1u << lane) - 1u))] = s;
      n += __popc(b);
    }
    if (lane == 0) s_n_steps = n;
  }
  __syncthreads();
  if (s_left == 0 || s_active == 0) return;
  const int n_steps = s_n_steps;

  // The weight stream: requests the CTA's next n stages.  By one lane, behind a barrier that all warps reach when they have read the stages that it fills.
  auto feed = [&](int n) {
    int step = s_feed[0], u = s_feed[1], k = s_feed[2];
    const int issued = s_feed[3];
    for (int i = 0; i < n; ++i) {
      const Step& sp = s_steps[step];
      int r0, r1;
      unit_rows((Phase)sp.ph, u, hd, P.F, r0, r1);
      const int stage = (issued + i) % Cfg::kStages;
      uint8_t* dst = smem + (size_t)stage * kStage;
      uint64_t* bar = &bar_full[stage];
      mbar_expect_tx(bar, kStage);
      if (F32) {
        tma_load_2d(dst, sp.map, bar, k, r0);
        tma_load_2d(dst + kStage / 2, sp.map, bar, k, r1);
      } else {
        tma_load_3d(dst, sp.map, bar, 0, r0, k / 64);
        tma_load_3d(dst + kStage / 2, sp.map, bar, 0, r1, k / 64);
      }
      k += StageK<F32>::value;
      if (k >= sp.K) {
        k = 0;
        u += grid;
        if (u >= sp.n_units) {
          do { step = step + 1 == n_steps ? 0 : step + 1; } while (s_steps[step].ph == kAttn);
          u = s_steps[step].u0;
        }
      }
    }
    s_feed[0] = step; s_feed[1] = u; s_feed[2] = k; s_feed[3] = issued + n;
  };
  // every CTA has gate/up units, so there is a product among its steps
  if (threadIdx.x == 0) {
    int step = 0;
    while (s_steps[step].ph == kAttn) ++step;
    s_feed[0] = step; s_feed[1] = s_steps[step].u0; s_feed[2] = 0; s_feed[3] = 0;
    feed(Cfg::kStages);
  }
  // Emptying, in iteration `it` >= 1: the set that iteration it - 1 has filled, which everybody has read once all ids of it - 1 are there, and of the four
  // places of the ids the one of it - 2.  The steps go round the warps; the ids of `it` make it known.
  auto empty_slots = [&](int it) {
    uint32_t* set = P.slots + ((it & 1) ? 0u : P.set_words);
    const uint2 e2 = make_uint2(kEmpty, kEmpty);
    const uint4 e4 = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    for (int i = warp; i < n_steps; i += kWarps) {
      const Step& sp = s_steps[i];
      if (sp.ph == kHead) continue;
      uint32_t* dst = set + sp.dst;
      for (int u = sp.u0; u < sp.n_units; u += grid) {
        if (sp.ph == kAttn) {
          const int per = F32 ? P.H : P.KV, cols = (F32 ? 1 : P.H / P.KV) * hd, m = u / per, f0 = (u % per) * cols;
          for (int k = 0; k < cols; k += 32) st_word(dst + (F32 ? m * hq + f0 + k : ((f0 + k) / 32 * kRows + m) * 32) + lane, kEmpty);
        } else if (sp.ph == kGateUp) {
          st_word(dst + (u * 32 + lane) * 2, e2);
        } else {
          st_word(dst + (u * 32 + lane) * 4, e4);
          if (!F32 && sp.ph != kQkv && lane < kRows) st_word(dst + d * kRows + u * 32 + lane, kEmpty);
        }
      }
    }
    if (warp == kWarps - 1) {
      if (F32) {                               // the embeddings
        for (int u = ((int)blockIdx.x - (n_qkv / 16) % grid + grid) % grid; u < d / 16; u += grid) st_word(set + P.at_x + (u * 32 + lane) * 4, e4);
      }
      if (it >= 2 && lane < 2 * kRows) st_word(P.slots + P.at_s + (((it - 2) & 3) * 160 + blockIdx.x) * 32 + lane, kEmpty);
    }
  };
  // ---------------- workers ----------------
  Wait wait{P.err, false};
  Ring ring{Cfg::kStages, 0, 0u};
  int turn = 0;                                // whose turn the next epilogue is (bf16)
  uint32_t* set = P.slots;                     // this iteration's slots
  unsigned active = (unsigned)s_active;
  const float inv_d = 1.f / (float)d;
  const bool noisy = P.temperature > 0.f;
  const float inv_t = noisy ? 1.f / P.temperature : 1.f;
  float best_score = -INFINITY;                // of this lane's row, among the ids that it has seen
  int best_id = 0x7FFFFFFF;
  int iter = s_iter;
  // Gumbel noise for this lane's ids of a head unit, u * 16 + 2t, + 1 and + 8, + 9, into s_noise.  (In a loop: the logarithms are long.)
  auto unit_noise = [&](int u) {
    const uint2 key = make_uint2((uint32_t)(P.seed & 0xFFFFFFFFull), (uint32_t)(P.seed >> 32));
#pragma unroll 1
    for (int i = 0; i < 2; ++i) {
      const uint4 r = philox4x32_10(make_uint4((uint32_t)(u * 4 + 2 * i + (t >> 1)), (uint32_t)(s_pos[g] + 1), (uint32_t)s_row[g], (uint32_t)P.model_id), key);
      s_noise[warp][lane][2 * i] = gumbel((t & 1) ? r.z : r.x);
      s_noise[warp][lane][2 * i + 1] = gumbel((t & 1) ? r.w : r.y);
    }
  };
  auto candidate = [&](int m, int id, float logit, int i) {
    if (id >= P.V) return;
    if (P.dbg_logits != nullptr) P.dbg_logits[((size_t)s_row[m] * st.C + iter) * P.V + id] = logit;
    if (id >= P.v_limit) return;
    const float sc = noisy ? fmaf(logit, inv_t, s_noise[warp][lane][i]) : logit;
    if (sc > best_score || (sc == best_score && id < best_id)) { best_score = sc; best_id = id; }
  };
  // RMSNorm's denominator of row m
  auto inv_rms = [&](int m) {
    const float4 a = *reinterpret_cast<const float4*>(&s_ssq[m][0]), b = *reinterpret_cast<const float4*>(&s_ssq[m][4]);
    return rsqrtf((((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w))) * inv_d + P.eps);
  };

  constexpr int NC = 2;                        // neighbouring columns that a lane finishes in each group of a unit
  // What becomes of a unit's sums of row m, columns n (, n + 1): v0 of the first group, v1 of the second.
  auto epilogue = [&](const Step& sp, int u, int m, int n, const float (&v0)[NC], const float (&v1)[NC]) {
    const float inv = inv_rms(m);
    uint32_t* dst = set + sp.dst;
    if (sp.ph == kQkv) {
      int r0, r1;
      unit_rows(kQkv, u, hd, P.F, r0, r1);
      const int dim = r0 % hd + n;             // (hd is 64 or 128)
      uint32_t a[NC], b[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        float x = v0[i] * inv, y = v1[i] * inv;
        if (r0 < hq + P.KV * hd) {
          const float2 cs = s_rope[m][dim + i];
          const float z = rotate_lo(x, y, cs);
          y = rotate_hi(x, y, cs);
          x = z;
        }
        a[i] = word_of(x); b[i] = word_of(y);
      }
      st_word(dst + (u * 32 + lane) * 4, make_uint4(a[0], a[1], b[0], b[1]));
    } else if (sp.ph == kGateUp) {
      const float x = swiglu(v0[0] * inv, v1[0] * inv), y = swiglu(v0[1] * inv, v1[1] * inv);
      st_word(dst + (u * 32 + lane) * 2, F32 ? make_uint2(word_of(x), word_of(y)) : operand_words(x, y));
    } else {
#pragma unroll
      for (int i = 0; i < 2 * NC; ++i) candidate(m, u * 16 + (i / NC) * 8 + n + i % NC, (i < NC ? v0[i % NC] : v1[i % NC]) * inv, i);
    }
  };
  // x += v for the residual stream's features u * 16 + n (, + 1) and + 8, and x to those who wait: bf16 x * gain as hi + lo and the sums of
  // squares, fp32 x itself.  All lanes of a warp call it.
  auto residual = [&](uint32_t* dst, int u, int ul, int m, bool on, const float (&gain)[4], const float (&v0)[NC], const float (&v1)[NC]) {
    float4 x = own[ul][lane];
    x.x += v0[0]; x.y += v0[1]; x.z += v1[0]; x.w += v1[1];
    own[ul][lane] = x;
    uint32_t* at = dst + (u * 32 + lane) * 4;
    if (F32) {
      if (on) st_word(at, make_uint4(word_of(x.x), word_of(x.y), word_of(x.z), word_of(x.w)));
    } else {
      const uint2 lo = operand_words(x.x * gain[0], x.y * gain[1]), hi = operand_words(x.z * gain[2], x.w * gain[3]);
      if (on) st_word(at, make_uint4(lo.x, lo.y, hi.x, hi.y));
      float ss = (x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w);
      ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 1);
      ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 2);
      if (on && t == 0) st_word(dst + d * kRows + u * 32 + m, word_of(ss));
    }
  };
  auto wait_stage = [&](int stage, uint32_t par) {
    if (wait.dead) return;
    for (uint32_t i = 0; !mbar_try_wait_sleep(&bar_full[stage], par, 1000); ++i)
      if (wait.give_up(i)) break;
    wait.dead = __any_sync(0xFFFFFFFFu, wait.dead);
  };

  // Behind the barrier of a unit: its stages are free.  Not by the warp of the epilogue.
  auto behind_unit = [&](int stages) {
    if (warp == ((turn + 4) & (kWarps - 1)) && lane == 0) feed(stages);
  };

  // One product: its operand, the CTA's units, their epilogues; false when a wait has expired.
  auto product = [&](const Step& sp) -> bool {
    const int K = sp.K, n_units = sp.n_units, ph = sp.ph;
    const uint32_t* in = set + sp.src;
    const bool normed = ph == kQkv || ph == kGateUp || ph == kHead;
    if constexpr (F32) {
      // a warp, or two, per row of the operand
      constexpr int PER = kWarps / MT;
      const int m = warp % MT, part = warp / MT, n_vec = K / 4, Kp = (K + 255) & ~255;
      const bool row_on = ((active >> m) & 1u) != 0;
      if (ph == kHead && noisy && ((active >> g) & 1u)) {    // of the first unit whose epilogue is this warp's
        const int ahead = sp.u0 + ((warp - turn) & (kWarps - 1)) * grid;
        if (ahead < n_units) unit_noise(ahead);
      }
      const int waited = min((K + 255) / 256, Cfg::kStages);             // weights of the first unit, ahead of the operand
      {
        Ring r = ring;
        for (int i = 0; i < waited; ++i) { wait_stage(r.s, r.phase); r.step(); }
      }
      auto gather = [&](auto nv) -> bool {
        constexpr int NV = decltype(nv)::value;
        constexpr bool kAhead = NV <= 4;       // the gains of a norm ahead of the operand
        uint4 v[NV];
        float gn[kAhead ? NV : 1][4];
        uint32_t need = 0;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int k = (i * PER + part) * 32 + lane;
          v[i] = make_uint4(0, 0, 0, 0);
          if (row_on && k < n_vec) need |= 1u << i;
          if (kAhead && normed && k < n_vec) {
            const float* gp = (const float*)sp.gain + (k >> 2) * 16 + (k & 3) * 2;
            gn[kAhead ? i : 0][0] = gp[0]; gn[kAhead ? i : 0][1] = gp[1]; gn[kAhead ? i : 0][2] = gp[8]; gn[kAhead ? i : 0][3] = gp[9];
          }
        }
        poll<NV>(v, need, wait, [&](bool on, uint4& x, int i) {
          const int k = (i * PER + part) * 32 + lane;
          ld4_if(on, x, in + (ph == kWo ? m * K + k * 4 : ph == kDown ? (k >> 1) * 64 + m * 8 + (k & 1) * 4 : (k >> 2) * 128 + m * 16 + (k & 3) * 4));
        });
        if (sync_or(wait.dead)) return false;  // and nobody reads the operand before this one any more
        float* xs = reinterpret_cast<float*>(buffer) + m * Kp;
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int k = (i * PER + part) * 32 + lane;
          if (k * 4 >= Kp) continue;
          float4 x = make_float4(__uint_as_float(v[i].x), __uint_as_float(v[i].y), __uint_as_float(v[i].z), __uint_as_float(v[i].w));
          if (normed) {                        // columns 2t, 2t + 1, 2t + 8, 2t + 9 of a unit
            const int c = (k >> 2) * 16 + (k & 3) * 2;
            if (k < n_vec) {
              ss += (x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w);
              const float* gp = (const float*)sp.gain + c;
              x.x *= kAhead ? gn[kAhead ? i : 0][0] : gp[0]; x.y *= kAhead ? gn[kAhead ? i : 0][1] : gp[1];
              x.z *= kAhead ? gn[kAhead ? i : 0][2] : gp[8]; x.w *= kAhead ? gn[kAhead ? i : 0][3] : gp[9];
            }
            *reinterpret_cast<float2*>(xs + c) = make_float2(x.x, x.y);
            *reinterpret_cast<float2*>(xs + c + 8) = make_float2(x.z, x.w);
          } else {
            *reinterpret_cast<float4*>(xs + k * 4) = x;
          }
        }
        if (normed) {
          ss = warp_sum(ss);
          if (lane == part || (part == 0 && lane >= PER && lane < kWarps)) s_ssq[m][lane] = lane == part ? ss : 0.f;
        }
        return true;
      };
      bool ok;
      // (of Kp columns, not of K: the products take whole stages, and what lies beyond K must be zeros like the weights there)
      const int nv = (Kp / 4 + 32 * PER - 1) / (32 * PER);
      if (nv <= 1) ok = gather(std::integral_constant<int, 1>());
      else if (nv <= 2) ok = gather(std::integral_constant<int, 2>());
      else if (nv <= 4) ok = gather(std::integral_constant<int, 4>());
      else if (nv <= 8) ok = gather(std::integral_constant<int, 8>());
      else ok = gather(std::integral_constant<int, 16>());
      if (!ok) { wait.dead = true; return false; }
      (void)sync_or(false);
      // A warp takes a row of each group.  (Two rows of each and half of the columns read a third less of the operand and have twice the sums over lanes:
      // an iteration of four fp32 layers of 512 columns, 4 / 8 rows, 69 / 96 us so, 72 / 105 then.)
      const float* xb = reinterpret_cast<const float*>(buffer) + lane * 4;
      int ul = 0;
      for (int u = sp.u0; u < n_units; u += grid, ++ul, ++turn) {
        // a stage's products by themselves, then into the sums: chains of four and of K / 256 instead of one of K / 64 (a layer of 2048
        // columns, logits against fp64: 3.8e-7, with the long chain 4.3, by single kernels 4.0)
        float v[2 * MT];
#pragma unroll
        for (int i = 0; i < 2 * MT; ++i) v[i] = 0.f;
        int at = 0;
#pragma unroll 1
        for (int k0 = 0; k0 < K; k0 += 256, ++at) {
          if (ul > 0 || at >= waited) wait_stage(ring.s, ring.phase);
          const uint8_t* stg = smem + (size_t)ring.s * kStage + warp * 1024 + lane * 16;
          float acc[2 * MT][2];
#pragma unroll
          for (int blk = 0; blk < 2; ++blk) {
            const float4 w0 = *reinterpret_cast<const float4*>(stg + blk * 512), w1 = *reinterpret_cast<const float4*>(stg + kStage / 2 + blk * 512);
#pragma unroll
            for (int mm = 0; mm < MT; ++mm) {
              const float4 x = *reinterpret_cast<const float4*>(xb + mm * Kp + k0 + blk * 128);
              acc[mm][0] = fmaf(w0.y, x.y, blk == 0 ? w0.x * x.x : fmaf(w0.x, x.x, acc[mm][0]));
              acc[mm][1] = fmaf(w0.w, x.w, blk == 0 ? w0.z * x.z : fmaf(w0.z, x.z, acc[mm][1]));
              acc[MT + mm][0] = fmaf(w1.y, x.y, blk == 0 ? w1.x * x.x : fmaf(w1.x, x.x, acc[MT + mm][0]));
              acc[MT + mm][1] = fmaf(w1.w, x.w, blk == 0 ? w1.z * x.z : fmaf(w1.z, x.z, acc[MT + mm][1]));
            }
          }
#pragma unroll
          for (int i = 0; i < 2 * MT; ++i) v[i] += acc[i][0] + acc[i][1];
          ring.step();
        }
        // over the lanes: each step halves the values that a lane carries; lane ends with value lane / (32 / (2 MT))
#pragma unroll
        for (int n = 2 * MT, o = 16; o > 0; o >>= 1) {
          if (n > 1) {
            n /= 2;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < n; ++i) {
              const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
              v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
            }
          } else {
            v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
          }
        }
        constexpr int LPV = 16 / MT;           // lanes that hold the same value: row mm of a group's column `warp`
        if (lane % LPV == 0) red[turn & 1][0][lane >> 4][(lane & 15) / LPV][warp] = v[0];
        if (ph == kQkv) asm volatile("cp.async.wait_all;" ::: "memory");     // the angles
        if (sync_or(wait.dead)) { wait.dead = true; return false; }
        behind_unit((K + 255) / 256);
        if (warp == (turn & (kWarps - 1)) && g < MT) {
          const float2 p0 = *reinterpret_cast<const float2*>(&red[turn & 1][0][0][g][2 * t]), p1 = *reinterpret_cast<const float2*>(&red[turn & 1][0][1][g][2 * t]);
          const float v0[NC] = {p0.x, p0.y}, v1[NC] = {p1.x, p1.y};
          const bool on = ((active >> g) & 1u) != 0;
          if (ph == kWo || ph == kDown) {
            const float none[4] = {};
            residual(set + sp.dst, u, ul, g, on, none, v0, v1);
          } else if (on) {
            epilogue(sp, u, g, 2 * t, v0, v1);
          }
          if (ph == kHead && noisy && on && u + kWarps * grid < n_units) unit_noise(u + kWarps * grid);
        }
      }
      return true;
    } else {
      const bool mine = ((active >> g) & 1u) != 0;
      const int slabs = (K + 511) / 512;
      // Ahead of the operand: what the first epilogues need beside the sums, and the first unit's weights.
      float extra[4] = {};
      auto fill_extra = [&](int u) {
        if (ph == kHead) {
          if (noisy) unit_noise(u);
        } else {
          const __nv_bfloat16* gp = (const __nv_bfloat16*)sp.next + u * 16 + 2 * t;
          extra[0] = to_f32(gp[0]); extra[1] = to_f32(gp[1]); extra[2] = to_f32(gp[8]); extra[3] = to_f32(gp[9]);
        }
      };
      const bool extras = (ph == kHead || ph == kWo || ph == kDown) && mine;
      const int ahead = sp.u0 + ((warp - turn) & (kWarps - 1)) * grid;   // the first unit whose epilogue is this warp's
      {
        Ring r = ring;
        for (int i = 0; i < slabs; ++i) { wait_stage(r.s, r.phase); r.step(); }
      }
      // The operand, in the order of the MMA's registers: (hi, lo) of columns 2t, 2t + 1 and of those eight further on.  With a norm ahead its
      // sums of squares come in the same polls: unit and row by thread.  The first layer's is the embedding, whoever needs it reads it.
      uint4 a[kSlabs * 4];
      auto gather = [&](auto sl) {
        constexpr int SL = decltype(sl)::value;
        float ss = 0.f;
        if (ph == kQkv && sp.l == 0) {
          const __nv_bfloat16 *e = (const __nv_bfloat16*)P.embed + (size_t)s_tok[g] * d, *gp = (const __nv_bfloat16*)sp.gain;
#pragma unroll
          for (int i = 0; i < SL * 4; ++i) {
            const int k = (((i >> 2) * 8 + warp) * 4 + (i & 3)) * 16 + 2 * t;
            a[i] = make_uint4(0, 0, 0, 0);
            if (mine && k < K) {
              const __nv_bfloat162 e0 = *reinterpret_cast<const __nv_bfloat162*>(e + k), e1 = *reinterpret_cast<const __nv_bfloat162*>(e + k + 8);
              const float x[4] = {__low2float(e0), __high2float(e0), __low2float(e1), __high2float(e1)};
              const uint2 w0 = operand_words(x[0] * to_f32(gp[k]), x[1] * to_f32(gp[k + 1])), w1 = operand_words(x[2] * to_f32(gp[k + 8]), x[3] * to_f32(gp[k + 9]));
              a[i] = make_uint4(w0.x, w0.y, w1.x, w1.y);
              ss += (x[0] * x[0] + x[1] * x[1]) + (x[2] * x[2] + x[3] * x[3]);
            }
          }
          ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 1);
          ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 2);
          if (t == 0) s_ssq[g][warp] = ss;
          return;
        }
        uint32_t need = 0, q[SL];
        const bool row_on = normed && ((active >> (threadIdx.x & 7)) & 1u) != 0;
#pragma unroll
        for (int i = 0; i < SL * 4; ++i) {
          a[i] = make_uint4(0, 0, 0, 0);
          if (mine && ((i >> 2) * 8 + warp) * 64 < K) need |= 1u << i;
        }
#pragma unroll
        for (int i = 0; i < SL; ++i) {
          q[i] = 0u;
          if (row_on && i * 32 + (int)(threadIdx.x >> 3) < d / 16) need |= 1u << (SL * 4 + i);
        }
        const uint32_t* at = in + (ph == kWo ? (warp * 2 * kRows + g) * 32 + t * 4 : ph == kDown ? warp * 512 + lane * 2 : (warp * 4 * 32 + lane) * 4);
        const uint32_t* at_q = in + d * kRows + (threadIdx.x >> 3) * 32 + (threadIdx.x & 7);
        const int odd = ph == kWo ? 16 : 128;  // words between the two units of 32 columns
        for (uint32_t polls = 0; !wait.dead; ++polls) {
#pragma unroll
          for (int i = 0; i < SL * 4; ++i) {
            const uint32_t* p = at + (i >> 2) * 4096 + ((i & 3) >> 1) * 256 + (i & 1) * odd;
            if (ph == kDown) {
              uint2 lo = make_uint2(a[i].x, a[i].y), hi = make_uint2(a[i].z, a[i].w);
              ld2_if((need >> i) & 1u, lo, p);
              ld2_if((need >> i) & 1u, hi, p + 64);
              a[i] = make_uint4(lo.x, lo.y, hi.x, hi.y);
            } else {
              ld4_if((need >> i) & 1u, a[i], p);
            }
          }
#pragma unroll
          for (int i = 0; i < SL; ++i) ld1_if((need >> (SL * 4 + i)) & 1u, q[i], at_q + i * 32 * 32);
#pragma unroll
          for (int i = 0; i < SL * 4; ++i)
            if (full(a[i])) need &= ~(1u << i);
#pragma unroll
          for (int i = 0; i < SL; ++i)
            if (full(q[i])) need &= ~(1u << (SL * 4 + i));
          if (!__any_sync(0xFFFFFFFFu, need != 0)) break;
          wait.give_up(polls);
          wait.dead = __any_sync(0xFFFFFFFFu, wait.dead);
        }
        if (normed) {
#pragma unroll
          for (int i = 0; i < SL; ++i) ss += __uint_as_float(q[i]);
          ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 8);
          ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 16);
          if (lane < kRows) s_ssq[lane][warp] = ss;
        }
      };
      if (extras && ahead < n_units) fill_extra(ahead);
      switch (slabs) {
        case 1: gather(std::integral_constant<int, 1>()); break;
        case 2: gather(std::integral_constant<int, 2>()); break;
        case 3: gather(std::integral_constant<int, 3>()); break;
        default: gather(std::integral_constant<int, 4>()); break;
      }
      const uint32_t row = lane & 7, mat = lane >> 3, lane_off = warp * 1024 + row * 128;
      const uint32_t c0 = (mat ^ row) * 16, c1 = ((4 + mat) ^ row) * 16, ring0 = smem_u32(smem) + lane_off;
      int ul = 0;
      for (int u = sp.u0; u < n_units; u += grid, ++ul, ++turn) {
        float acc[2][2][4];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[r][h][i] = 0.f;
#pragma unroll
        for (int s = 0; s < kSlabs; ++s) {
          if (s >= slabs) break;
          if (ul > 0) wait_stage(ring.s, ring.phase);
          if ((s * 8 + warp) * 64 < K) {
            const uint32_t at = ring0 + ring.s * kStage;
            uint32_t b[2][2][4];
#pragma unroll
            for (int r = 0; r < 2; ++r) { ldmatrix4(at + r * (kStage / 2) + c0, b[r][0]); ldmatrix4(at + r * (kStage / 2) + c1, b[r][1]); }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) mma_bf16(acc[r][h], a[s * 4 + h * 2 + j], b[r][h][2 * j], b[r][h][2 * j + 1]);
          }
          ring.step();
        }
        float(*rb)[2][kRows][8] = red[turn & 1];
#pragma unroll
        for (int r = 0; r < 2; ++r)
          *reinterpret_cast<float2*>(&rb[warp][r][g][2 * t]) = make_float2((acc[r][0][0] + acc[r][1][0]) + (acc[r][0][2] + acc[r][1][2]),
                                                                          (acc[r][0][1] + acc[r][1][1]) + (acc[r][0][3] + acc[r][1][3]));
        if (ph == kQkv) asm volatile("cp.async.wait_all;" ::: "memory");     // the angles
        if (sync_or(wait.dead)) { wait.dead = true; return false; }
        behind_unit(slabs);
        if (warp == (turn & (kWarps - 1))) {
          float2 p0[kWarps], p1[kWarps];
#pragma unroll
          for (int w = 0; w < kWarps; ++w) {
            p0[w] = *reinterpret_cast<const float2*>(&rb[w][0][g][2 * t]);
            p1[w] = *reinterpret_cast<const float2*>(&rb[w][1][g][2 * t]);
          }
#pragma unroll
          for (int n = kWarps / 2; n > 0; n /= 2)
#pragma unroll
            for (int w = 0; w < n; ++w) { p0[w].x += p0[w + n].x; p0[w].y += p0[w + n].y; p1[w].x += p1[w + n].x; p1[w].y += p1[w + n].y; }
          const float v0[NC] = {p0[0].x, p0[0].y}, v1[NC] = {p1[0].x, p1[0].y};
          if (ph == kWo || ph == kDown) {
            residual(set + sp.dst, u, ul, g, mine, extra, v0, v1);
          } else if (mine) {
            epilogue(sp, u, g, 2 * t, v0, v1);
          }
          if (extras && u + kWarps * grid < n_units) fill_extra(u + kWarps * grid);
        }
      }
      return true;
    }
  };

  // ---- attention ----
  __shared__ float s_m[kWarps][8], s_l[kWarps][8];
  __shared__ __align__(16) float s_f32[F32 ? 3 : 1][64];                     // fp32: query, new key, new value
  __shared__ __align__(16) __half s_q[F32 ? 1 : (EXT ? 2 : 1)][8][128 + 32], s_new[F32 ? 1 : (EXT ? 4 : 2)][128];
  auto attention_f32 = [&](const Step& sp) -> bool {
    constexpr int HD = 64, NK = HD / 8, DPL = HD / 32, NV = DPL * 4;
    const int G = P.H / P.KV;
    float* pool = reinterpret_cast<float*>(sp.kv);
    const size_t block = (size_t)P.KV * kPageTokens * HD;
    const float scale = rsqrtf((float)HD);
    for (int unit = sp.u0; unit < sp.n_units; unit += grid) {
      const int m = unit / P.H, h = unit % P.H, kvh = h / G;
      if (!((active >> m) & 1u)) continue;
      const int pos = s_pos[m], n_pages = pos / kPageTokens + 1;
      const int32_t* pt = P.page_table + (size_t)s_row[m] * P.max_pages;
      const int tok = lane & 15, hf = lane >> 4;
      // keys: this lane's token and half of the dims; values: its dims, all tokens
      uint4 kr[NK], vr[NV];
      auto fetch = [&](int page) {
        const float* kb = pool + (size_t)page * 2 * block + (size_t)kvh * kPageTokens * HD + tok * HD + hf * (HD / 2);
        const float* vb = pool + (size_t)page * 2 * block + block + (size_t)kvh * kPageTokens * HD + lane * DPL * kPageTokens;
#pragma unroll
        for (int i = 0; i < NK; ++i) kr[i] = __ldcg(reinterpret_cast<const uint4*>(kb + i * 4));
#pragma unroll
        for (int i = 0; i < NV; ++i) vr[i] = __ldcg(reinterpret_cast<const uint4*>(vb + i * 4));
      };
      if (warp < n_pages) fetch(pt[warp]);
      int next = warp + kWarps < n_pages ? pt[warp + kWarps] : 0;
      const int new_page = pt[n_pages - 1];
      // query, key and value of the new token: HD words each
      uint4 w[1] = {make_uint4(0, 0, 0, 0)};
      constexpr int VPH = HD / 4;              // vectors of a head: dims 8 j + 2 tt, + 1 and those that they turn with
      const int part = threadIdx.x / VPH, j = (threadIdx.x % VPH) / 4, tt = threadIdx.x & 3;
      poll<1>(w, part < 3 ? 1u : 0u, wait, [&](bool on, uint4& x, int) {
        const int head = part == 0 ? h : P.H + (part - 1) * P.KV + kvh;
        ld4_if(on, x, set + sp.src + ((head * (HD / 16) + j) * 32 + m * 4 + tt) * 4);
      });
      if (part < 3) {
        const uint32_t e[4] = {w[0].x, w[0].y, w[0].z, w[0].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int dim = 8 * j + 2 * tt + (i & 1) + (i >> 1) * (HD / 2), slot = pos % kPageTokens;
          const float v = __uint_as_float(e[i]);
          s_f32[F32 ? part : 0][dim] = part == 0 ? v * scale : v;
          if (part > 0 && h % G == 0)
            pool[(size_t)new_page * 2 * block + (part == 1 ? ((size_t)kvh * kPageTokens + slot) * HD + dim : block + ((size_t)kvh * HD + dim) * kPageTokens + slot)] = v;
        }
      }
      if (sync_or(wait.dead)) { wait.dead = true; return false; }
      float mx_run = -INFINITY, l_run = 0.f, o[DPL] = {};
      for (int pg = warp; pg < n_pages; pg += kWarps) {
        const int n = min(kPageTokens, pos + 1 - pg * kPageTokens);
        const bool has_new = pg == n_pages - 1;
        if (pg != warp) {
          fetch(next);
          if (pg + kWarps < n_pages) next = pt[pg + kWarps];
        }
        if (has_new && tok == n - 1) {
#pragma unroll
          for (int i = 0; i < NK; ++i) kr[i] = *reinterpret_cast<const uint4*>(&s_f32[F32 ? 1 : 0][hf * (HD / 2) + i * 4]);
        }
        if (has_new) {                         // slots beyond the context hold anything, NaN included; their weights are zero
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            uint32_t* e = reinterpret_cast<uint32_t*>(&vr[i]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int tk = (i & 3) * 4 + j;
              if (tk >= n) e[j] = 0u;
              if (tk == n - 1) e[j] = __float_as_uint(s_f32[F32 ? 2 : 0][lane * DPL + i / 4]);
            }
          }
        }
        float p4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < NK; ++i) {
          const float4 q4 = *reinterpret_cast<const float4*>(&s_f32[0][hf * (HD / 2) + i * 4]);
          p4[0] = fmaf(q4.x, __uint_as_float(kr[i].x), p4[0]); p4[1] = fmaf(q4.y, __uint_as_float(kr[i].y), p4[1]);
          p4[2] = fmaf(q4.z, __uint_as_float(kr[i].z), p4[2]); p4[3] = fmaf(q4.w, __uint_as_float(kr[i].w), p4[3]);
        }
        float sc = (p4[0] + p4[1]) + (p4[2] + p4[3]);
        sc += __shfl_xor_sync(0xFFFFFFFFu, sc, 16);
        if (tok >= n) sc = -INFINITY;
        float mx = sc;
#pragma unroll
        for (int x = 1; x < 16; x <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, x));
        mx = fmaxf(mx_run, mx);                // finite: token 0 of a walked page is always valid
        const float corr = __expf(mx_run - mx), pr = __expf(sc - mx);
        l_run = l_run * corr + (hf == 0 ? pr : 0.f);
#pragma unroll
        for (int i = 0; i < DPL; ++i) o[i] *= corr;
#pragma unroll
        for (int j = 0; j < kPageTokens; ++j) {
          const float pj = __shfl_sync(0xFFFFFFFFu, pr, j);
#pragma unroll
          for (int i = 0; i < DPL; ++i) o[i] = fmaf(pj, __uint_as_float(reinterpret_cast<const uint32_t*>(&vr[i * 4 + j / 4])[j % 4]), o[i]);
        }
        mx_run = mx;
      }
      l_run = warp_sum(l_run);
      if (lane == 0) { s_m[warp][0] = mx_run; s_l[warp][0] = l_run; }
      float* s_o = reinterpret_cast<float*>(buffer);             // [8][HD]: the operand rows are not in use here
#pragma unroll
      for (int i = 0; i < DPL; ++i) s_o[warp * HD + lane * DPL + i] = o[i];
      (void)sync_or(false);
      if (threadIdx.x < HD) {
        float M = s_m[0][0], L = 0.f, O = 0.f;
#pragma unroll
        for (int x = 1; x < kWarps; ++x) M = fmaxf(M, s_m[x][0]);
#pragma unroll
        for (int x = 0; x < kWarps; ++x) {
          const float e = __expf(s_m[x][0] - M);                 // 0 for a warp without pages
          L += s_l[x][0] * e;
          O += s_o[x * HD + threadIdx.x] * e;
        }
        st_word(set + sp.dst + m * hq + h * HD + threadIdx.x, word_of(O / L));
      }
      (void)sync_or(false);                    // before the next pair, or operand, takes the buffers
    }
    return true;
  };

  auto attention_bf16 = [&](const Step& sp) -> bool {
    constexpr int HD = 128, KB = HD / 32, NT = HD / 8, kBlockElems = kPageTokens * HD, kParts = EXT ? 4 : 2, kBufs = Cfg::kBufs;
    const int KV = P.KV, G = P.H / KV;
    __half* pool = reinterpret_cast<__half*>(sp.kv);
    const size_t page_elems = (size_t)kParts * KV * kBlockElems;
    const float scale = rsqrtf((float)HD);
    __half* const ring_w = reinterpret_cast<__half*>(buffer) + (size_t)warp * kBufs * kParts * kBlockElems;
    for (int unit = sp.u0; unit < sp.n_units; unit += grid) {
      const int m = unit / KV, kvh = unit % KV, h0 = kvh * G;
      if (unit != sp.u0) (void)sync_or(false); // the pair before this one is merged
      if (!((active >> m) & 1u)) continue;
      const int pos = s_pos[m], ctx = pos + 1, n_pages = (ctx + kPageTokens - 1) / kPageTokens;
      const int32_t* pt = P.page_table + (size_t)s_row[m] * P.max_pages;
      // keys of token t: chunk c of its row at c ^ 4 (t & 1) (attn_decode.cu)
      auto fetch = [&](int page, int buf) {
        __half* pg_buf = ring_w + (size_t)buf * kParts * kBlockElems;
        const __half* src = pool + (size_t)page * page_elems + (size_t)kvh * kBlockElems + lane * 8;
        constexpr int kChunks = kBlockElems / 8, kRow = HD / 8;
#pragma unroll
        for (int part = 0; part < kParts; ++part)
#pragma unroll
          for (int i = 0; i < kChunks / 32; ++i) {
            const int c = i * 32 + lane, dd = (part & 1) ? c : (c ^ (((c / kRow) & 1) << 2));
            cp_async16(pg_buf + part * kBlockElems + dd * 8, src + (size_t)part * KV * kBlockElems + i * 256);
          }
      };
#pragma unroll
      for (int b = 0; b < kBufs; ++b) {
        if (warp + b * kWarps < n_pages) fetch(pt[warp + b * kWarps], b);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      const int new_page = (ctx - 1) / kPageTokens, new_slot = (ctx - 1) % kPageTokens;
      const int new_id = pt[new_page];
      for (int idx = threadIdx.x; idx < (8 - G) * (HD / 8); idx += kWorkers) {    // the tile's rows beyond the group
        const uint4 z = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(&s_q[0][G + idx / (HD / 8)][(idx % (HD / 8)) * 8]) = z;
        if (EXT) *reinterpret_cast<uint4*>(&s_q[EXT ? 1 : 0][G + idx / (HD / 8)][(idx % (HD / 8)) * 8]) = z;
      }
      // queries of the group, new key and value: 32 vectors a head, dims 8 j + 2 tt, + 1 and those that they turn with
      uint4 w[2];
      uint32_t need = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        w[i] = make_uint4(0, 0, 0, 0);
        if (warp + i * kWarps < G + 2) need |= 1u << i;
      }
      const int dd = 8 * (lane >> 2) + 2 * t;
      poll<2>(w, need, wait, [&](bool on, uint4& x, int i) {
        const int hh = warp + i * kWarps, head = hh < G ? h0 + hh : P.H + (hh - G) * KV + kvh;
        ld4_if(on, x, set + sp.src + ((head * 8 + (lane >> 2)) * 32 + m * 4 + t) * 4);
      });
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int hh = warp + i * kWarps;
        if (hh >= G + 2) continue;
        const float v[4] = {__uint_as_float(w[i].x), __uint_as_float(w[i].y), __uint_as_float(w[i].z), __uint_as_float(w[i].w)};
        uint32_t hi[2], lo[2];
        pack_h2_split(v[0], v[1], hi[0], lo[0]);
        pack_h2_split(v[2], v[3], hi[1], lo[1]);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int dim = dd + x * (HD / 2);
          if (hh < G) {
            *reinterpret_cast<uint32_t*>(&s_q[0][hh][dim]) = hi[x];
            if (EXT) *reinterpret_cast<uint32_t*>(&s_q[EXT ? 1 : 0][hh][dim]) = lo[x];
          } else {
            const int part = hh - G;
            *reinterpret_cast<uint32_t*>(&s_new[F32 ? 0 : part][dim]) = hi[x];
            if (EXT) *reinterpret_cast<uint32_t*>(&s_new[EXT ? part + 2 : 0][dim]) = lo[x];
            __half* blk = pool + (size_t)new_id * page_elems + (size_t)part * KV * kBlockElems + (size_t)kvh * kBlockElems;
#pragma unroll
            for (int e = 0; e < (EXT ? 2 : 1); ++e) {
              const uint32_t word = e == 0 ? hi[x] : lo[x];
              __half* at = blk + (size_t)e * 2 * KV * kBlockElems;
              if (part == 0) {
                *reinterpret_cast<uint32_t*>(at + new_slot * HD + dim) = word;
              } else {
                at[dim * kPageTokens + new_slot] = __ushort_as_half((unsigned short)(word & 0xFFFFu));
                at[(dim + 1) * kPageTokens + new_slot] = __ushort_as_half((unsigned short)(word >> 16));
              }
            }
          }
        }
      }
      if (sync_or(wait.dead)) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        wait.dead = true;
        return false;
      }
      __align__(16) uint32_t qa[KB][2][2], ql[EXT ? KB : 1][2][2];
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        *reinterpret_cast<uint4*>(qa[j]) = *reinterpret_cast<const uint4*>(&s_q[0][g][32 * j + 8 * t]);
        if (EXT) *reinterpret_cast<uint4*>(ql[EXT ? j : 0]) = *reinterpret_cast<const uint4*>(&s_q[EXT ? 1 : 0][g][32 * j + 8 * t]);
      }
      float o[NT][2];
#pragma unroll
      for (int i = 0; i < NT; ++i) o[i][0] = o[i][1] = 0.f;
      float m_run = -INFINITY, l_run = 0.f;
      const int tok0 = 4 * (g >> 1) + (g & 1), tok1 = tok0 + 2, key_off = (t ^ ((g & 1) << 2)) * 8;
      int buf = 0;
#pragma unroll 1
      for (int p = warp; p < n_pages; p += kWarps) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kBufs - 1) : "memory");
        __syncwarp();
        __half *kb = ring_w + (size_t)buf * kParts * kBlockElems, *vb = kb + kBlockElems;
        if (p == new_page) {                   // the page was fetched before its last token was known
#pragma unroll
          for (int part = 0; part < kParts; part += 2) {
            if (lane < HD / 8)
              *reinterpret_cast<uint4*>(kb + part * kBlockElems + new_slot * HD + (lane ^ ((new_slot & 1) << 2)) * 8) = *reinterpret_cast<const uint4*>(&s_new[F32 ? 0 : part][lane * 8]);
#pragma unroll
            for (int i = 0; i < HD / 32; ++i)
              vb[part * kBlockElems + (i * 32 + lane) * kPageTokens + new_slot] = s_new[F32 ? 0 : part + 1][i * 32 + lane];
          }
          __syncwarp();
        }
        float s0[2] = {0.f, 0.f}, s1[2] = {0.f, 0.f};
#pragma unroll
        for (int j = 0; j < KB; ++j) {
          const int off = (32 * j) ^ key_off;
          const uint4 k0 = *reinterpret_cast<const uint4*>(kb + tok0 * HD + off), k1 = *reinterpret_cast<const uint4*>(kb + tok1 * HD + off);
          mma_f16_top(s0[0], s0[1], qa[j][0][0], qa[j][0][1], k0.x, k0.y);
          mma_f16_top(s0[0], s0[1], qa[j][1][0], qa[j][1][1], k0.z, k0.w);
          mma_f16_top(s1[0], s1[1], qa[j][0][0], qa[j][0][1], k1.x, k1.y);
          mma_f16_top(s1[0], s1[1], qa[j][1][0], qa[j][1][1], k1.z, k1.w);
          if (EXT) {
            const uint4 e0 = *reinterpret_cast<const uint4*>(kb + 2 * kBlockElems + tok0 * HD + off), e1 = *reinterpret_cast<const uint4*>(kb + 2 * kBlockElems + tok1 * HD + off);
            mma_f16_top(s0[0], s0[1], qa[j][0][0], qa[j][0][1], e0.x, e0.y);
            mma_f16_top(s0[0], s0[1], qa[j][1][0], qa[j][1][1], e0.z, e0.w);
            mma_f16_top(s1[0], s1[1], qa[j][0][0], qa[j][0][1], e1.x, e1.y);
            mma_f16_top(s1[0], s1[1], qa[j][1][0], qa[j][1][1], e1.z, e1.w);
            mma_f16_top(s0[0], s0[1], ql[EXT ? j : 0][0][0], ql[EXT ? j : 0][0][1], k0.x, k0.y);
            mma_f16_top(s0[0], s0[1], ql[EXT ? j : 0][1][0], ql[EXT ? j : 0][1][1], k0.z, k0.w);
            mma_f16_top(s1[0], s1[1], ql[EXT ? j : 0][0][0], ql[EXT ? j : 0][0][1], k1.x, k1.y);
            mma_f16_top(s1[0], s1[1], ql[EXT ? j : 0][1][0], ql[EXT ? j : 0][1][1], k1.z, k1.w);
          }
        }
        const int n_valid = min(kPageTokens, ctx - p * kPageTokens);
        float sc[4] = {s0[0] * scale, s0[1] * scale, s1[0] * scale, s1[1] * scale};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * t + e >= n_valid) sc[e] = -INFINITY;
        float mx = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
        const float m_new = fmaxf(m_run, mx), corr = __expf(m_run - m_new);
        float pr[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) pr[e] = __expf(sc[e] - m_new);
        l_run = l_run * corr + (pr[0] + pr[1] + pr[2] + pr[3]);
        m_run = m_new;
        uint32_t pa0, pa2, pl0 = 0u, pl2 = 0u;
        if (EXT) { pack_h2_split(pr[0], pr[1], pa0, pl0); pack_h2_split(pr[2], pr[3], pa2, pl2); }
        else { pa0 = pack_h2(pr[0], pr[1]); pa2 = pack_h2(pr[2], pr[3]); }
        uint32_t mlo = 0xFFFFFFFFu, mhi = 0xFFFFFFFFu;      // the halves of a value fragment that belong to cached tokens
        if (n_valid < kPageTokens) {
          mlo = (4 * t < n_valid ? 0x0000FFFFu : 0u) | (4 * t + 1 < n_valid ? 0xFFFF0000u : 0u);
          mhi = (4 * t + 2 < n_valid ? 0x0000FFFFu : 0u) | (4 * t + 3 < n_valid ? 0xFFFF0000u : 0u);
        }
#pragma unroll
        for (int i = 0; i < NT; ++i) {
          const uint2 vv = *reinterpret_cast<const uint2*>(vb + (8 * i + g) * kPageTokens + 4 * t);
          o[i][0] *= corr; o[i][1] *= corr;
          mma_f16_top(o[i][0], o[i][1], pa0, pa2, vv.x & mlo, vv.y & mhi);
          if (EXT) {
            const uint2 vl = *reinterpret_cast<const uint2*>(vb + 2 * kBlockElems + (8 * i + g) * kPageTokens + 4 * t);
            mma_f16_top(o[i][0], o[i][1], pl0, pl2, vv.x & mlo, vv.y & mhi);
            mma_f16_top(o[i][0], o[i][1], pa0, pa2, vl.x & mlo, vl.y & mhi);
          }
        }
        __syncwarp();                          // every lane has read the buffer
        if (p + kBufs * kWarps < n_pages) fetch(pt[p + kBufs * kWarps], buf);
        asm volatile("cp.async.commit_group;" ::: "memory");
        buf = buf + 1 == kBufs ? 0 : buf + 1;
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      // the warp's outputs take the place of its pages
      auto s_o = [&](int w) { return reinterpret_cast<float(*)[HD + 8]>(buffer + (size_t)w * kBufs * Cfg::kPageBytes); };
      l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 1);
      l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 2);
      if (t == 0) { s_m[warp][g] = m_run; s_l[warp][g] = l_run; }
#pragma unroll
      for (int i = 0; i < NT; ++i) *reinterpret_cast<float2*>(&s_o(warp)[g][8 * i + 2 * t]) = make_float2(o[i][0], o[i][1]);
      (void)sync_or(false);
      // two neighbouring outputs a thread: HD / 2 threads a head
#pragma unroll 1
      for (int idx = threadIdx.x; idx < G * (HD / 2); idx += kWorkers) {
        const int gg = idx / (HD / 2), dd = 2 * (idx % (HD / 2));
        float M = s_m[0][gg];
#pragma unroll
        for (int x = 1; x < kWarps; ++x) M = fmaxf(M, s_m[x][gg]);
        float L = 0.f, O[2] = {0.f, 0.f};
#pragma unroll
        for (int x = 0; x < kWarps; ++x) {
          const float e = __expf(s_m[x][gg] - M);                 // 0 for a warp without pages
          const float2 v = *reinterpret_cast<const float2*>(&s_o(x)[gg][dd]);
          L += s_l[x][gg] * e;
          O[0] += v.x * e; O[1] += v.y * e;
        }
        const float inv = 1.f / L;
        st_word(set + sp.dst + attn_word((h0 + gg) * HD + dd, m), operand_words(O[0] * inv, O[1] * inv));
      }
    }
    return true;
  };

  for (int round = 0;; ++round) {
    const bool failed = threadIdx.x == 0 && ld_cg(P.err) != 0;       // raised elsewhere: the phase ends with this iteration
    // the embedding, into the residual stream (fp32: and to those who multiply it)
    {
      int ul = 0;
      for (int u = ((int)blockIdx.x - (n_qkv / 16) % grid + grid) % grid; u < d / 16; u += grid, ++ul) {
        if (warp == kWarps - 1) {
          const bool on = ((active >> g) & 1u) != 0;
          const size_t at = (size_t)s_tok[g] * d + u * 16 + 2 * t;
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (on) {
            if (F32) { const float* e = (const float*)P.embed + at; x = make_float4(e[0], e[1], e[8], e[9]); }
            else { const __nv_bfloat16* e = (const __nv_bfloat16*)P.embed + at; x = make_float4(to_f32(e[0]), to_f32(e[1]), to_f32(e[8]), to_f32(e[9])); }
          }
          own[ul][lane] = x;
          if (F32 && on) st_word(set + P.at_x + (u * 32 + lane) * 4, make_uint4(word_of(x.x), word_of(x.y), word_of(x.z), word_of(x.w)));
        }
      }
    }
    if (s_steps[0].ph == kQkv) {
      // (read behind a barrier of the qkv product, ahead of which every thread waits for its copies)
      for (int i = threadIdx.x; i < n_slots * (hd / 2); i += kWorkers) {
        const int m = i / (hd / 2), dim = i % (hd / 2);
        if ((active >> m) & 1u)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(&s_rope[m][dim])), "l"(P.rope + (size_t)s_pos[m] * (hd / 2) + dim) : "memory");
      }
    }
    best_score = -INFINITY;
    best_id = 0x7FFFFFFF;
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i < n_steps && ok; ++i) {
      const Step& sp = s_steps[i];
      if (sp.ph == kAttn) {
        if constexpr (F32) ok = attention_f32(sp);
        else ok = attention_bf16(sp);
      } else {
        ok = product(sp);
      }
      // (behind the first step: whoever waits for it does not wait for this)
      if (i == 0 && ok && round > 0) empty_slots(round);
    }
    if (!ok) break;
    // this CTA's best id of every row, to all CTAs
    unsigned long long mine = best_id == 0x7FFFFFFF ? 0ull : (((unsigned long long)score_key(best_score) << 32) | (uint32_t)(0xFFFFFFFFu - (uint32_t)best_id));
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {            // the four lanes of a row
      const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, mine, o);
      mine = v > mine ? v : mine;
    }
    if (t == 0) s_best[warp][g] = mine;
    if (sync_or(wait.dead || failed)) break;
    uint32_t* ids = P.slots + P.at_s + (round & 3) * 160 * 32;
    if (warp == 0) {
      unsigned long long top = s_best[2 * t][g], v = s_best[2 * t + 1][g];
      top = v > top ? v : top;
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        v = __shfl_xor_sync(0xFFFFFFFFu, top, o);
        top = v > top ? v : top;
      }
      // what this CTA has written in this iteration is there for everybody who reads an id of it
      fence_gpu();
      // (score, id + 1): neither is ever kEmpty, a score with those bits would be a NaN
      if (t == 0 && ((active >> g) & 1u))
        st_word(ids + blockIdx.x * 32 + g * 2, top == 0ull ? make_uint2(0u, 0u) : make_uint2((uint32_t)(top >> 32), 0xFFFFFFFFu - (uint32_t)top + 1u));
    }
    {
      // rows 2t, 2t + 1 of eight CTAs a vector
      constexpr int NP = 3;                      // 192 CTAs
      const unsigned two = (active >> (2 * t)) & 3u;
      uint4 v[NP];
      uint32_t need = 0;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (two != 0 && i * 64 + warp * 8 + g < grid) need |= 1u << i;
      }
      poll<NP>(v, need, wait, [&](bool on, uint4& x, int i) {
        ld4_if(on, x, ids + (i * 64 + warp * 8 + g) * 32 + t * 4);
        if (!(two & 1u)) x.x = x.y = 0u;         // rows that have ended publish nothing
        if (!(two & 2u)) x.z = x.w = 0u;
      });
      fence_gpu();                               // and what the others had written ahead of their ids is seen from here on
      unsigned long long top[2] = {0ull, 0ull};
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const unsigned long long a = v[i].y == 0u ? 0ull : (((unsigned long long)v[i].x << 32) | (uint32_t)(0xFFFFFFFFu - (v[i].y - 1u)));
        const unsigned long long b = v[i].w == 0u ? 0ull : (((unsigned long long)v[i].z << 32) | (uint32_t)(0xFFFFFFFFu - (v[i].w - 1u)));
        top[0] = a > top[0] ? a : top[0];
        top[1] = b > top[1] ? b : top[1];
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const unsigned long long c = __shfl_xor_sync(0xFFFFFFFFu, top[r], o);
          top[r] = c > top[r] ? c : top[r];
        }
      if (g == 0) { s_top[warp][2 * t] = top[0]; s_top[warp][2 * t + 1] = top[1]; }
    }
    if (sync_or(wait.dead)) break;
    const int m = warp;                          // a row per warp
    const bool live = ((active >> m) & 1u) != 0;
    int sampled = 0;
    {
      unsigned long long top = lane < kWarps ? s_top[lane][m] : 0ull;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const unsigned long long c = __shfl_xor_sync(0xFFFFFFFFu, top, o);
        top = c > top ? c : top;
      }
      if (lane == 0) {
        // decode_update_kernel's work for this row, in every CTA alike; one of them keeps the books (below)
        bool ends = true;
        if (live) {
          sampled = top ? (int)(0xFFFFFFFFu - (uint32_t)(top & 0xFFFFFFFFull)) : 0;
          const int flen = s_flen[m];
          const int tk = flen > 0 ? st.forced_tok[phase][(size_t)s_row[m] * st.C + iter] : sampled;
          ends = ends_step(tk, lp) || iter + 1 == st.C || (flen > 0 && iter + 1 == flen);
          s_tok[m] = tk;
          s_pos[m] += 1;
        }
        s_on[m] = ends ? 0 : 1;
      }
    }
    if (sync_or(wait.dead)) break;
    unsigned left = 0;
#pragma unroll
    for (int i = 0; i < kRows; ++i) left |= (s_on[i] != 0 ? 1u : 0u) << i;
    if (blockIdx.x == gridDim.x - 1 && lane == 0) {
      if (live) {
        const int row = s_row[m], pos = s_pos[m], tk = s_tok[m];       // pos: the new token's
        st.sampled[phase][(size_t)row * st.C + iter] = sampled;
        st.tok[(size_t)row * st.S + pos] = tk;
        st.gen_tok[phase][(size_t)row * st.C + iter] = tk;
        st.kv_len[which][row] = pos;
        st.gen_len[phase][row] = iter + 1;
        if (!((left >> m) & 1u)) { st.gen_active[row] = 0; st.pass_tok_row[m] = -1; }
        else { st.pass_tok_id[m] = tk; st.pass_tok_pos[m] = pos; }
      }
      if (warp == 0 && left == 0) {
        st.n_active[0] = 0;
        st.iter[0] = iter + 1;
        const unsigned long long failed = ld_cg(st.wait_err) != 0 || ld_cg(st.err) != 0;
        *(volatile unsigned long long*)st.progress = (failed << 63) | ((unsigned long long)(iter + 2) << 32);
      }
    }
    ++iter;
    active = left;
    if (left == 0) break;
    set = P.slots + ((round & 1) ? 0u : P.set_words);
  }
  // copies in flight land before the CTA goes away (after an expired wait this looks at stages that have landed, too)
  if (sync_or(false)) return;
  if (threadIdx.x == 0) {
    const int issued = s_feed[3];
    for (int i = max(0, issued - Cfg::kStages); i < issued; ++i)
      for (uint32_t k = 0; k < (1u << 16); ++k)
        if (mbar_try_wait(&bar_full[i % Cfg::kStages], (uint32_t)(i / Cfg::kStages) & 1u)) break;
  }
}

int device_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return n;
}

template <typename F> void driver_entry(F& fn, const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  fn = cudaGetDriverEntryPoint(name, &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess ? (F)p : nullptr;
  (void)cudaGetLastError();
}

// SMs that launches into `s` may come to: the device's, or those of the part of it that the stream's green context, or the current context, has.
int stream_sms(cudaStream_t s) {
  struct Driver {
    decltype(&cuStreamGetGreenCtx) green_of;
    decltype(&cuGreenCtxGetDevResource) of_green;
    decltype(&cuCtxGetCurrent) current;
    decltype(&cuCtxGetDevResource) of_ctx;
    Driver() {
      driver_entry(green_of, "cuStreamGetGreenCtx");
      driver_entry(of_green, "cuGreenCtxGetDevResource");
      driver_entry(current, "cuCtxGetCurrent");
      driver_entry(of_ctx, "cuCtxGetDevResource");
    }
  };
  static const Driver drv;
  int n = device_sms();
  CUdevResource r{};
  CUgreenCtx green = nullptr;
  CUcontext ctx = nullptr;
  const bool named = s != nullptr && s != cudaStreamLegacy && s != cudaStreamPerThread;
  if (named && drv.green_of && drv.of_green && drv.green_of((CUstream)s, &green) == CUDA_SUCCESS && green != nullptr) {
    if (drv.of_green(green, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS) n = std::min(n, (int)r.sm.smCount);
  } else if (drv.current && drv.of_ctx && drv.current(&ctx) == CUDA_SUCCESS && ctx != nullptr) {
    if (drv.of_ctx(ctx, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS) n = std::min(n, (int)r.sm.smCount);
  }
  return n;
}

int grid_of(const ResidentShape& m, int sms) { return std::min(std::min(sms, m.F / 8), 160); }

struct Words { uint32_t x, y, q, a, f, s, set, all; };
Words words_of(const ResidentShape& m) {
  const uint32_t xw = (uint32_t)(m.d * kRows + m.d / 16 * 32), L = (uint32_t)m.n_layers;
  Words w;
  w.x = 0;
  w.y = w.x + (L + 1) * xw;
  w.q = w.y + L * xw;
  w.a = w.q + L * kRows * (uint32_t)((m.H + 2 * m.KV) * m.hd);
  w.f = w.a + L * kRows * (uint32_t)(m.H * m.hd);
  w.s = w.f + L * kRows * (uint32_t)m.F;
  w.set = (w.s + 63) & ~63u;
  w.s = 2 * w.set;                             // the ids lie behind both sets, four places of them
  w.all = w.s + 4 * 160 * 32;
  return w;
}

}  // namespace

bool resident_supported(const ResidentShape& m) {
  const int hq = m.H * m.hd;
  if (m.n_layers < 1 || 5 * m.n_layers + 1 > kMaxSteps || m.H % m.KV != 0 || m.d > kMaxK || hq > kMaxK || m.F > kMaxK || m.d < 16 || m.F < 8) return false;
  if (m.d % 16 != 0 || m.F % 8 != 0 || (m.d / 16 + grid_of(m, 148) - 1) / grid_of(m, 148) > kOwn) return false;
  if ((size_t)words_of(m).all * 4 > ((size_t)64 << 20)) return false;
  if (m.f32) return m.hd == 64;
  return m.hd == 128 && m.H / m.KV <= 8 && m.d % 64 == 0 && m.F % 64 == 0;
}

// Where the one launch is faster than graphs of the single kernels (kernels / here, us an iteration, two to 24 layers; each line where it stops):
//   split       the grid is d_ffn / 8 CTAs at most.  With fewer than 80, fewer than columns / 8 (bf16: or than 148), more qkv units than CTAs or more pairs of the attention the
//               CTAs take turns, while kernels choose another split: d_ffn 64 to 640 at 64 to 1792 columns 0.1-0.9, 16 heads of 128 for 256 columns 0.94.
//               fp32 products of five to eight rows gain more than that (2048 columns, 192 units, 256 pairs, 1.27).  Where d_ffn is more than four times the
//               columns, or the heads more than twice, the residual stream has few owners that work while all wait: 0.78-0.97.
//   vocabulary  a head unit is 0.4 us and a barrier here, kernels stream: bf16, two layers of 512 columns, 4096 / 8192 / 16384 / 32000 / 151936 ids
//               1.25 / 1.18 / 1.06 / 0.83 / 0.45; a layer makes up for 1000 ids (24 layers, 32000 ids 1.06).  fp32, whose kernels' head is slower, by columns:
//               256 (88 CTAs), 8192 / 16384 / 50000 ids, one row 1.12 / 1.00 / 0.75, 8 rows, 32000 1.02; 512, 50000 / 100000 1.03 / 0.96; 1024, 100000 1.05.
//   width       the weights come no faster here: bf16, one row, 1792 / 2048 columns 1.03 / 0.94; fp32, one / four rows (the products are for four), 1024 1.10 / 1.18,
//               1280 0.90 / 1.05, 2048 0.85 / 0.99, five rows 1.07, and columns that do not fill their last stage, 384 to 1248, 0.82-0.96.
//   context     one CTA walks all of a pair's, attn_decode.cu splits it: bf16, 512 columns, one / eight rows, 200 / 600 / 800 / 2000 / 12000 tokens
//               1.21 / 1.03 / 0.96 / 0.74 / 0.27 and 1.26 / 1.10 / 1.01 / 0.79 / 0.32, 1024 columns, one row, 400 / 600 1.04 / 0.99; fp32, 256 columns,
//               one / eight rows, 400 / 600 / 1000 1.01 / 0.98 / 0.92 and 1.17 / 1.11 / 1.03, 768, four rows, 400 / 600 1.02 / 0.95, 1024, one / two / four
//               rows, 200 0.97 / 1.00 / 1.06, 400 0.92 / 0.93 / 0.99, 1536, eight rows, 400 / 600 1.07 / 0.99.  A layer gains less than head, sampling and update do, which one
//               iteration has once: 22 layers of 512 columns, bf16, six rows, 600 0.86; 18 of 384, fp32, one row, 300 0.87.
// 84 shapes, rows and contexts drawn at random from what is taken: 0.93-1.40, a tenth below 0.99, 1.11 in the middle.
bool resident_pays(const ResidentShape& m, int rows, int tokens) {
  const int grid = grid_of(m, 148), pairs = rows * (m.f32 ? m.H : m.KV);
  const bool many = m.f32 && rows > 4;
  if (grid < 80 || m.F < (m.f32 ? m.d : std::min(m.d, 1184)) || m.F > 4 * m.d || m.H * m.hd > 2 * m.d) return false;
  if (((m.H + 2 * m.KV) * m.hd / 16 > grid && !(many && m.d >= 1536)) || pairs > (many ? 2 * grid : grid)) return false;
  const auto walk = [&](int at_most, int a_layer, int once) { return tokens <= std::min(at_most, a_layer + once / m.n_layers); };
  if (!m.f32) return m.vocab <= 1024 * (m.n_layers + 6) && m.d <= 1792 && walk(512 + 32 * rows, 320 + 16 * rows, 1200);
  if (m.vocab > (many ? 128 : 64) * m.d * grid / 148 || (m.d > 256 && m.d % StageK<true>::value != 0)) return false;
  if (many) return walk(m.d <= 512 ? 800 : 448, 400, 1200);
  return m.d <= 1024 && walk(m.d <= 512 ? 448 : m.d <= 768 ? 320 : 64 * (rows + 1), 200, 750);
}

size_t resident_block_bytes(int n_layers) { return (size_t)n_layers * sizeof(ResidentLayer); }
size_t resident_slot_bytes(const ResidentShape& m) { return (size_t)words_of(m).all * 4; }

static_assert(sizeof(ResidentParams) <= sizeof(ResidentPlan) && alignof(ResidentParams) <= alignof(ResidentPlan), "room for the parameters");

cudaError_t resident_build(ResidentPlan* plan, void* dev_block, const ResidentBuild& a, cudaStream_t s) {
  const ResidentShape& m = a.shape;
  const int grid = grid_of(m, device_sms());
  int dev = 0, cooperative = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&cooperative, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !cooperative) return cudaErrorNotSupported;
  if (!resident_supported(m) || grid < 1 || (m.d / 16 + grid - 1) / grid > kOwn || (m.f32 && ((uintptr_t)a.kv_pool & 15))) return cudaErrorNotSupported;
  const std::unique_ptr<uint8_t[]> host(new (std::nothrow) uint8_t[resident_block_bytes(m.n_layers) + 128]);
  if (!host) return cudaErrorMemoryAllocation;
  uint8_t* hb = (uint8_t*)(((uintptr_t)host.get() + 127) & ~(uintptr_t)127);
  ResidentParams* P = new (plan->bytes) ResidentParams();
  ResidentLayer* Ls = reinterpret_cast<ResidentLayer*>(hb);
  const int hq = m.H * m.hd, nq = (m.H + 2 * m.KV) * m.hd;
  P->L = m.n_layers; P->d = m.d; P->H = m.H; P->KV = m.KV; P->hd = m.hd; P->F = m.F; P->V = m.vocab;
  P->v_limit = a.v_limit; P->max_pages = a.max_pages; P->model_id = a.model_id; P->eps = m.eps;
  P->temperature = a.temperature; P->seed = a.seed; P->embed = a.embed; P->final_norm = a.final_norm; P->rope = a.rope;
  P->page_table = a.page_table; P->slots = a.slots; P->err = a.err; P->dbg_logits = a.dbg_logits;
  const Words w = words_of(m);
  P->set_words = w.set; P->at_x = w.x; P->at_y = w.y; P->at_q = w.q; P->at_a = w.a; P->at_f = w.f; P->at_s = w.s;
  if (!tc_tensor_map_rows(a.head, m.f32, m.vocab, m.d, &P->head)) return cudaErrorNotSupported;
  for (int l = 0; l < m.n_layers; ++l) {
    ResidentLayer* Ly = new (Ls + l) ResidentLayer();
    if (!tc_tensor_map_rows(a.wqkv[l], m.f32, nq, m.d, &Ly->w[0]) || !tc_tensor_map_rows(a.wo[l], m.f32, m.d, hq, &Ly->w[1]) ||
        !tc_tensor_map_rows(a.wgu[l], m.f32, 2 * m.F, m.d, &Ly->w[2]) || !tc_tensor_map_rows(a.wdown[l], m.f32, m.d, m.F, &Ly->w[3]))
      return cudaErrorNotSupported;
    Ly->norm1 = a.norm1[l]; Ly->norm2 = a.norm2[l];
    Ly->kv = a.kv_pool + (size_t)l * a.layer_stride;
  }
  const cudaError_t e = cudaMemcpyAsync(dev_block, hb, resident_block_bytes(m.n_layers), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(s);             // the staging block goes away
}

namespace {

template <bool F32, bool EXT, int MT>
cudaError_t launch_as(const ResidentPlan& plan, const void* dev_block, int grid, const RowState& st, int which, int phase, int n_slots, const LoopParams& lp, cudaStream_t s) {
  static OncePerDevice configured;
  constexpr size_t smem = ResidentCfg<F32, EXT>::kSmem;
  const cudaError_t set = allow_smem(configured, decode_resident_kernel<F32, EXT, MT>, smem);
  if (set != cudaSuccess) return set;
  const ResidentParams& P = *reinterpret_cast<const ResidentParams*>(plan.bytes);
  const ResidentLayer* Ls = reinterpret_cast<const ResidentLayer*>(dev_block);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kBlock); cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;   // the CTAs wait for one another: all of them run, or none
  attr[0].val.cooperative = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, decode_resident_kernel<F32, EXT, MT>, P, Ls, st, which, phase, n_slots, lp);
  if (e == cudaErrorCooperativeLaunchTooLarge) (void)cudaGetLastError();     // the caller has another way
  return e != cudaSuccess ? e : launched(1);
}

}  // namespace

cudaError_t launch_decode_resident(const ResidentPlan& plan, const void* dev_block, const ResidentShape& m, bool kv_extended, const RowState& st, int which,
                                   int phase, int n_slots, const LoopParams& lp, int sharers, int sm_limit, cudaStream_t s) {
  if (n_slots < 1 || n_slots > kRows) return cudaErrorNotSupported;
  const int sms = device_sms();
  if (sms <= 0) return cudaErrorInvalidDevice;
  // A CTA takes the shared memory of its SM, so two phases of as many CTAs as there are SMs take turns.  Which CTA does a unit changes no bit: callers that
  // run at the same time get a part of the chip each, down to a quarter.  us an iteration of all, 1 / 2 / 4 callers of four rows each, steps of 24 tokens and all that
  // is around them, graphs -> so (all SMs each, two / four): bf16, 2 x 512 columns 49 / 55 / 68 -> 41 / 52 / 66 (70 / 136), 3 x 768 72 / 92 / 100 -> 63 / 85 / 128
  // (115 / 228), 8 x 1536 210 / 251 / 347 -> 188 / 287 / 409; fp32, 2 x 256 49 / 66 / 73 -> 43 / 47 / 62 (82 / 164), 4 x 512 99 / 132 / 198 -> 86 / 123 / 161 (183 / 363).
  // Graphs remain ahead for many callers of wide bf16 models, and for six of any (2 x 512 74 -> 91).
  // (Never fewer CTAs than own the residual stream's units, kOwn each: the full grid has as many.)
  const int grid = std::max(grid_of(m, sms / std::max(1, std::min(sharers, kSharers))), (m.d / 16 + kOwn - 1) / kOwn);
  if (grid > (sm_limit > 0 ? std::min(sm_limit, stream_sms(s)) : stream_sms(s))) return cudaErrorCooperativeLaunchTooLarge;
  const cudaError_t e = cudaMemsetAsync(reinterpret_cast<const ResidentParams*>(plan.bytes)->slots, 0xFF, resident_slot_bytes(m), s);
  if (e != cudaSuccess) return e;
  if (m.f32) return n_slots <= 4 ? launch_as<true, false, 4>(plan, dev_block, grid, st, which, phase, n_slots, lp, s)
                                 : launch_as<true, false, 8>(plan, dev_block, grid, st, which, phase, n_slots, lp, s);
  return kv_extended ? launch_as<false, true, 8>(plan, dev_block, grid, st, which, phase, n_slots, lp, s)
                     : launch_as<false, false, 8>(plan, dev_block, grid, st, which, phase, n_slots, lp, s);
}

}  // namespace rsd
