// Tensor-core kernel (more than 16 tokens) of the packed LM-head forward
// (paper, Section 3.2, Eq. 7; no dense W_hat is formed, the residual is
// dequantised tile by tile inside the kernel as Appendix B allows).
//
// A unit of work is one 128-row vocabulary tile x TM tokens (64, 128 or 256).
// The vocabulary rows are the MMA's M side (one TMEM lane each), the tokens
// the N side.  Per stage of 128 of d:
//   - one producer warp loads the x tiles (up to 128 tokens each, bf16,
//     128-byte swizzle) by TMA into its ring, another the 8 KB of codes into
//     theirs, so codes run ahead of x as far as their ring allows;
//   - a converter warpgroup (two or four take stages in turn) turns the codes
//     into exact bf16 integers and stores them as the A operand in tensor
//     memory: the code layout is that of m16n8k16 fragments, which is the
//     register layout of tcgen05.st.16x128b;
//   - one thread issues eight tcgen05.mma (kind::f16, 128 rows x nt tokens x
//     16, nt a multiple of 16 up to 128, A from TMEM, B = x from shared memory,
//     fp32 accumulate) into a ring of TMEM accumulators; with 256 tokens, eight
//     for each half of them, so that each conversion serves 256 tokens and one
//     half's finished group is drained while the other computes;
//   - promotion warps read each finished block with tcgen05.ld and add
//     s[row, group] * partial to fp32 registers (group-wise scales cannot be
//     folded into exact bf16 operands).
// The rank-r branches are further k steps: 64 columns of int8 codes of A_c
// (factor 1) or A_w (factor = row scale of A_w) a stage, each 16 of them
// multiplied with the bf16 hi and lo parts of the pre-pass's t, read through a
// second tensor map.
//
// In the paper's packed format (SC4) a group scale is s_row * (q + 1) with a
// 4-bit code q.  The converters fold q + 1 into the operand (code * (q + 1)
// stays an exact bf16 integer, |.| <= 128), and blocks are 512 wide,
// promoted by s_row.
//
// What bounds it.  With A and x in shared memory (the earlier form of this
// kernel) a 128 x 256 x 16 MMA reads 12 KB in its 128 cycles, the x copy of a
// 64-wide k step writes 32 KB and the converters 16 KB: together more than the
// 128 bytes a cycle that shared memory moves, and it ran at 62 % of the
// measured tensor peak.  With A in TMEM an MMA of N tokens takes about N / 2 +
// 5 cycles (measured alone: 39 for 64, 67 for 128), and what is left is the
// issuing warp's own instructions (two turns a stage: about 1400 cycles, 1070
// of them MMAs).  Up to 64 tokens no role is busy all the time: an issuer's
// turn takes some 740 cycles for 200 to 310 of MMAs, and what does not depend
// on the tokens (the conversion of the codes, the promotion of the instance's
// whole width, group by group, the boundaries of units) shares the rest.
// Qwen3-8B shape, before and now: 24 tokens 150 -> 132 us, 64 tokens 246 ->
// 140, 4096 tokens 4.51 -> 3.66 ms; the paper's format 200 tokens 318 -> 223
// us, cross entropy of 2048 tokens 2.15 -> 1.65 ms; Gemma shape, cross entropy
// of 512 tokens 776 -> 570 us.
//
// Epilogues: logits (each promotion thread stores one row of its tokens),
// greedy partials (largest logit and its row per token over each warp's 32
// rows) and cross-entropy partials (max and sum of exp per token over each
// warp's 32 rows, plus the target's logit).  For the latter two a unit's sums
// pass through TMEM once more, read back in the 16x256b shape, so that a
// thread holds 4 rows of a quarter of the tokens and most of the reduction
// over rows is thread-local.
#pragma once

#include <cfloat>
#include <cuda.h>

#include "device.cuh"
#include "internal.h"

namespace archead {

constexpr int kPfTmemCols = 512;
constexpr float kLog2e = 1.4426950408889634f;  // log2(e)
constexpr float kLn2 = 0.6931471805599453f;    // ln(2)

// Instance geometry for TM tokens a unit, in kH halves of NT.  A stage is 128
// of d (or four 16-wide rank-r steps); x slots hold one half's.  TMEM: kNB
// accumulators of NT columns, then one A stage (128 rows x 128 k, 64 columns)
// a converter warpgroup.  Up to 128 tokens a stage's MMAs are short and its
// conversion is not (it does not depend on the tokens): four converter
// warpgroups; 256 tokens need the registers for 128 accumulators a promotion
// thread.
template <int TM>
struct PfGeom {
  static constexpr int NT = TM == 64 ? 64 : 128;
  static constexpr int kH = TM / NT;
  static constexpr int kConv = TM == 256 ? 2 : 4;    // converter warpgroups
  static constexpr int kPromo = TM == 64 ? 1 : 2;    // promotion warpgroups
  static constexpr int kCols = TM == 256 ? 128 : 64; // accumulator columns a promotion thread holds
  static constexpr int kThreads = 128 * (1 + kConv + kPromo);
  static constexpr int kNB = TM == 64 ? 4 : TM == 128 ? 2 : 3;
  static constexpr int kABase = kNB * NT;
  static constexpr int kAParts = TM == 256 ? 2 : 1;  // an A stage is released in parts (256 tokens: halves)
  static constexpr int kBoxBytes = NT * 64 * 2;      // one TMA box of x: 64 of d
  static constexpr int kXBytes = 2 * kBoxBytes;
  static constexpr int kXS = TM == 64 ? 8 : TM == 128 ? 4 : 5;
  static constexpr int kScaleOff = 2 * kChunkBytes;  // SC4: up to two byte rows of scale codes
  static constexpr int kCodeSlot = kScaleOff + 2 * kTileRows;
  static constexpr int kCS = TM == 64 ? 11 : TM == 128 ? 11 : 7;
  static constexpr int kCodeOff = kXS * kXBytes;
  static constexpr int kBarOff = kCodeOff + kCS * kCodeSlot;
  static constexpr int kBars = 2 * kXS + 2 * kCS + kConv * (1 + kAParts) + 2 * kNB + 1;
  static constexpr int kSmem = (TM == 128 ? 1024 : 0) + kBarOff + kBars * 8 + 16;
  // Registers a thread of the producer/MMA warpgroup, the converters and the
  // promotion warpgroups (launched with the largest multiple of 8 that fits);
  // their sum is that of the launch.
  static constexpr int kRegs0 = TM == 256 ? 48 : 56;
  static constexpr int kRegsC = TM == 64 ? 72 : 56;
  static constexpr int kRegsP = TM == 64 ? 128 : TM == 128 ? 112 : 160;
  static_assert(128 * (kRegs0 + kConv * kRegsC + kPromo * kRegsP) <= 65536 / kThreads / 8 * 8 * kThreads, "registers");
  static_assert(kABase + kConv * 64 <= kPfTmemCols, "TMEM columns");
  // A converter warpgroup waits for stage n in a code slot whose last stage, n
  // - kCS, was another's.  What it knows is that the MMAs of stage n - 2 kConv
  // are done (its own A stage was free for n - kConv); with fewer slots than
  // that the slot's barrier could still be a phase behind, which its parity
  // does not show.
  static_assert(kCS >= 2 * kConv, "code slots");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

struct PrefillParams {
  CUtensorMap tmap_x;   // bf16 [M][d], box 64 x nt, 128B swizzle
  CUtensorMap tmap_t;   // bf16 [M][2*LR], box 64 x nt, 128B swizzle
  const uint8_t *codes;
  const uint16_t *scales;  // fp16 group scales (INT8 format)
  const uint8_t *scodes;   // 4-bit group-scale codes (SC4 format)
  const uint16_t *s_row;   // residual row scales (SC4 format)
  const uint8_t *lr_codes;
  const uint16_t *s_a;
  int64_t V;
  int M, num_vt, num_mt, d_pad, G_pad, g, nls, nls_core;
  int nt;  // tokens of an MMA and of an x box, a multiple of 16 up to the instance's NT
  int G_pad2;
  int blk_log2;  // log2 of a residual block's 16-wide steps (g / 16; SC4: kSc4BlockLog2)
  void *out;
  int out_fp32;
  const int32_t *targets;  // global vocabulary rows
  int row0;                // global row of this pack's first row (vocabulary shards; 0 otherwise)
  float2 *ce_part;   // [num_vt * 4][M]
  float *ce_tlogit;  // [M]
  int *err;
  int64_t wait_budget;
};

// SC4: the residual is promoted every 512 of d.  (Longer blocks lose fp32
// accuracy in the tensor core's running sum; the promotion costs little.)
constexpr int kSc4BlockLog2 = 5;

// ------------------------------------------------------------------------
// tcgen05 / TMA wrappers (inline PTX).
// ------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(cols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_commit_a(uint32_t bar) {  // shared-memory address of the barrier
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// D (TMEM) = A (TMEM, 128 x 16) * B^T (shared memory) (+ D).
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 16 lanes x 32 columns from registers: a[4j + i] is register i of the
// m16n8k16 A fragment of 16-wide step j (rows t/4 and t/4 + 8 in the lanes,
// bf16 pairs along k in the columns).
__device__ __forceinline__ void tmem_st_frag4(uint32_t taddr, const uint32_t (&a)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(
          taddr),
      "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]), "r"(a[9]),
      "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]), "r"(a[15])
      : "memory");
}

// 32 lanes x 32 columns from registers, one value per column per thread.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float *a) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n" ::"r"(taddr),
      "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])), "r"(__float_as_uint(a[3])),
      "r"(__float_as_uint(a[4])), "r"(__float_as_uint(a[5])), "r"(__float_as_uint(a[6])), "r"(__float_as_uint(a[7])),
      "r"(__float_as_uint(a[8])), "r"(__float_as_uint(a[9])), "r"(__float_as_uint(a[10])),
      "r"(__float_as_uint(a[11])), "r"(__float_as_uint(a[12])), "r"(__float_as_uint(a[13])),
      "r"(__float_as_uint(a[14])), "r"(__float_as_uint(a[15])), "r"(__float_as_uint(a[16])),
      "r"(__float_as_uint(a[17])), "r"(__float_as_uint(a[18])), "r"(__float_as_uint(a[19])),
      "r"(__float_as_uint(a[20])), "r"(__float_as_uint(a[21])), "r"(__float_as_uint(a[22])),
      "r"(__float_as_uint(a[23])), "r"(__float_as_uint(a[24])), "r"(__float_as_uint(a[25])),
      "r"(__float_as_uint(a[26])), "r"(__float_as_uint(a[27])), "r"(__float_as_uint(a[28])),
      "r"(__float_as_uint(a[29])), "r"(__float_as_uint(a[30])), "r"(__float_as_uint(a[31]))
      : "memory");
}

// Loads of 16 registers that tmem_wait_ld completes.  kQuad false: 32 lanes x
// 16 columns, one value per column (32x32b).  kQuad true: 16 lanes x 32
// columns in the 16x256b shape: in repetition c thread t holds v[4c + j] =
// (lane t/4 + 8 (j >> 1), column 8c + 2 (t % 4) + (j & 1)).
template <bool kQuad>
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  if constexpr (kQuad)
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
  else
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// The registers pass through the wait, so nothing reads them before it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// 2^x by the special-function unit (ex2.approx, flushes denormal results).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

// d0 += a * b0 and d1 += a * b1 as one packed fp32x2 FMA (round to nearest).
__device__ __forceinline__ void fma2(float &d0, float &d1, float a, float b0, float b1) {
  asm("{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %2};\n mov.b64 rb, {%3, %4};\n mov.b64 rd, {%0, %1};\n"
      " fma.rn.f32x2 rd, ra, rb, rd;\n mov.b64 {%0, %1}, rd;\n}\n"
      : "+f"(d0), "+f"(d1)
      : "f"(a), "f"(b0), "f"(b1));
}

// One step of the base-2 log-sum-exp merge: (m, s) of two disjoint sets, s
// the sum of 2^(y - m), -> (m, s) of their union.  Maxima are finite: rows
// past the vocabulary enter as -FLT_MAX, whose difference with itself is 0
// and with any logit rounds to +-FLT_MAX or +-inf (weight 0).
__device__ __forceinline__ void lse2_merge(float am, float as, float bm, float bs, float &m, float &s) {
  const float d = am - bm;
  const float e = ex2_approx(-fabsf(d));
  s = d >= 0.f ? fmaf(bs, e, as) : fmaf(as, e, bs);
  m = fmaxf(am, bm);
}

// Shared-memory matrix descriptor: K-major operand in the 128-byte swizzle
// layout (8-row groups of 128-byte rows, 1024 bytes apart).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t desc = 0;
  desc |= (uint64_t)((saddr >> 4) & 0x3FFF);        // start address
  desc |= (uint64_t)1 << 16;                        // leading byte offset (unused for this layout)
  desc |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset: 8 rows x 128 B
  desc |= (uint64_t)1 << 46;                        // descriptor version (tcgen05)
  desc |= (uint64_t)2 << 61;                        // 128-byte swizzle
  return desc;
}

// Instruction descriptor: kind::f16, A = B = bf16, D = f32, K-major A and B.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Prefetch of a contiguous range into L2 (16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"(bytes) : "memory");
}

// bf16x2 fused multiply-add a * b + c (round to nearest even).
__device__ __forceinline__ uint32_t bf16x2_fma(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;\n" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// For a 4-bit scale code q: bf16x2 m = (q+1, q+1) and nb = (-136 (q+1), ...),
// so that fma(136 + code, m, nb) = code * (q + 1) exactly.  Every step is
// exact in bf16: 128 + q from the bits, minus 127; 136 (q+1) = 8 * 17 (q+1)
// has at most 8 significant bits.
struct Sc4Mult {
  uint32_t m, nb;
  __device__ __forceinline__ void set(uint32_t byte, int sh) {
    const uint32_t b = 0x43004300u + ((byte >> sh) & 15u) * 0x00010001u;
    m = bf16x2_sub(b, 0x42FE42FEu);  // 127
    asm("mul.rn.bf16x2 %0, %1, %2;\n" : "=r"(nb) : "r"(m), "r"(0xC308C308u));  // -136
  }
};

template <int N>
struct Int {
  static constexpr int value = N;
};

// Position of a ring of N slots: slot and phase parity, advanced in order.
template <int N>
struct RingPos {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int by = 1) {
    s += by;
    const bool wrap = s >= N;
    s = wrap ? s - N : s;
    ph ^= wrap;
  }
  __device__ __forceinline__ RingPos ahead(int by) const {
    RingPos r = *this;
    r.next(by);
    return r;
  }
};

// After a failed wait: lets the copies a producer has issued land before the
// block exits (`issued` of them over a ring of n slots; a whole warp calls it).
__device__ __forceinline__ void drain_copies(uint64_t *full, int n, int issued, int64_t budget, int *err) {
  for (int k = issued > n ? issued - n : 0; k < issued; ++k)
    mbar_wait_warp(&full[k % n], (uint32_t)(k / n) & 1, budget, nullptr, err);
}

// Per-token reductions over a warp's 32 rows of 64 token columns (half HH of
// the tile's NT), accumulators in the quad layout: acc[(NT/2) h + 4 kk + j] =
// row 8 (2h + (j >> 1)) + lane / 4, token column 8 kk + 2 (lane % 4) + (j & 1).
// So a thread holds rows ru + 8 kr (kr = 0..3, ru = lane / 4) of 16 columns
// col(k) = 8 (k >> 1) + 2 cq + (k & 1), row kr at acc[i0(k) + {0, 2, NT/2,
// NT/2 + 2}[kr]].  A butterfly over lane bits 4, 3, 2 halves the column set
// per step: lane (ru, cq) ends with columns 8 ru + 2 cq + j, j = 0, 1.
template <int NT, int HH>
__device__ __forceinline__ constexpr int quad_i0(int k) {
  return 4 * (8 * HH + (k >> 1)) + (k & 1);
}

// Greedy partials: the largest logit of each token and its row (lowest on ties).
template <int NT, int HH>
__device__ __forceinline__ void quad_argmax(const PrefillParams &p, const float (&acc)[NT], int64_t rbase, int64_t part, int m0,
                                            int mend, int lane) {
  const int ru = lane >> 2, cq = lane & 3;
  const int valid = rbase + 32 > p.V ? (int)(p.V - rbase) : 32;  // rows of the warp inside V
  float bv[16];
  int bi[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i0 = quad_i0<NT, HH>(k);
    float v = ru < valid ? acc[i0] : -INFINITY;
    int ix = ru;
    if (ru + 8 < valid && acc[i0 + 2] > v) v = acc[i0 + 2], ix = ru + 8;
    if (ru + 16 < valid && acc[i0 + NT / 2] > v) v = acc[i0 + NT / 2], ix = ru + 16;
    if (ru + 24 < valid && acc[i0 + NT / 2 + 2] > v) v = acc[i0 + NT / 2 + 2], ix = ru + 24;
    bv[k] = v;
    bi[k] = ix;
  }
#pragma unroll
  for (int n = 16, o = 16; n > 2; n >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < n / 2; ++j) {
      const float kv = up ? bv[j + n / 2] : bv[j];
      const int ki = up ? bi[j + n / 2] : bi[j];
      const float gv = up ? bv[j] : bv[j + n / 2];
      const int gi = up ? bi[j] : bi[j + n / 2];
      const float rv = __shfl_xor_sync(0xffffffffu, gv, o);
      const int ri = __shfl_xor_sync(0xffffffffu, gi, o);
      const bool take = rv > kv || (rv == kv && ri < ki);
      bv[j] = take ? rv : kv;
      bi[j] = take ? ri : ki;
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int m = m0 + 64 * HH + 8 * ru + 2 * cq + j;
    if (m < mend) p.ce_part[part * p.M + m] = make_float2(bv[j], __int_as_float((int)rbase + bi[j]));
  }
}

// Cross-entropy partials: (max, sum of exp(y - max)) of each token, and the
// target's logit.  The accumulators are in units of ln 2.
template <int NT, int HH>
__device__ __forceinline__ void quad_ce(const PrefillParams &p, float (&acc)[NT], int64_t rbase, int64_t part, int m0,
                                            int mend, int lane) {
  const int ru = lane >> 2, cq = lane & 3;
  m0 += 64 * HH;
  // Target logits first: a token whose target is one of this warp's 32 rows
  // takes its value from the thread holding it (a warp-uniform branch, taken
  // for 64 * 32 / V of the warps' halves).  Lane (ru, cq) reads the targets of
  // the columns it ends with; each thread then looks at its own 16 columns.
  // (Two shuffles for each of the 64 columns, in some warp of most units at
  // V = 32000, took up to half of the time: paper's format, d = 1024, 4096
  // tokens 447 us, now 256.)
  uint32_t tg = 0;  // row + 1 within the warp's 32 of column j's target in byte j, 0: elsewhere
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int m = m0 + 8 * ru + 2 * cq + j;
    const int64_t t64 = m < mend ? (int64_t)p.targets[m] - p.row0 - rbase : -1;  // row within the warp's 32
    if (t64 >= 0 && t64 < 32) tg |= (uint32_t)(t64 + 1) << (8 * j);
  }
  if (__any_sync(0xffffffffu, tg != 0)) {
    // (With the whole address formed per column the INT8 128-token instance
    // spilled 64 bytes and took up to 22 % longer.)
    float *tl = p.ce_tlogit + m0 + 2 * cq;
#pragma unroll
    for (int k = 0; k < 16; k += 2) {  // the thread's columns, their targets from lane (k / 2, cq)
      const uint32_t rs = __shfl_sync(0xffffffffu, tg, 4 * (k >> 1) + cq);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = (int)(rs >> (8 * j) & 255) - 1;
        if (r >= 0 && (r & 7) == ru) {
          const int i0 = quad_i0<NT, HH>(k + j);
          const float v =
              r & 16 ? (r & 8 ? acc[i0 + NT / 2 + 2] : acc[i0 + NT / 2]) : (r & 8 ? acc[i0 + 2] : acc[i0]);
          tl[8 * (k >> 1) + j] = v * kLn2;
        }
      }
    }
  }
  // Rows past V (last tile only) enter as -FLT_MAX: weight 0 against any
  // logit, and a finite (max, count) when the warp holds no real row.
  if (rbase + 32 > p.V) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int i0 = quad_i0<NT, HH>(k);
      if (rbase + ru >= p.V) acc[i0] = -FLT_MAX;
      if (rbase + ru + 8 >= p.V) acc[i0 + 2] = -FLT_MAX;
      if (rbase + ru + 16 >= p.V) acc[i0 + NT / 2] = -FLT_MAX;
      if (rbase + ru + 24 >= p.V) acc[i0 + NT / 2 + 2] = -FLT_MAX;
    }
  }
  float mx[16], sm[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i0 = quad_i0<NT, HH>(k);
    const float v0 = acc[i0], v1 = acc[i0 + 2], v2 = acc[i0 + NT / 2], v3 = acc[i0 + NT / 2 + 2];
    const float mk = fmaxf(fmaxf(v0, v1), fmaxf(v2, v3));
    mx[k] = mk;
    sm[k] = (ex2_approx(v0 - mk) + ex2_approx(v1 - mk)) + (ex2_approx(v2 - mk) + ex2_approx(v3 - mk));
  }
#pragma unroll
  for (int n = 16, o = 16; n > 2; n >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < n / 2; ++j) {
      const float km = up ? mx[j + n / 2] : mx[j], ks = up ? sm[j + n / 2] : sm[j];
      const float gm = up ? mx[j] : mx[j + n / 2], gs = up ? sm[j] : sm[j + n / 2];
      const float rm = __shfl_xor_sync(0xffffffffu, gm, o), rs = __shfl_xor_sync(0xffffffffu, gs, o);
      lse2_merge(km, ks, rm, rs, mx[j], sm[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int m = m0 + 8 * ru + 2 * cq + j;
    if (m < mend) p.ce_part[part * p.M + m] = make_float2(mx[j] * kLn2, sm[j]);
  }
}

// TM: tokens per unit; kMode 0: logits, 1: cross-entropy partials, 2: greedy
// (largest logit, row) partials; kSC4: the paper's packed format (group-scale
// codes times row scales).
template <int TM, int kMode, bool kSC4>
__global__ void __launch_bounds__(PfGeom<TM>::kThreads, 1) prefill_kernel(const __grid_constant__ PrefillParams p) {
  using G = PfGeom<TM>;
  constexpr int NT = G::NT, kNB = G::kNB, kXS = G::kXS, kCS = G::kCS, kConv = G::kConv, kCols = G::kCols;
  // The kernel has no static shared memory, so the dynamic window starts on a
  // 1 KB boundary, which the 128-byte-swizzled boxes rely on (checked).  The
  // 128-token instance rounds the address up all the same: with a base the
  // compiler knows its INT8 form takes 203 us for 100 tokens against 174 (the
  // 64-token instance gains 3 %).
  extern __shared__ uint8_t pf_smem_raw[];
  uint8_t *smem = pf_smem_raw;
  if constexpr (TM == 128)
    smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(pf_smem_raw) + 1023) & ~(uintptr_t)1023);
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0) atomicOr(p.err, kErrLayout);
    return;
  }
  uint64_t *x_full = reinterpret_cast<uint64_t *>(smem + G::kBarOff);
  uint64_t *x_empty = x_full + kXS;
  uint64_t *c_full = x_empty + kXS;
  uint64_t *c_empty = c_full + kCS;
  uint64_t *a_full = c_empty + kCS;
  uint64_t *a_empty = a_full + kConv;  // [kConv][kAParts]
  uint64_t *acc_full = a_empty + kConv * G::kAParts;
  uint64_t *acc_empty = acc_full + kNB;
  uint64_t *drain = acc_empty + kNB;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KC = p.d_pad / 128;      // residual stages
  const int KE = (p.nls + 3) / 4;    // rank-r stages of four 16-wide steps (the last: two or four)
  const int KS = KC + KE;
  const int num_units = p.num_vt * p.num_mt;
  // Promotion blocks of a tile: residual blocks, then the core and the
  // correction branches.
  const int nres = ((KC * 8 - 1) >> p.blk_log2) + 1;
  const bool has_core = p.nls_core > 0, has_corr = p.nls > p.nls_core;
  const int nb = nres + has_core + has_corr;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kXS; ++i) mbar_init(&x_full[i], 1), mbar_init(&x_empty[i], 1);
    for (int i = 0; i < kCS; ++i) mbar_init(&c_full[i], 1), mbar_init(&c_empty[i], 4);
    for (int i = 0; i < kConv; ++i) mbar_init(&a_full[i], 4);
    for (int i = 0; i < kConv * G::kAParts; ++i) mbar_init(&a_empty[i], 1);
    for (int i = 0; i < kNB; ++i) mbar_init(&acc_full[i], 1), mbar_init(&acc_empty[i], TM == 128 ? 8 : 4);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, kPfTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  bool mma_leader = false;  // the lane of warp 1 that issues the MMAs

  // Registers are rebalanced between warpgroups (PfGeom).  Each role's code
  // follows its own setmaxnreg so that the compiler allocates within that budget.
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(G::kRegs0) : "memory");
    if (warp == 0) {
      // ------------------------------ x producer ------------------------------
      // The whole warp runs the loop (uniform waits); one elected lane issues.
      const bool leader = elect_one();
      RingPos<kXS> r;
      int issued = 0;
      bool t_ready = false;
      for (int u = blockIdx.x; u < num_units; u += gridDim.x) {
        const int m0 = (u % p.num_mt) * (G::kH * p.nt);
        for (int e = 0; e < KS; ++e) {
          if (e == KC && !t_ready) {
            asm volatile("griddepcontrol.wait;\n" ::: "memory");  // t comes from the pre-pass grid
            t_ready = true;
          }
          for (int t = 0; t < G::kH; ++t) {
            if (!mbar_wait_warp(&x_empty[r.s], r.ph ^ 1, p.wait_budget, abort_flag, p.err)) {
              drain_copies(x_full, kXS, issued, p.wait_budget, p.err);
              goto done;
            }
            if (leader) {
              uint8_t *dst = smem + r.s * G::kXBytes;
              const CUtensorMap *map = e < KC ? &p.tmap_x : &p.tmap_t;
              const int c = (e < KC ? e : e - KC) * 128;
              const bool two = e < KC || 4 * (e - KC) + 2 < p.nls;
              mbar_arrive_expect_tx(&x_full[r.s], (uint32_t)p.nt * (two ? 256 : 128));
              tma_load_2d(dst, map, c, m0 + t * p.nt, &x_full[r.s]);
              if (two) tma_load_2d(dst + G::kBoxBytes, map, c + 64, m0 + t * p.nt, &x_full[r.s]);
            }
            ++issued;
            r.next();
            __syncwarp();
          }
        }
      }
    } else if (warp == 2) {
      // ------------------------------ code producer ------------------------------
      const bool leader = elect_one();
      RingPos<kCS> r;
      int issued = 0;
      const int lg = __ffs(p.g) - 1;
      const uint32_t scale_bytes = (uint32_t)p.G_pad * kTileRows * 2;
      for (int u = blockIdx.x; u < num_units; u += gridDim.x) {
        const int64_t vt = u / p.num_mt;
        if (!kSC4 && leader) {
          // The group scales are read by the promotion warps from global
          // memory: bring this block's first and then each next unit's to L2.
          if (u == (int)blockIdx.x) bulk_prefetch_l2(p.scales + vt * p.G_pad * kTileRows, scale_bytes);
          const int un = u + (int)gridDim.x;
          if (un < num_units && un / p.num_mt != vt)
            bulk_prefetch_l2(p.scales + (int64_t)(un / p.num_mt) * p.G_pad * kTileRows, scale_bytes);
        }
        for (int e = 0; e < KS; ++e) {
          if (!mbar_wait_warp(&c_empty[r.s], r.ph ^ 1, p.wait_budget, abort_flag, p.err)) {
            drain_copies(c_full, kCS, issued, p.wait_budget, p.err);
            goto done;
          }
          if (leader) {
            uint8_t *dst = smem + G::kCodeOff + r.s * G::kCodeSlot;
            if (e < KC) {
              // SC4: the byte rows of scale codes holding this stage's groups.
              const uint32_t sc = kSC4 ? (lg == 5 ? 2 * kTileRows : kTileRows) : 0;
              mbar_arrive_expect_tx(&c_full[r.s], 2 * kChunkBytes + sc);
              bulk_g2s(dst, p.codes + (vt * KC + e) * 2 * kChunkBytes, 2 * kChunkBytes, &c_full[r.s]);
              if (kSC4)
                bulk_g2s(dst + G::kScaleOff, p.scodes + (vt * p.G_pad2 + ((e * 128) >> lg >> 1)) * kTileRows, sc,
                         &c_full[r.s]);
            } else {
              const uint32_t bytes = min(4, p.nls - 4 * (e - KC)) * kLrStepBytes;
              mbar_arrive_expect_tx(&c_full[r.s], bytes);
              bulk_g2s(dst, p.lr_codes + (vt * p.nls + 4 * (e - KC)) * kLrStepBytes, bytes, &c_full[r.s]);
            }
          }
          ++issued;
          r.next();
          __syncwarp();
        }
      }
    } else if (warp == 1) {
      // ------------------------------ MMA issuer ------------------------------
      // As for the producers: the warp runs the loop, one elected lane issues.
      //
      // The halves of a unit take turns of at most one stage of a block (one
      // rank-r step, hi and lo), so that block starts alternate between them:
      // accumulator i of the ring is the unit's block (i - base) / kH of half
      // (i - base) % kH.
      const bool leader = elect_one();
      mma_leader = leader;
      const uint32_t idesc = idesc_bf16(128, p.nt);
      const uint64_t xdesc = smem_desc_sw128(smem_u32(smem));
      const uint32_t x_full_a = smem_u32(x_full), x_empty_a = smem_u32(x_empty), a_full_a = smem_u32(a_full),
                     a_empty_a = smem_u32(a_empty), acc_full_a = smem_u32(acc_full), acc_empty_a = smem_u32(acc_empty);
      constexpr uint32_t kBox = G::kBoxBytes >> 4;  // descriptor step to the second box of a slot
      RingPos<kXS> xr;
      RingPos<kConv> ar;
      RingPos<kNB> accr;  // next accumulator to start

      auto wait = [&](uint32_t bar, uint32_t ph) { return mbar_wait_warp_a(bar, ph, p.wait_budget, abort_flag, p.err); };
      // Starts the next accumulator once it is drained: its columns in d, its barrier in f.
      auto acc_take = [&](uint32_t &d, uint32_t &f) {
        d = tmem_base + accr.s * NT;
        f = acc_full_a + 8 * accr.s;
        accr.next();
      };
      auto acc_start = [&](uint32_t &d, uint32_t &f) {
        if (!wait(acc_empty_a + 8 * accr.s, accr.ph ^ 1)) return false;
        acc_take(d, f);
        return true;
      };
      // A satisfied mbarrier probe takes ~90 cycles here, and three in a row
      // before every eight MMAs left the tensor pipe idle.  So the next turn's
      // barriers are probed together between this turn's MMAs; only a turn
      // whose probe failed waits.  (Barriers a turn does not need repeat x's.)
      uint32_t polled = 0;  // this turn's barriers were all seen complete
      auto poll = [&](const RingPos<kXS> &x, bool need_a, const RingPos<kConv> &a, bool need_acc) {
        const uint32_t xb = x_full_a + 8 * x.s;
        polled = mbar_test3_a(xb, x.ph, need_a ? a_full_a + 8 * a.s : xb, need_a ? a.ph : x.ph,
                              need_acc ? acc_empty_a + 8 * accr.s : xb, need_acc ? accr.ph ^ 1 : x.ph);
      };
      // Before a half's first MMAs of a stage: its x, and (first half) the A stage.
      auto operands = [&](int t, const RingPos<kXS> &x) {
        return wait(x_full_a + 8 * x.s, x.ph) && (t > 0 || wait(a_full_a + 8 * ar.s, ar.ph));
      };
      // N MMAs from 16-wide step q0 of a residual stage; first: the block
      // starts here; f != 0: it ends here; free_a: no later half reads these A
      // columns.  With eight, `mid` runs between the first four and the rest.
      auto steps = [&](auto n, int q0, const RingPos<kXS> &x, uint32_t d, bool first, uint32_t f, bool free_a, auto mid) {
        constexpr int N = decltype(n)::value;
        tc_fence_after();
        const uint32_t a = tmem_base + G::kABase + ar.s * 64 + 8 * q0;
        const uint32_t ae = a_empty_a + 8 * G::kAParts * ar.s, xe = x_empty_a + 8 * x.s;
        const uint64_t b = xdesc + (uint32_t)(x.s * (G::kXBytes >> 4)) + (q0 >> 2) * kBox + 2 * (q0 & 3);
        if (leader) {
#pragma unroll
          for (int q = 0; q < (N < 4 ? N : 4); ++q)  // +2 in the descriptor: 32 bytes in 16-byte units
            tc_mma_ts(d, a + 8 * q, b + 2 * q, idesc, q > 0 || !first);
          if (q0 + N == 4 || N == 8) {
            if (G::kAParts == 2 && free_a) tc_commit_a(ae);
          }
        }
        __syncwarp();
        mid();
        if (leader) {
#pragma unroll
          for (int q = 4; q < N; ++q) tc_mma_ts(d, a + 8 * q, b + kBox + 2 * (q & 3), idesc, 1);
          if (q0 + N == 8) {
            tc_commit_a(xe);
            if (free_a) tc_commit_a(ae + 8 * (G::kAParts - 1));
          }
          if (f) tc_commit_a(f);
        }
        __syncwarp();
      };

      for (int u = blockIdx.x; u < num_units; u += gridDim.x) {
        uint32_t d0 = 0, d1 = 0, f0 = 0, f1 = 0;
        if (p.blk_log2 >= 3) {  // blocks of whole stages
          const int per = 1 << (p.blk_log2 - 3);
          int left = 0;  // stages to go in the block
          for (int e = 0; e < KC; ++e) {
            const bool first = left == 0;
            if (first) left = per;
            --left;
            const bool last = left == 0 || e + 1 == KC;
            if (!__all_sync(0xffffffffu, polled)) {
              if (first && !wait(acc_empty_a + 8 * accr.s, accr.ph ^ 1)) goto done;
              if (!operands(0, xr)) goto done;
            }
            if (first) acc_take(d0, f0);
            if constexpr (G::kH == 2) {
              const RingPos<kXS> x1 = xr.ahead(1);
              steps(Int<8>{}, 0, xr, d0, first, last ? f0 : 0, false, [&] { poll(x1, false, ar, first); });
              if (!__all_sync(0xffffffffu, polled)) {
                if (first && !wait(acc_empty_a + 8 * accr.s, accr.ph ^ 1)) goto done;
                if (!operands(1, x1)) goto done;
              }
              if (first) acc_take(d1, f1);
              xr.next(2);
              steps(Int<8>{}, 0, x1, d1, first, last ? f1 : 0, true, [&] { poll(xr, true, ar.ahead(1), left == 0); });
            } else {
              const RingPos<kXS> x0 = xr;
              xr.next();
              steps(Int<8>{}, 0, x0, d0, first, last ? f0 : 0, true, [&] { poll(xr, true, ar.ahead(1), left == 0); });
            }
            ar.next();
          }
          polled = 0;  // (the last probe may be of a rank-r stage)
        } else {  // groups of 64 (two blocks a stage) or 32 (four)
          const int nq = p.blk_log2 == 2 ? 4 : 2;
          for (int e = 0; e < KC; ++e) {
            for (int q0 = 0; q0 < 8; q0 += nq) {
              for (int t = 0; t < G::kH; ++t) {
                const RingPos<kXS> x = xr.ahead(t);
                uint32_t d, f;
                if (!acc_start(d, f)) goto done;
                if (q0 == 0 && !operands(t, x)) goto done;
                if (nq == 4)
                  steps(Int<4>{}, q0, x, d, true, f, t == G::kH - 1, [] {});
                else
                  steps(Int<2>{}, q0, x, d, true, f, t == G::kH - 1, [] {});
              }
            }
            ar.next();
            xr.next(G::kH);
          }
        }
        // Rank-r columns: step l of a stage is one branch's 16 columns (A
        // columns 8 l), hi and lo 16 columns of t each.
        for (int e = KC; e < KS; ++e) {
          const int ls0 = 4 * (e - KC), n = min(4, p.nls - ls0);
          if (ls0 + n <= p.nls_core || ls0 >= p.nls_core) {
            // All of one branch: issued together.  (Step by step the ten steps
            // of the Qwen3-8B shape took a tenth of a unit's time.)
            const bool first = ls0 == 0 || ls0 == p.nls_core;
            const bool last = ls0 + n == p.nls_core || ls0 + n == p.nls;
            const uint32_t ae = a_empty_a + 8 * G::kAParts * ar.s;
            const uint32_t a = tmem_base + G::kABase + ar.s * 64;
#pragma unroll
            for (int t = 0; t < G::kH; ++t) {
              const RingPos<kXS> x = xr.ahead(t);
              if (first) {
                if (t ? !acc_start(d1, f1) : !acc_start(d0, f0)) goto done;
              }
              if (!operands(t, x)) goto done;
              tc_fence_after();
              const uint64_t b = xdesc + (uint32_t)(x.s * (G::kXBytes >> 4));
              const uint32_t d = t ? d1 : d0;
              if (leader) {
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                  if (l >= 2 && n == 2) break;
                  tc_mma_ts(d, a + 8 * l, b + (l >> 1) * kBox + 4 * (l & 1), idesc, l > 0 || !first);
                  tc_mma_ts(d, a + 8 * l, b + (l >> 1) * kBox + 4 * (l & 1) + 2, idesc, 1);
                }
                tc_commit_a(x_empty_a + 8 * x.s);
                if (t == G::kH - 1) {
                  tc_commit_a(ae);
                  if (G::kAParts == 2) tc_commit_a(ae + 8);
                }
                if (last) tc_commit_a(t ? f1 : f0);
              }
              __syncwarp();
            }
          } else {
            for (int l = 0; l < n; ++l) {
              const int ls = 4 * (e - KC) + l;
              const bool first = ls == 0 || ls == p.nls_core;
              const bool last = ls == p.nls_core - 1 || ls == p.nls - 1;
              for (int t = 0; t < G::kH; ++t) {
                const RingPos<kXS> x = xr.ahead(t);
                if (first) {
                  uint32_t d, f;
                  if (!acc_start(d, f)) goto done;
                  if (t) d1 = d, f1 = f;
                  else d0 = d, f0 = f;
                }
                if (l == 0 && !operands(t, x)) goto done;
                tc_fence_after();
                const uint32_t a = tmem_base + G::kABase + ar.s * 64 + 8 * l;
                const uint32_t ae = a_empty_a + 8 * G::kAParts * ar.s;
                const uint64_t b = xdesc + (uint32_t)(x.s * (G::kXBytes >> 4)) + (l >> 1) * kBox + 4 * (l & 1);
                const uint32_t d = t ? d1 : d0;
                if (leader) {
                  tc_mma_ts(d, a, b, idesc, !first);
                  tc_mma_ts(d, a, b + 2, idesc, 1);
                  if (l == n - 1) {
                    tc_commit_a(x_empty_a + 8 * x.s);
                    if (t == G::kH - 1) {
                      tc_commit_a(ae);
                      if (G::kAParts == 2) tc_commit_a(ae + 8);
                    }
                  }
                  if (last) tc_commit_a(t ? f1 : f0);
                }
                __syncwarp();
              }
            }
          }
          ar.next();
          xr.next(G::kH);
        }
      }
    }
  } else if (warp < 4 + 4 * kConv) {
    // ------------------------------ converters ------------------------------
    // The converter warpgroups take the block's stages in turn, each into its
    // own A stage.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(G::kRegsC) : "memory");
    const int cg = (warp - 4) >> 2, cw = warp & 3;
    const int lg = __ffs(p.g) - 1;  // log2 g
    const uint32_t acol = tmem_base + ((uint32_t)(cw * 32) << 16) + G::kABase + cg * 64;
    uint64_t *ae = &a_empty[G::kAParts * cg];
    RingPos<kCS> cr;
    cr.next(cg);
    uint32_t aph = 0;
    for (int u = blockIdx.x, e = cg;; e += kConv) {
      while (e >= KS) e -= KS, u += gridDim.x;
      if (u >= num_units) break;
      if (!mbar_wait_warp(&c_full[cr.s], cr.ph, p.wait_budget, abort_flag, p.err)) goto done;
      const uint8_t *slot = smem + G::kCodeOff + cr.s * G::kCodeSlot;
      const uint8_t *codes = slot + (cw * 64 + lane) * 16;
      if (e < KC) {
        // The warp's codes of the stage first (m-tiles 2 cw and 2 cw + 1 of
        // two 64-wide halves); one m-tile's conversion overlaps the store of
        // the one before.
        uint4 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const uint4 *>(codes + (i >> 1) * kChunkBytes + (i & 1) * 512);
        uint32_t q[kSC4 ? 4 : 1];  // SC4: scale-code bytes of rows lane/4 + 8 i
        uint32_t q1[kSC4 ? 4 : 1];  // and of the second half where g = 32
        if constexpr (kSC4) {
          const uint8_t *sb = slot + G::kScaleOff + cw * 32 + (lane >> 2);
#pragma unroll
          for (int i = 0; i < 4; ++i) q[i] = sb[8 * i];
          if (lg == 5) {
#pragma unroll
            for (int i = 0; i < 4; ++i) q1[i] = sb[kTileRows + 8 * i];
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int hf = i >> 1, h = i & 1;
          uint32_t ah[16];
          const uint32_t ws[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
          Sc4Mult lo, hi;  // SC4: multipliers q + 1 of the half's group (two groups where g = 32)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t a[4];
            if constexpr (kSC4) {
              if (j == 0 || (j == 2 && lg == 5)) {
                const int sh = 4 * (((e * 128 + hf * 64 + 16 * j) >> lg) & 1);
                const bool second = hf == 1 && lg == 5;
                lo.set(second ? q1[2 * h] : q[2 * h], sh);
                hi.set(second ? q1[2 * h + 1] : q[2 * h + 1], sh);
              }
              unpack_int4x8_biased(ws[j], a);
              a[0] = bf16x2_fma(a[0], lo.m, lo.nb);
              a[1] = bf16x2_fma(a[1], hi.m, hi.nb);
              a[2] = bf16x2_fma(a[2], lo.m, lo.nb);
              a[3] = bf16x2_fma(a[3], hi.m, hi.nb);
            } else {
              unpack_int4x8(ws[j], a);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) ah[4 * j + k] = a[k];
          }
          if (h == 0 && hf < G::kAParts) {
            if (!mbar_wait_warp(ae + hf, aph ^ 1, p.wait_budget, abort_flag, p.err)) goto done;
            tc_fence_after();
          }
          tmem_st_frag4(acol + ((uint32_t)(16 * h) << 16) + 32 * hf, ah);
        }
      } else {  // four rank-r steps: the first half's 32 columns
        const uint8_t *lc = slot + (cw * 64 + lane) * 8;
        const int n = p.nls - 4 * (e - KC);
        uint2 w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          w[i] = i < 4 || n > 2 ? *reinterpret_cast<const uint2 *>(lc + (i >> 1) * kLrStepBytes + (i & 1) * 256)
                                : make_uint2(0x80808080u, 0x80808080u);
        // (The last part's release: the others come before it.)
        if (!mbar_wait_warp(ae + G::kAParts - 1, aph ^ 1, p.wait_budget, abort_flag, p.err)) goto done;
        tc_fence_after();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t ah[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t a[4];
            unpack_int8x8(w[2 * j + h].x, w[2 * j + h].y, a);
#pragma unroll
            for (int k = 0; k < 4; ++k) ah[4 * j + k] = a[k];
          }
          tmem_st_frag4(acol + ((uint32_t)(16 * h) << 16), ah);
        }
      }
      // The code slot is free once its words have gone into the A stage.  An
      // arrive right behind the loads had some of them moved behind it by the
      // compiler, where the refill could meet them (5 of 720 passes over 4096
      // tokens, Qwen3-8B shape, had a unit with wrong codes; none of 2880 since).
      asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&c_empty[cr.s]), mbar_arrive(&a_full[cg]);
      aph ^= 1;
      cr.next(kConv);
    }
  } else {
    // ------------------------------ promotion + epilogue ------------------------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(G::kRegsP) : "memory");
    const int pw = (warp - 4 - 4 * kConv) >> 2;  // warpgroup: half of the unit's tokens (256), or of the columns (128)
    const int hf = G::kH == 2 ? pw : 0;
    const int col0 = TM == 128 ? 64 * pw : 0;    // first accumulator column
    const int lg = warp & 3;                     // TMEM lane group (rows 32*lg .. 32*lg+31)
    // A thread sums one row x kCols tokens (32x32b).  Cross entropy and greedy
    // reduce over rows, with 4 rows x kCols/4 tokens per thread (16x256b): their
    // sums change shape through the tensor memory of the unit's last block.
    // (Promoting in that shape takes four factors a thread and half-height
    // loads for every block: 4.27 against 3.56 ms for 4096 tokens, Qwen3-8B
    // shape.)  Cross entropy accumulates in base 2, its factors times log2 e.
    const int rt0 = lg * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(lg * 32) << 16) + col0;
    RingPos<kNB> base;  // the unit's first accumulator
    for (int u = blockIdx.x; u < num_units; u += gridDim.x) {
      const int64_t vt = u / p.num_mt;
      const int mu = (u % p.num_mt) * (G::kH * p.nt);
      RingPos<kNB> accr = base.ahead(hf);
      {
        const int end = base.s + nb * G::kH;
        base.s = end % kNB;
        base.ph ^= (end / kNB) & 1;
      }
      const int m0 = mu + hf * p.nt + col0;               // token of the thread's first column
      const int mend = min(p.M, mu + (hf + 1) * p.nt);  // end of the half's tokens
      float acc[kCols];
#pragma unroll
      for (int i = 0; i < kCols; ++i) acc[i] = 0.f;
      // Promotion factor of a block's row, fp16 bits, loaded a block ahead.
      const uint16_t *fsrc = (kSC4 ? p.s_row + vt * kTileRows : p.scales + vt * p.G_pad * kTileRows) + rt0;
      uint16_t fn = *fsrc;
      for (int b = 0; b < nb; ++b) {
        const float f = fp16_bits_to_f32(fn) * (kMode == 1 ? kLog2e : 1.f);
        if (b + 1 < nres) {
          if (!kSC4) {
            fsrc += kTileRows;
            fn = *fsrc;
          }
        } else if (b + 1 == nres && has_core) {
          fn = 0x3C00;  // 1
        } else if (has_corr) {
          fn = p.s_a[vt * kTileRows + rt0];
        }
        if (!mbar_wait_warp(&acc_full[accr.s], accr.ph, p.wait_budget, abort_flag, p.err)) goto done;
        tc_fence_after();
        const uint32_t taddr = lane_addr + accr.s * NT;
        // Chunks of 16 registers, the next one loading while one is added.
        constexpr int kChunks = kCols / 16;
        uint32_t v[2][16];
        tmem_ld16<false>(taddr, v[0]);
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
          tmem_wait_ld(v[c & 1]);
          if (c + 1 < kChunks) tmem_ld16<false>(taddr + 16 * (c + 1), v[(c + 1) & 1]);
          float *a = acc + 16 * c;
          const uint32_t(&w)[16] = v[c & 1];
#pragma unroll
          for (int i = 0; i < 16; i += 2) fma2(a[i], a[i + 1], f, __uint_as_float(w[i]), __uint_as_float(w[i + 1]));
        }
        if (kMode != 0 && b + 1 == nb) {
          // To the shape of the row reductions, through the drained block.
#pragma unroll
          for (int c = 0; c < kCols; c += 32) tmem_st32(taddr + c, acc + c);
          asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
#pragma unroll
          for (int c = 0; c < kChunks; ++c) {  // rows 16 (c / (kCols/32)), columns 32 (c % (kCols/32))
            tmem_ld16<true>(taddr + ((uint32_t)(16 * (c / (kCols / 32))) << 16) + 32 * (c % (kCols / 32)), v[0]);
            tmem_wait_ld(v[0]);
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[16 * c + i] = __uint_as_float(v[0][i]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[accr.s]);
        accr.next(G::kH);
      }
      if constexpr (kMode == 0) {
        // Columns are tokens m0 + i, this thread's row is `row`.
        const int64_t row = vt * kTileRows + rt0;
        if (row < p.V) {
          const int mcount = mend - m0 < kCols ? mend - m0 : kCols;
          if (p.out_fp32) {
            float *o = reinterpret_cast<float *>(p.out) + (int64_t)m0 * p.V + row;
#pragma unroll
            for (int i = 0; i < kCols; ++i, o += p.V)
              if (i < mcount) *o = acc[i];
          } else {
            __nv_bfloat16 *o = reinterpret_cast<__nv_bfloat16 *>(p.out) + (int64_t)m0 * p.V + row;
#pragma unroll
            for (int i = 0; i < kCols; ++i, o += p.V)
              if (i < mcount) *o = __float2bfloat16_rn(acc[i]);
          }
        }
      } else {
        const int64_t rbase = vt * kTileRows + lg * 32, part = vt * 4 + lg;
        if constexpr (kMode == 2) {
          quad_argmax<kCols, 0>(p, acc, rbase, part, m0, mend, lane);
          if constexpr (kCols == 128) quad_argmax<kCols, 1>(p, acc, rbase, part, m0, mend, lane);
        } else {
          quad_ce<kCols, 0>(p, acc, rbase, part, m0, mend, lane);
          if constexpr (kCols == 128) quad_ce<kCols, 1>(p, acc, rbase, part, m0, mend, lane);
        }
      }
    }
  }
done:
  if (warp == 1 && mma_leader) {
    // Every MMA this thread issued has completed before TMEM is released.
    tc_commit(drain);
    mbar_wait(drain, 0, p.wait_budget, nullptr, p.err);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kPfTmemCols);
  }
}

// ------------------------------------------------------------------------
// Host side: tensor maps and launch.
// ------------------------------------------------------------------------
template <int TM, int kMode, bool kSC4>
cudaError_t launch_prefill_t(const PrefillParams &p, int grid, bool pdl, cudaStream_t s) {
  auto kern = prefill_kernel<TM, kMode, kSC4>;
  cudaError_t e = opt_in_smem(reinterpret_cast<const void *>(kern), PfGeom<TM>::kSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(PfGeom<TM>::kThreads);
  cfg.dynamicSmemBytes = PfGeom<TM>::kSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

// One packed format's kernel instances (INT8 in prefill.cu, SC4 in prefill_sc4.cu).
template <bool kSC4>
cudaError_t launch_prefill_fmt(const archead_pack *pk, const void *x, int M, const uint16_t *T, void *out,
                               int out_fp32, bool argmax, const int32_t *targets, int row0, float2 *ce_part,
                               float *ce_tlogit, bool pdl, cudaStream_t s) {
  PrefillParams p{};
  // Conversion of the codes is the same for any number of tokens, so a unit
  // takes as many as there are, up to 256.
  const int tm = M <= 64 ? 64 : M <= 128 ? 128 : 256;
  // Tokens spread evenly over the halves of the units.
  const int num_mt = (M + tm - 1) / tm, parts = num_mt * (tm == 256 ? 2 : 1);
  const int nt = ((M + parts - 1) / parts + 15) / 16 * 16;
  if (!make_tma_map_bf16(&p.tmap_x, x, M, pk->d, nt)) return cudaErrorInvalidValue;
  if (pk->lr > 0 && !make_tma_map_bf16(&p.tmap_t, T, M, 2 * pk->lr, nt)) return cudaErrorInvalidValue;
  p.codes = pk->codes;
  p.scales = pk->scales;
  p.scodes = pk->scodes;
  p.s_row = pk->s_row;
  p.G_pad2 = pk->G_pad2;
  p.lr_codes = pk->lr_codes;
  p.s_a = pk->s_a;
  p.V = pk->V;
  p.M = M;
  p.nt = nt;
  p.num_vt = pk->num_tiles;
  p.num_mt = num_mt;
  p.d_pad = pk->d_pad;
  p.G_pad = pk->G_pad;
  p.g = pk->g;
  p.blk_log2 = kSC4 ? kSc4BlockLog2 : __builtin_ctz(pk->g) - 4;
  p.nls = pk->nls;
  p.nls_core = pk->nls_core;
  p.out = out;
  p.out_fp32 = out_fp32;
  p.targets = targets;
  p.row0 = row0;
  p.ce_part = ce_part;
  p.ce_tlogit = ce_tlogit;
  p.err = pk->err;
  p.wait_budget = pk->wait_budget;
  const int64_t units = (int64_t)p.num_vt * p.num_mt;
  if (units > 0x7fffffff - pk->sm_count) return cudaErrorInvalidValue;
  const int grid = (int)(units < pk->sm_count ? units : pk->sm_count);
  const int mode = out ? 0 : argmax ? 2 : 1;
  const auto run = [&](auto t) {
    constexpr int TM = decltype(t)::value;
    return mode == 0   ? launch_prefill_t<TM, 0, kSC4>(p, grid, pdl, s)
           : mode == 1 ? launch_prefill_t<TM, 1, kSC4>(p, grid, pdl, s)
                       : launch_prefill_t<TM, 2, kSC4>(p, grid, pdl, s);
  };
  return tm == 64 ? run(Int<64>{}) : tm == 128 ? run(Int<128>{}) : run(Int<256>{});
}


}  // namespace archead
