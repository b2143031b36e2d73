// Quantisation and packing steps of the offline construction of a packed
// head (paper, Section 3.4, Algorithm 1; Appendix B steps 3-7): symmetric
// group-wise quantisers for the core factors (Q_8, Q_5), the group-wise INT4
// residual (one fp16 scale per group, or the paper's 4-bit scale codes times
// a row scale), the row-wise and group-wise INT8 correction factors, the
// packing of the codes into the canonical byte layouts, and the
// dequantisation of what was stored (the realized core W_d whose error the
// correction fits).  The dense linear algebra of the construction (the
// covariance product, the eigendecomposition, the randomized SVDs) is left to
// library routines; these kernels take the integer decisions.
//
// Quantiser (every variant): scale = fp16(max|x| / qmax) over the scale's
// group (fp32 division, round to nearest even), code = clamp(rint(x / scale),
// -qmax, qmax) with the division and the rounding (ties to even) in fp32, and
// code 0 where the scale is 0.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"

namespace archead {

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The code of one value by the definition above.
__device__ __forceinline__ uint32_t quant_code_div(float v, float s, float qmax) {
  if (!(s > 0.f)) return 0;
  return (uint32_t)(int)fminf(fmaxf(rintf(__fdiv_rn(v, s)), -qmax), qmax) & 255u;
}

// Codes of four values against their scales s with reciprocals inv = 1 / s
// (rounded), as the bytes of a word: bit for bit those of the definition, four
// operations a value instead of a division.  Adding 1.5 * 2^23 in the FMA
// rounds v * inv to an integer n, ties to even, in the sum's low bits.  v *
// inv and the rounded quotient differ by less than 2^-22 of their size, below
// 5e-5 for |v / s| < 200, so unless v * inv lies within 1e-4 of a half-integer
// both round to n (about 1 value in 5000 does).  Those, NaNs and infinities,
// and scales below the fp16 normal range (zero, or so coarse that |v / s| may
// exceed qmax; a normal scale leaves it below qmax + 0.1), take the definition.
__device__ __forceinline__ uint32_t quant_code4(float4 v, float4 s, float4 inv, float qmax) {
  constexpr float kMagic = 12582912.f;
  const float tx = fmaf(v.x, inv.x, kMagic), ty = fmaf(v.y, inv.y, kMagic);
  const float tz = fmaf(v.z, inv.z, kMagic), tw = fmaf(v.w, inv.w, kMagic);
  float off = fabsf(fmaf(v.x, inv.x, -(tx - kMagic)));  // distance from n; max.NaN keeps a NaN
  asm("max.NaN.f32 %0, %0, %1;\n" : "+f"(off) : "f"(fabsf(fmaf(v.y, inv.y, -(ty - kMagic)))));
  asm("max.NaN.f32 %0, %0, %1;\n" : "+f"(off) : "f"(fabsf(fmaf(v.z, inv.z, -(tz - kMagic)))));
  asm("max.NaN.f32 %0, %0, %1;\n" : "+f"(off) : "f"(fabsf(fmaf(v.w, inv.w, -(tw - kMagic)))));
  constexpr float kNormal = 6.103515625e-05f;  // 2^-14
  if (off < 0.4999f && fminf(fminf(s.x, s.y), fminf(s.z, s.w)) >= kNormal)
    return __byte_perm(__byte_perm(__float_as_uint(tx), __float_as_uint(ty), 0x0040),
                       __byte_perm(__float_as_uint(tz), __float_as_uint(tw), 0x0040), 0x5410);
  return quant_code_div(v.x, s.x, qmax) | quant_code_div(v.y, s.y, qmax) << 8 | quant_code_div(v.z, s.z, qmax) << 16 |
         quant_code_div(v.w, s.w, qmax) << 24;
}
__device__ __forceinline__ uint32_t quant_code4(float4 v, float s, float inv, float qmax) {
  return quant_code4(v, make_float4(s, s, s, s), make_float4(inv, inv, inv, inv), qmax);
}

__device__ __forceinline__ float abs_max4(float4 v) {
  return fmaxf(fmaxf(fmaxf(0.f, fabsf(v.x)), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));  // 0 if all are NaN
}

// Groups of kGc consecutive values of a row (32, 64, 128 or 256): with whole
// groups per row the matrix is one flat run of groups.  Memory bound (5 bytes
// a value).  A warp takes 512 values, four 16-byte loads a lane in flight,
// and keeps them in registers between the group maxima and the codes, so x is
// read once; the one-warp-per-group kernel below read it twice, 4 bytes a
// lane, and divided every value.
template <int kGc>
__global__ void __launch_bounds__(256) quantize_rows_kernel(const float4 *__restrict__ x, int64_t n4, float qmax,
                                                            uint32_t *__restrict__ codes,
                                                            uint16_t *__restrict__ scales) {
  constexpr int kU = 4;                               // float4 per lane
  constexpr int kLanes = kGc / 4 < 32 ? kGc / 4 : 32;  // lanes sharing a group
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); w * (32 * kU) < n4; w += warps) {
    const int64_t base = w * (32 * kU) + lane;
    float4 v[kU];
    float mx[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      v[u] = base + 32 * u < n4 ? __ldcs(x + base + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      mx[u] = abs_max4(v[u]);
#pragma unroll
      for (int o = kLanes / 2; o > 0; o >>= 1) mx[u] = fmaxf(mx[u], __shfl_xor_sync(0xffffffffu, mx[u], o));
    }
    if (kGc == 256) {  // two of the lane's values a group
#pragma unroll
      for (int u = 0; u < kU; u += 2) mx[u] = mx[u + 1] = fmaxf(mx[u], mx[u + 1]);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t i = base + 32 * u;
      if (i >= n4) break;
      const __half s16 = __float2half_rn(__fdiv_rn(mx[u], qmax));
      const float s = __half2float(s16);
      if ((i & (kGc / 4 - 1)) == 0) scales[i / (kGc / 4)] = __half_as_ushort(s16);
      codes[i] = quant_code4(v[u], s, __frcp_rn(s), qmax);
    }
  }
}

// Groups of gr >= 512 rows of one column (the core factors: gr = all rows),
// for any number of columns and any alignment.  A cluster of blocks takes one group of rows of eight adjacent
// columns (one 32-byte sector of a row), each block a slice of the rows:
// column maxima over its slice, the maximum over the cluster through
// distributed shared memory, then the codes, x coming mostly from L2 the
// second time.  One warp per column read one value per sector, on as many
// warps as there are columns (8.8 ms for 151936 x 128).
// kVec: cols is a multiple of 8, x 16-byte and codes 4-byte aligned.
constexpr int kColThreads = 512;
template <bool kVec>
__global__ void __launch_bounds__(kColThreads) quantize_columns_kernel(const float *__restrict__ x, int64_t cols,
                                                                       int64_t gr, float qmax,
                                                                       int8_t *__restrict__ codes,
                                                                       uint16_t *__restrict__ scales) {
  __shared__ float wmax[kColThreads / 32][8];
  __shared__ float bmax[8];  // this block's maxima, read by the cluster
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = threadIdx.x & 1;
  uint32_t rank, nrank;
  asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(nrank));
  const int64_t strips = (cols + 7) / 8;
  const int64_t job = blockIdx.x / nrank;  // (row group, strip)
  const int64_t c0 = (job % strips) * 8, r0 = (job / strips) * gr;
  const int nc = (int)(cols - c0 < 8 ? cols - c0 : 8);
  // Two threads a row, four columns each, eight rows in flight a thread.
  constexpr int kU = 8;
  const float *xs = x + r0 * cols + c0 + 4 * half;
  int8_t *cs = codes + r0 * cols + c0 + 4 * half;
  const int64_t step = (int64_t)nrank * (kColThreads / 2);
  const int64_t first = (int64_t)rank * (kColThreads / 2) + (threadIdx.x >> 1);
  auto load = [&](int64_t r) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < gr) {
      if (kVec) {
        v = *reinterpret_cast<const float4 *>(xs + r * cols);
      } else {
        if (4 * half + 0 < nc) v.x = xs[r * cols];
        if (4 * half + 1 < nc) v.y = xs[r * cols + 1];
        if (4 * half + 2 < nc) v.z = xs[r * cols + 2];
        if (4 * half + 3 < nc) v.w = xs[r * cols + 3];
      }
    }
    return v;
  };
  float mx[4] = {0.f, 0.f, 0.f, 0.f};
  for (int64_t r = first; r < gr; r += kU * step) {
    float4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = load(r + u * step);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      mx[0] = fmaxf(mx[0], fabsf(v[u].x));
      mx[1] = fmaxf(mx[1], fabsf(v[u].y));
      mx[2] = fmaxf(mx[2], fabsf(v[u].z));
      mx[3] = fmaxf(mx[3], fabsf(v[u].w));
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int o = 16; o > 1; o >>= 1) mx[j] = fmaxf(mx[j], __shfl_xor_sync(0xffffffffu, mx[j], o));
    if (lane < 2) wmax[warp][4 * half + j] = mx[j];
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    float m = 0.f;
#pragma unroll
    for (int w = 0; w < kColThreads / 32; ++w) m = fmaxf(m, wmax[w][threadIdx.x]);
    bmax[threadIdx.x] = m;
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  float s[4], inv[4];
  {
    float m = 0.f;  // lane j < 8 of every warp: column j over the cluster's blocks
    for (uint32_t b = 0; b < nrank; ++b) {
      uint32_t addr;
      float v;
      asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(addr) : "r"(smem_u32(&bmax[lane & 7])), "r"(b));
      asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(addr) : "memory");
      m = fmaxf(m, v);
    }
    const __half s16 = __float2half_rn(__fdiv_rn(m, qmax));
    if (rank == 0 && threadIdx.x < nc) scales[(job / strips) * cols + c0 + threadIdx.x] = __half_as_ushort(s16);
    const float sj = __half2float(s16);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      s[j] = __shfl_sync(0xffffffffu, sj, 4 * half + j);
      inv[j] = __frcp_rn(s[j]);
    }
  }
  // No block leaves while another may still read its maxima.
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  for (int64_t r = first; r < gr; r += kU * step) {
    float4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = load(r + u * step);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t ru = r + u * step;
      if (ru >= gr) break;
      const uint32_t q = quant_code4(v[u], make_float4(s[0], s[1], s[2], s[3]),
                                     make_float4(inv[0], inv[1], inv[2], inv[3]), qmax);
      if (kVec) {
        *reinterpret_cast<uint32_t *>(cs + ru * cols) = q;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (4 * half + j < nc) cs[ru * cols + j] = (int8_t)(q >> (8 * j));
      }
    }
  }
}

// The same where whole rows are read at once (cols a multiple of 4 up to
// 1024, 16-byte aligned, thousands of rows a group): three passes over x read
// as it lies, 16 bytes a lane.  A strip of eight columns touches a 128-byte
// line per row for 32 bytes of it, which held the kernel above at 93 us (L1
// bound) for 151936 x 128; the three passes take 38 us.
//   1: blocks (row slice, group) leave their column maxima at the start of
//      the group's codes, which are written only by pass 3;
//   2: a block per group turns them into scales;
//   3: codes.
constexpr int kColSlices = 304;  // most row slices of a group: two a multiprocessor
__global__ void __launch_bounds__(256) column_maxima_kernel(const float4 *__restrict__ x, int cols4, int64_t gr,
                                                            int8_t *__restrict__ codes) {
  __shared__ float4 red[256];
  const int lanes = 256 / cols4;  // rows read at a time by a block
  const int c = threadIdx.x % cols4, l = threadIdx.x / cols4;
  const float4 *xs = x + (int64_t)blockIdx.y * gr * cols4 + c;
  const int64_t step = (int64_t)gridDim.x * lanes;
  constexpr int kU = 8;
  float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int64_t r = (int64_t)blockIdx.x * lanes + l; l < lanes && r < gr; r += kU * step) {
    float4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = r + u * step < gr ? xs[(r + u * step) * cols4] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kU; ++u)
      m = make_float4(fmaxf(m.x, fabsf(v[u].x)), fmaxf(m.y, fabsf(v[u].y)), fmaxf(m.z, fabsf(v[u].z)),
                      fmaxf(m.w, fabsf(v[u].w)));
  }
  red[threadIdx.x] = m;
  __syncthreads();
  if (threadIdx.x < cols4) {
    for (int i = 1; i < lanes; ++i) {
      const float4 o = red[i * cols4 + c];
      m = make_float4(fmaxf(m.x, o.x), fmaxf(m.y, o.y), fmaxf(m.z, o.z), fmaxf(m.w, o.w));
    }
    float *part = reinterpret_cast<float *>(codes + (int64_t)blockIdx.y * gr * (4 * cols4)) + (int64_t)blockIdx.x * 4 * cols4;
    part[4 * c] = m.x, part[4 * c + 1] = m.y, part[4 * c + 2] = m.z, part[4 * c + 3] = m.w;
  }
}

__global__ void __launch_bounds__(256) column_scales_kernel(const int8_t *__restrict__ codes, int cols, int64_t gr,
                                                            int slices, float qmax, uint16_t *__restrict__ scales) {
  // Block (32 columns, group): warps stride over the slices.
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  const float *part = reinterpret_cast<const float *>(codes + (int64_t)blockIdx.y * gr * cols);
  float m = 0.f;
  if (c < cols) {
#pragma unroll 8
    for (int i = warp; i < slices; i += 8) m = fmaxf(m, part[(int64_t)i * cols + c]);
  }
  red[warp][lane] = m;
  __syncthreads();
  if (warp == 0 && c < cols) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = fmaxf(m, red[w][lane]);
    scales[(int64_t)blockIdx.y * cols + c] = __half_as_ushort(__float2half_rn(__fdiv_rn(m, qmax)));
  }
}

__global__ void __launch_bounds__(256) column_codes_kernel(const float4 *__restrict__ x, int cols4, int64_t gr,
                                                           float qmax, const uint16_t *__restrict__ scales,
                                                           uint32_t *__restrict__ codes) {
  const int lanes = 256 / cols4;
  const int c = threadIdx.x % cols4, l = threadIdx.x / cols4;
  if (l >= lanes) return;
  const int64_t base = (int64_t)blockIdx.y * gr * cols4 + c;
  const int64_t step = (int64_t)gridDim.x * lanes;
  const uint16_t *sc = scales + ((int64_t)blockIdx.y * cols4 + c) * 4;
  const float4 s = make_float4(fp16_bits_to_f32(sc[0]), fp16_bits_to_f32(sc[1]), fp16_bits_to_f32(sc[2]),
                               fp16_bits_to_f32(sc[3]));
  const float4 inv = make_float4(__frcp_rn(s.x), __frcp_rn(s.y), __frcp_rn(s.z), __frcp_rn(s.w));
  constexpr int kU = 8;
  for (int64_t r = (int64_t)blockIdx.x * lanes + l; r < gr; r += kU * step) {
    float4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      v[u] = r + u * step < gr ? x[base + (r + u * step) * cols4] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (r + u * step < gr) codes[base + (r + u * step) * cols4] = quant_code4(v[u], s, inv, qmax);
  }
}

// One warp per scale group of gr x gc elements of x [rows][cols]: the shapes
// that the kernels above do not take.
__global__ void quantize_symmetric_kernel(const float *__restrict__ x, int64_t rows, int64_t cols, int64_t gr,
                                          int64_t gc, int qmax, int8_t *__restrict__ codes,
                                          uint16_t *__restrict__ scales) {
  const int lane = threadIdx.x & 31;
  const int64_t ngc = cols / gc;
  const int64_t ngroups = (rows / gr) * ngc;
  const int64_t gsize = gr * gc;
  for (int64_t grp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; grp < ngroups;
       grp += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t r0 = (grp / ngc) * gr, c0 = (grp % ngc) * gc;
    float mx = 0.f;
    for (int64_t i = lane; i < gsize; i += 32) mx = fmaxf(mx, fabsf(x[(r0 + i / gc) * cols + c0 + i % gc]));
    mx = warp_max(mx);
    const __half s16 = __float2half_rn(__fdiv_rn(mx, (float)qmax));
    const float s = __half2float(s16);
    if (lane == 0) scales[grp] = __half_as_ushort(s16);
    for (int64_t i = lane; i < gsize; i += 32) {
      const int64_t idx = (r0 + i / gc) * cols + c0 + i % gc;
      float q = 0.f;
      if (s > 0.f) q = fminf(fmaxf(rintf(__fdiv_rn(x[idx], s)), (float)-qmax), (float)qmax);
      codes[idx] = (int8_t)q;
    }
  }
}

// The paper's format: one warp per row.  Group maxima, s_row = fp16(max /
// (7 * 16)), q = clamp(ceil(max_g / (7 s_row)) - 1, 0, 15), codes against
// s_row (q + 1) (exact in fp32).  gmax: per-warp scratch of G floats in
// shared memory.
__global__ void quantize_residual_sc4_kernel(const float *__restrict__ r, int64_t rows, int64_t cols, int g,
                                             int8_t *__restrict__ codes, uint8_t *__restrict__ qcodes,
                                             uint16_t *__restrict__ row_scale) {
  extern __shared__ float sc4_smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int G = (int)(cols / g);
  float *gmax = sc4_smem + (size_t)wib * G;
  for (int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; row < rows;
       row += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const float *rr = r + row * cols;
    float rmax = 0.f;
    for (int grp = 0; grp < G; ++grp) {
      float mx = 0.f;
      for (int i = lane; i < g; i += 32) mx = fmaxf(mx, fabsf(rr[(int64_t)grp * g + i]));
      mx = warp_max(mx);
      if (lane == 0) gmax[grp] = mx;
      rmax = fmaxf(rmax, mx);
    }
    __syncwarp();
    const __half sr16 = __float2half_rn(__fdiv_rn(rmax, 112.f));
    const float sr = __half2float(sr16);
    if (lane == 0) row_scale[row] = __half_as_ushort(sr16);
    for (int grp = 0; grp < G; ++grp) {
      int q = 0;
      if (sr > 0.f) q = min(max((int)ceilf(__fdiv_rn(gmax[grp], 7.f * sr)) - 1, 0), 15);
      if (lane == 0) qcodes[row * G + grp] = (uint8_t)q;
      const float s = sr * (float)(q + 1);
      for (int i = lane; i < g; i += 32) {
        const int64_t idx = row * cols + (int64_t)grp * g + i;
        float c = 0.f;
        if (s > 0.f) c = fminf(fmaxf(rintf(__fdiv_rn(r[idx], s)), -7.f), 7.f);
        codes[idx] = (int8_t)c;
      }
    }
    __syncwarp();
  }
}

// The same for g = 32, 64, 128 or 256 and rows from several groups (see the
// dispatch) up to 256 kNV float4 (cols <= 8192), 16-byte aligned: a block per
// row, the row held in registers, so r is read once (5 bytes a value in all,
// which bounds it).  Group maxima come from the kLanes lanes holding a group (two halves, for g
// = 256, meet in shared memory), the row maximum from the warps'; then one
// thread per group takes its scale code, scale and reciprocal, while the next
// row is on its way; four blocks a multiprocessor (151936 x 4096: 546 us;
// three, as the registers would have it, 577; five 586; 3.4 TB/s without the
// next row's loads).  The one-warp-per-row kernel read r twice, 4 bytes a
// lane, and divided every value.
constexpr int kSc4Threads = 256;
template <int kNV>
__global__ void __launch_bounds__(kSc4Threads, kNV <= 4 ? 4 : 2) quantize_residual_sc4_rows_kernel(
    const float4 *__restrict__ r, int64_t rows, int cols4, int lg, uint32_t *__restrict__ codes,
    uint8_t *__restrict__ qcodes, uint16_t *__restrict__ row_scale) {
  __shared__ float pmax[kSc4Threads * kNV / 8];  // per 32..128-wide piece of the row
  __shared__ float wmax[kSc4Threads / 32];
  __shared__ float2 gs[kSc4Threads * kNV / 8];   // (scale, reciprocal) per group
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g4 = 1 << (lg - 2);          // float4 per group
  const int lanes = g4 < 32 ? g4 : 32;   // lanes sharing a piece
  const int lp = lg - 2 < 5 ? lg - 2 : 5;  // log2 of the piece's float4 count
  const int G = cols4 >> (lg - 2);
  auto load = [&](int64_t row, float4 (&d)[kNV]) {
#pragma unroll
    for (int u = 0; u < kNV; ++u) {
      const int i = threadIdx.x + kSc4Threads * u;
      d[u] = row < rows && i < cols4 ? __ldcs(r + row * cols4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  float4 next[kNV];
  load(blockIdx.x, next);
  for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
    float4 v[kNV];
#pragma unroll
    for (int u = 0; u < kNV; ++u) v[u] = next[u];
    load(row + gridDim.x, next);
    float rmax = 0.f;
#pragma unroll
    for (int u = 0; u < kNV; ++u) {
      const int i = threadIdx.x + kSc4Threads * u;
      float m = abs_max4(v[u]);
      for (int o = lanes >> 1; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if ((lane & (lanes - 1)) == 0 && i < cols4) pmax[i >> lp] = m;
      rmax = fmaxf(rmax, m);
    }
    rmax = warp_max(rmax);
    if (lane == 0) wmax[warp] = rmax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kSc4Threads / 32; ++w) rmax = fmaxf(rmax, wmax[w]);
    const __half sr16 = __float2half_rn(__fdiv_rn(rmax, 112.f));
    const float sr = __half2float(sr16);
    if (threadIdx.x == 0) row_scale[row] = __half_as_ushort(sr16);
    for (int grp = threadIdx.x; grp < G; grp += kSc4Threads) {
      const float m = lg == 8 ? fmaxf(pmax[2 * grp], pmax[2 * grp + 1]) : pmax[grp];
      int q = 0;
      if (sr > 0.f) q = min(max((int)ceilf(__fdiv_rn(m, 7.f * sr)) - 1, 0), 15);
      qcodes[row * G + grp] = (uint8_t)q;
      const float s = sr * (float)(q + 1);
      gs[grp] = make_float2(s, __frcp_rn(s));
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kNV; ++u) {
      const int i = threadIdx.x + kSc4Threads * u;
      if (i >= cols4) break;
      const float2 sc = gs[i >> (lg - 2)];
      codes[row * cols4 + i] = quant_code4(v[u], sc.x, sc.y, 7.f);
    }
  }
}

// bits 4: two's complement (or unsigned 0..15) nibbles, byte j of a row =
// columns 2j (low) and 2j+1 (high), a missing last column packed as 0.
// bits 5: code j of a row in bits 5j..5j+4 of the row's little-endian bit
// string, ceil(5 cols / 8) bytes per row, unused top bits 0.
__global__ void pack_codes_kernel(const int8_t *__restrict__ codes, int64_t rows, int64_t cols, int bits,
                                  uint8_t *__restrict__ packed, int64_t row_bytes) {
  const int64_t total = rows * row_bytes;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / row_bytes, b = e % row_bytes;
    const int8_t *cr = codes + row * cols;
    uint32_t v = 0;
    if (bits == 4) {
      const uint32_t lo = (uint32_t)cr[2 * b] & 15u;
      const uint32_t hi = 2 * b + 1 < cols ? (uint32_t)cr[2 * b + 1] & 15u : 0u;
      v = lo | (hi << 4);
    } else {
      for (int k = 0; k < 8; ++k) {
        const int64_t bit = 8 * b + k, j = bit / 5;
        if (j < cols && ((((uint32_t)cr[j] & 31u) >> (bit % 5)) & 1u)) v |= 1u << k;
      }
    }
    packed[e] = (uint8_t)v;
  }
}

// 4-bit codes of an even number of columns: rows follow one another without
// padding, so the arrays are flat.  16 codes (one 16-byte load, four in
// flight) to 8 bytes a thread; a thread per byte with two 64-bit divisions
// took most of the packing time.
__global__ void __launch_bounds__(256) pack_nibbles_kernel(const uint4 *__restrict__ codes, int64_t n16,
                                                           uint2 *__restrict__ packed) {
  auto pack8 = [](uint32_t a, uint32_t b) {  // 8 codes -> 4 bytes
    a &= 0x0F0F0F0Fu;
    b &= 0x0F0F0F0Fu;
    return __byte_perm(a | a >> 4, b | b >> 4, 0x6420);
  };
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; i + 3 * step < n16; i += 4 * step) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = __ldcs(codes + i + u * step);
#pragma unroll
    for (int u = 0; u < 4; ++u) packed[i + u * step] = make_uint2(pack8(v[u].x, v[u].y), pack8(v[u].z, v[u].w));
  }
  for (; i < n16; i += step) {
    const uint4 v = codes[i];
    packed[i] = make_uint2(pack8(v.x, v.y), pack8(v.z, v.w));
  }
}

// out = code * scale for scales over gr x gc groups (fp32; exact).
__global__ void dequant_symmetric_kernel(const int8_t *__restrict__ codes, const uint16_t *__restrict__ scales,
                                         int64_t rows, int64_t cols, int64_t gr, int64_t gc, float *__restrict__ out) {
  const int64_t total = rows * cols, ngc = cols / gc;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / cols, c = e % cols;
    out[e] = (float)codes[e] * __half2float(__ushort_as_half(scales[(r / gr) * ngc + c / gc]));
  }
}

// The same for groups of 2^lgc >= 4 consecutive values of a row (the matrix
// is one flat run of groups): four codes to one 16-byte store a thread, four
// in flight, no divisions.
__global__ void __launch_bounds__(256) dequant_rows_kernel(const uint32_t *__restrict__ codes,
                                                           const uint16_t *__restrict__ scales, int64_t n4, int lgc,
                                                           float4 *__restrict__ out) {
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  auto store = [&](int64_t i, uint32_t w, uint16_t s16) {
    const float s = __half2float(__ushort_as_half(s16));
    out[i] = make_float4((float)(int8_t)w * s, (float)(int8_t)(w >> 8) * s, (float)(int8_t)(w >> 16) * s,
                         (float)(int8_t)(w >> 24) * s);
  };
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  for (; i + 3 * step < n4; i += 4 * step) {
    uint32_t w[4];
    uint16_t s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = codes[i + u * step], s[u] = scales[(i + u * step) >> (lgc - 2)];
#pragma unroll
    for (int u = 0; u < 4; ++u) store(i + u * step, w[u], s[u]);
  }
  for (; i < n4; i += step) store(i, codes[i], scales[i >> (lgc - 2)]);
}

// The paper's format: out = code * s_row * (q + 1).
__global__ void dequant_residual_sc4_kernel(const int8_t *__restrict__ codes, const uint8_t *__restrict__ qcodes,
                                            const uint16_t *__restrict__ row_scale, int64_t rows, int64_t cols, int g,
                                            float *__restrict__ out) {
  const int64_t total = rows * cols, G = cols / g;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / cols, c = e % cols;
    const float s = __half2float(__ushort_as_half(row_scale[r])) * (float)(qcodes[r * G + c / g] + 1);
    out[e] = (float)codes[e] * s;
  }
}

static unsigned grid_for(int64_t threads) {
  int64_t b = (threads + 255) / 256;
  return (unsigned)(b < 1 ? 1 : (b > 65535 * 8 ? 65535 * 8 : b));
}

}  // namespace archead

using namespace archead;

namespace {

archead_status fail_cuda(cudaError_t e) {
  set_last_error_message(cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? ARCHEAD_ERR_OOM : ARCHEAD_ERR_CUDA;
}

bool aligned(const void *p, size_t n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; }

// Blocks for grid-stride kernels: enough for several a multiprocessor, so
// that a thread's independent loads are in flight on every one of them.  (As
// kColSlices, sized for 152; the results do not depend on it.)
unsigned stream_grid(int64_t blocks) { return (unsigned)(blocks < 1 ? 1 : blocks < 152 * 32 ? blocks : 152 * 32); }

template <int kGc>
void launch_quantize_rows(const float *x, int64_t n, int qmax, int8_t *codes, uint16_t *scales, cudaStream_t s) {
  quantize_rows_kernel<kGc><<<stream_grid((n + 4095) / 4096), 256, 0, s>>>(
      reinterpret_cast<const float4 *>(x), n / 4, (float)qmax, reinterpret_cast<uint32_t *>(codes), scales);
}

cudaError_t launch_quantize_columns(const float *x, int64_t rows, int64_t cols, int64_t gr, int qmax, int8_t *codes,
                                    uint16_t *scales, cudaStream_t s) {
  const int64_t groups = rows / gr;
  // (Below a million values one launch costs less than three.)
  if (rows * cols >= 1 << 20 && cols % 4 == 0 && cols <= 1024 && gr >= 4 * kColSlices && groups <= 65535 &&
      aligned(x, 16) && aligned(codes, 4)) {
    const int cols4 = (int)(cols / 4);
    // Slices of at least the eight rows that a thread has in flight, as long as
    // all groups' together are two a multiprocessor.  (304 for every group,
    // nearly empty where groups are many: 200 groups of 1216 x 128 281 us
    // against 64, of 2048 x 32 199 / 28.)
    const int64_t full = gr / (8 * (256 / cols4));
    const int64_t least = (kColSlices + groups - 1) / groups;
    const int slices = (int)std::max(least, std::min<int64_t>(kColSlices, full));
    const dim3 grid((unsigned)slices, (unsigned)groups);
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    column_maxima_kernel<<<grid, 256, 0, s>>>(x4, cols4, gr, codes);
    column_scales_kernel<<<dim3((unsigned)((cols + 31) / 32), (unsigned)groups), 256, 0, s>>>(
        codes, (int)cols, gr, slices, (float)qmax, scales);
    column_codes_kernel<<<grid, 256, 0, s>>>(x4, cols4, gr, (float)qmax, scales, reinterpret_cast<uint32_t *>(codes));
    return cudaGetLastError();
  }
  const int64_t jobs = groups * ((cols + 7) / 8);
  const int cluster = gr >= 8 * kColThreads ? 8 : 1;  // blocks sharing a group: at least two rows a thread pair each
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(jobs * cluster));
  cfg.blockDim = dim3(kColThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const bool vec = cols % 8 == 0 && aligned(x, 16) && aligned(codes, 4);
  return cudaLaunchKernelEx(&cfg, vec ? quantize_columns_kernel<true> : quantize_columns_kernel<false>, x, cols, gr,
                            (float)qmax, codes, scales);
}

template <int kNV>
void launch_sc4_rows(const float *r, int64_t rows, int64_t cols, int lg, int8_t *codes, uint8_t *qcodes,
                     uint16_t *row_scale, cudaStream_t s) {
  quantize_residual_sc4_rows_kernel<kNV><<<stream_grid(rows), kSc4Threads, 0, s>>>(
      reinterpret_cast<const float4 *>(r), rows, (int)(cols / 4), lg, reinterpret_cast<uint32_t *>(codes), qcodes,
      row_scale);
}

int qmax_of(int bits) { return bits == 8 ? 127 : bits == 5 ? 15 : bits == 4 ? 7 : 0; }

}  // namespace

extern "C" {

ARCHEAD_API archead_status archead_quantize_symmetric(const float *x, int64_t rows, int64_t cols, int64_t group_rows,
                                                      int64_t group_cols, int bits, int8_t *codes, uint16_t *scales,
                                                      void *stream) {
  if (rows < 0 || cols < 0 || group_rows < 1 || group_cols < 1) return ARCHEAD_ERR_INVALID_ARG;
  if (rows % group_rows || cols % group_cols || qmax_of(bits) == 0) return ARCHEAD_ERR_INVALID_ARG;
  if (rows == 0 || cols == 0) return ARCHEAD_OK;
  if (!x || !codes || !scales) return ARCHEAD_ERR_INVALID_ARG;
  const int64_t ngroups = (rows / group_rows) * (cols / group_cols);
  const int qmax = qmax_of(bits);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool vec = group_rows == 1 && aligned(x, 16) && aligned(codes, 4);
  if (vec && group_cols == 32) {
    launch_quantize_rows<32>(x, rows * cols, qmax, codes, scales, s);
  } else if (vec && group_cols == 64) {
    launch_quantize_rows<64>(x, rows * cols, qmax, codes, scales, s);
  } else if (vec && group_cols == 128) {
    launch_quantize_rows<128>(x, rows * cols, qmax, codes, scales, s);
  } else if (vec && group_cols == 256) {
    launch_quantize_rows<256>(x, rows * cols, qmax, codes, scales, s);
  } else if (group_cols == 1 && group_rows >= kColThreads && ngroups <= (1 << 24)) {
    cudaError_t e = launch_quantize_columns(x, rows, cols, group_rows, qmax, codes, scales, s);
    if (e != cudaSuccess) return fail_cuda(e);
  } else {
    quantize_symmetric_kernel<<<grid_for(ngroups * 32), 256, 0, s>>>(x, rows, cols, group_rows, group_cols, qmax,
                                                                     codes, scales);
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ARCHEAD_OK : fail_cuda(e);
}

ARCHEAD_API archead_status archead_quantize_residual_sc4(const float *r, int64_t rows, int64_t cols, int group_size,
                                                         int8_t *codes, uint8_t *scale_codes, uint16_t *row_scale,
                                                         void *stream) {
  if (rows < 0 || cols < 0 || group_size < 1 || cols % group_size) return ARCHEAD_ERR_INVALID_ARG;
  if (rows == 0 || cols == 0) return ARCHEAD_OK;
  if (!r || !codes || !scale_codes || !row_scale) return ARCHEAD_ERR_INVALID_ARG;
  const int64_t G = cols / group_size;
  if (G > 1024) return ARCHEAD_ERR_UNSUPPORTED;  // per-warp group maxima in shared memory
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int lg = group_size == 32 ? 5 : group_size == 64 ? 6 : group_size == 128 ? 7 : group_size == 256 ? 8 : 0;
  const int64_t per = cols / 4;  // float4 a row
  // A block per row costs 1.3 to 1.5 ns a row however short the row is, a warp
  // per row 0.18 (g = 32), 0.28, 0.29, 0.43 (256) ns a group (151936 rows of
  // 128 columns, g = 128: 199 us against 49; of 512: 217 / 170; of 768: 229 /
  // 263; of 1024, g = 256: 240 / 260).
  const int64_t block_cols = group_size == 32 ? 256 : group_size == 64 ? 384 : group_size == 128 ? 768 : 1024;
  if (lg && cols >= block_cols && per <= 8 * kSc4Threads && aligned(r, 16) && aligned(codes, 4)) {
    if (per <= kSc4Threads) launch_sc4_rows<1>(r, rows, cols, lg, codes, scale_codes, row_scale, s);
    else if (per <= 2 * kSc4Threads) launch_sc4_rows<2>(r, rows, cols, lg, codes, scale_codes, row_scale, s);
    else if (per <= 4 * kSc4Threads) launch_sc4_rows<4>(r, rows, cols, lg, codes, scale_codes, row_scale, s);
    else launch_sc4_rows<8>(r, rows, cols, lg, codes, scale_codes, row_scale, s);
  } else {
    const size_t smem = (size_t)8 * G * sizeof(float);
    quantize_residual_sc4_kernel<<<grid_for(rows * 32), 256, smem, s>>>(r, rows, cols, group_size, codes, scale_codes,
                                                                        row_scale);
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ARCHEAD_OK : fail_cuda(e);
}

ARCHEAD_API archead_status archead_pack_codes(const int8_t *codes, int64_t rows, int64_t cols, int bits,
                                              uint8_t *packed, void *stream) {
  if (rows < 0 || cols < 0 || (bits != 4 && bits != 5)) return ARCHEAD_ERR_INVALID_ARG;
  if (rows == 0 || cols == 0) return ARCHEAD_OK;
  if (!codes || !packed) return ARCHEAD_ERR_INVALID_ARG;
  const int64_t row_bytes = bits == 4 ? (cols + 1) / 2 : (5 * cols + 7) / 8;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (bits == 4 && rows * cols % 16 == 0 && cols % 2 == 0 && aligned(codes, 16) && aligned(packed, 8)) {
    const int64_t n16 = rows * cols / 16;
    pack_nibbles_kernel<<<stream_grid((n16 + 1023) / 1024), 256, 0, s>>>(reinterpret_cast<const uint4 *>(codes), n16,
                                                                         reinterpret_cast<uint2 *>(packed));
  } else {
    pack_codes_kernel<<<grid_for(rows * row_bytes), 256, 0, s>>>(codes, rows, cols, bits, packed, row_bytes);
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ARCHEAD_OK : fail_cuda(e);
}

ARCHEAD_API archead_status archead_dequant_symmetric(const int8_t *codes, const uint16_t *scales, int64_t rows,
                                                     int64_t cols, int64_t group_rows, int64_t group_cols, float *out,
                                                     void *stream) {
  if (rows < 0 || cols < 0 || group_rows < 1 || group_cols < 1 || rows % group_rows || cols % group_cols)
    return ARCHEAD_ERR_INVALID_ARG;
  if (rows == 0 || cols == 0) return ARCHEAD_OK;
  if (!codes || !scales || !out) return ARCHEAD_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (group_rows == 1 && group_cols >= 4 && (group_cols & (group_cols - 1)) == 0 && aligned(codes, 4) &&
      aligned(out, 16)) {
    int lgc = 2;
    while (((int64_t)1 << lgc) < group_cols) ++lgc;
    const int64_t n4 = rows * cols / 4;
    dequant_rows_kernel<<<stream_grid((n4 + 1023) / 1024), 256, 0, s>>>(reinterpret_cast<const uint32_t *>(codes),
                                                                        scales, n4, lgc,
                                                                        reinterpret_cast<float4 *>(out));
  } else {
    dequant_symmetric_kernel<<<grid_for(rows * cols), 256, 0, s>>>(codes, scales, rows, cols, group_rows, group_cols,
                                                                   out);
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ARCHEAD_OK : fail_cuda(e);
}

ARCHEAD_API archead_status archead_dequant_residual_sc4(const int8_t *codes, const uint8_t *scale_codes,
                                                        const uint16_t *row_scale, int64_t rows, int64_t cols,
                                                        int group_size, float *out, void *stream) {
  if (rows < 0 || cols < 0 || group_size < 1 || cols % group_size) return ARCHEAD_ERR_INVALID_ARG;
  if (rows == 0 || cols == 0) return ARCHEAD_OK;
  if (!codes || !scale_codes || !row_scale || !out) return ARCHEAD_ERR_INVALID_ARG;
  dequant_residual_sc4_kernel<<<grid_for(rows * cols), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      codes, scale_codes, row_scale, rows, cols, group_size, out);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ARCHEAD_OK : fail_cuda(e);
}

}  // extern "C"
