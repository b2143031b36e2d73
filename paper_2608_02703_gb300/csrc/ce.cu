// Second pass of the fused cross-entropy epilogue (paper, Section 4: CE over
// held-out tokens, PPL = exp(CE)).  The forward kernels leave, per token and
// per slice of the vocabulary, the running maximum and the sum of
// exp(y - max) of the fp32 logits, plus the target's logit.  This kernel
// merges the slices in a fixed order and returns
//
//   ce[m] = max + log(sum) - y[m, t_m].
//
// A cluster of up to eight blocks takes up to 32 tokens: threads are (slice
// stride, token) with the token fastest, so the reads are coalesced for any
// token count (one token: consecutive slices), and the blocks of a cluster
// split the slices.  Bound by reading the partials (8 bytes per token and
// slice).  Few tokens were one warp each, a chain of dependent loads: 16 us
// for one token over the 4748 slices of the Qwen3-8B-shaped head; 512 tokens
// were 16 blocks.  Threads, warps and blocks are merged in a fixed order, so
// the result is deterministic.
#include "device.cuh"
#include "internal.h"

namespace archead {

// Where the merged (max, sum) of a token goes.  Whole head (row0 < 0):
// ce[m]; a target outside [0, V) gives NaN and latches kErrTargetRange.
// Vocabulary shard (row0 >= 0): out[3m .. 3m+2] = (max, sum, target logit),
// the target logit -inf when the target is not one of the shard's rows
// [row0, row0 + V) (another shard owns it; the combine checks the range).
__device__ __forceinline__ void ce_store(const LsePair &acc, int m, const float *__restrict__ tlogit,
                                         const int32_t *__restrict__ targets, int64_t row0, int64_t V,
                                         float *__restrict__ out, int *err) {
  const int64_t t = (int64_t)targets[m] - (row0 < 0 ? 0 : row0);
  const bool mine = t >= 0 && t < V;
  if (row0 >= 0) {
    out[3 * (int64_t)m] = acc.m;
    out[3 * (int64_t)m + 1] = acc.s;
    out[3 * (int64_t)m + 2] = mine ? tlogit[m] : -INFINITY;
  } else if (!mine) {
    out[m] = __int_as_float(0x7fc00000);
    atomicOr(err, kErrTargetRange);
  } else {
    out[m] = acc.m + logf(acc.s) - tlogit[m];
  }
}

// Greedy partials merge by (value, row): the larger value, the lower row on
// ties, so the result is the first maximum as in argmax.
struct LseMerge {
  static __device__ __forceinline__ float2 empty() { return make_float2(-INFINITY, 0.f); }
  static __device__ __forceinline__ float2 merge(float2 a, float2 b) {
    const LsePair r = lse_merge(LsePair{a.x, a.y}, LsePair{b.x, b.y});
    return make_float2(r.m, r.s);
  }
};
struct ArgmaxMerge {
  static __device__ __forceinline__ float2 empty() { return make_float2(-INFINITY, __int_as_float(0x7fffffff)); }
  static __device__ __forceinline__ float2 merge(float2 a, float2 b) {
    return b.x > a.x || (b.x == a.x && __float_as_int(b.y) < __float_as_int(a.y)) ? b : a;
  }
};

constexpr int kFinThreads = 512;

// Merged partial of this block's tokens, valid in threads t < tw of the
// cluster's first block (token blockIdx / cluster * tw + t).  tw: tokens per
// cluster, a power of two up to 32.
template <class Op>
__device__ __forceinline__ float2 merge_partials(const float2 *__restrict__ part, int num_parts, int M, int tw,
                                                 uint32_t rank, uint32_t nrank) {
  __shared__ float2 red[kFinThreads];
  const int t = threadIdx.x;
  const int strides = kFinThreads / tw;  // slices read at a time by a block
  const int m = (int)(blockIdx.x / nrank) * tw + (t & (tw - 1));
  const int step = strides * (int)nrank;
  float2 acc = Op::empty();
  asm volatile("griddepcontrol.wait;\n" ::: "memory");  // the forward's partials
  if (m < M) {
    int i = (int)rank * strides + t / tw;
    for (; i + 7 * step < num_parts; i += 8 * step) {
      float2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = part[(int64_t)(i + u * step) * M + m];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = Op::merge(acc, v[u]);
    }
    for (; i < num_parts; i += step) acc = Op::merge(acc, part[(int64_t)i * M + m]);
  }
  red[t] = acc;
  for (int h = kFinThreads / 2; h >= tw; h >>= 1) {
    __syncthreads();
    if (t < h) red[t] = acc = Op::merge(acc, red[t + h]);
  }
  if (nrank > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    if (rank == 0 && t < tw) {
      for (uint32_t b = 1; b < nrank; ++b) {
        uint32_t addr;
        float2 v;
        asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(addr) : "r"(smem_u32(&red[t])), "r"(b));
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
        acc = Op::merge(acc, v);
      }
    }
    // No block leaves while the first may still read its result.
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  }
  return acc;
}

__device__ __forceinline__ void cluster_rank(uint32_t &rank, uint32_t &nrank) {
  asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(nrank));
}

__global__ void __launch_bounds__(kFinThreads) ce_finalize_kernel(const float2 *__restrict__ part, int num_parts,
                                                                  int tw, const float *__restrict__ tlogit,
                                                                  const int32_t *__restrict__ targets, int64_t row0,
                                                                  int64_t V, int M, float *__restrict__ ce, int *err) {
  uint32_t rank, nrank;
  cluster_rank(rank, nrank);
  const float2 acc = merge_partials<LseMerge>(part, num_parts, M, tw, rank, nrank);
  const int m = (int)(blockIdx.x / nrank) * tw + (int)threadIdx.x;
  if (rank == 0 && (int)threadIdx.x < tw && m < M) ce_store(LsePair{acc.x, acc.y}, m, tlogit, targets, row0, V, ce, err);
}

__global__ void __launch_bounds__(kFinThreads) argmax_finalize_kernel(const float2 *__restrict__ part, int num_parts,
                                                                      int tw, int M, int32_t *__restrict__ index,
                                                                      float *__restrict__ value) {
  uint32_t rank, nrank;
  cluster_rank(rank, nrank);
  const float2 acc = merge_partials<ArgmaxMerge>(part, num_parts, M, tw, rank, nrank);
  const int m = (int)(blockIdx.x / nrank) * tw + (int)threadIdx.x;
  if (rank == 0 && (int)threadIdx.x < tw && m < M) {
    index[m] = __float_as_int(acc.y);
    if (value) value[m] = acc.x;
  }
}

// Grid of a finalize launch: tokens per cluster (32, or all of fewer), and
// one block per cluster while its threads have at most four slices each,
// else eight.
struct FinalizeLaunch {
  int tw = 1;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2] = {};
  FinalizeLaunch(int num_parts, int M, cudaStream_t s) {
    while (tw < M && tw < 32) tw *= 2;
    const int cluster = num_parts <= 4 * (kFinThreads / tw) ? 1 : 8;
    cfg.gridDim = dim3((unsigned)(((int64_t)M + tw - 1) / tw * cluster));
    cfg.blockDim = dim3(kFinThreads);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    // Launched while the forward grid drains; it waits for that grid's end
    // before it reads.
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};

cudaError_t launch_argmax_finalize(const float2 *part, int num_parts, int M, int32_t *index, float *value,
                                   cudaStream_t s) {
  FinalizeLaunch l(num_parts, M, s);
  return cudaLaunchKernelEx(&l.cfg, argmax_finalize_kernel, part, num_parts, l.tw, M, index, value);
}

static cudaError_t launch_finalize(const float2 *part, int num_parts, const float *tlogit, const int32_t *targets,
                                   int64_t row0, int64_t V, int M, float *out, int *err, cudaStream_t s) {
  FinalizeLaunch l(num_parts, M, s);
  return cudaLaunchKernelEx(&l.cfg, ce_finalize_kernel, part, num_parts, l.tw, tlogit, targets, row0, V, M, out, err);
}

cudaError_t launch_ce_finalize(const float2 *part, int num_parts, const float *tlogit, const int32_t *targets,
                               int64_t V, int M, float *ce, int *err, cudaStream_t s) {
  return launch_finalize(part, num_parts, tlogit, targets, -1, V, M, ce, err, s);
}

cudaError_t launch_lse_partial_finalize(const float2 *part, int num_parts, const float *tlogit,
                                        const int32_t *targets, int64_t row0, int64_t V, int M, float *parts3,
                                        cudaStream_t s) {
  return launch_finalize(part, num_parts, tlogit, targets, row0, V, M, parts3, nullptr, s);
}

// Combine of vocabulary shards (the paper's forward is row-separable, Eq. 7:
// each shard holds a contiguous block of rows).  Per token, the shards'
// (max, sum) pairs are merged in shard order and the target logit is taken
// from the one shard that owns the target:
//   ce[m] = max + log(sum) - y[m, t_m];
// NaN if no shard, or more than one, reports the target.
__global__ void lse_combine_kernel(const float *__restrict__ parts3, int num_shards, int M, float *__restrict__ ce) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  LsePair acc{-INFINITY, 0.f};
  float t = 0.f;
  int owners = 0;
  for (int p = 0; p < num_shards; ++p) {
    const float *q = parts3 + ((int64_t)p * M + m) * 3;
    acc = lse_merge(acc, LsePair{q[0], q[1]});
    if (q[2] != -INFINITY) {
      t = q[2];
      ++owners;
    }
  }
  ce[m] = owners == 1 ? acc.m + logf(acc.s) - t : __int_as_float(0x7fc00000);
}

// Greedy output of vocabulary shards: the largest (value, global row) over
// the shards, lowest row on ties (global row = shard-local index + row0 of
// its shard).
__global__ void argmax_combine_kernel(const float *__restrict__ values, const int32_t *__restrict__ indices,
                                      const int32_t *__restrict__ row0, int num_shards, int M,
                                      int32_t *__restrict__ index, float *__restrict__ value) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int p = 0; p < num_shards; ++p) {
    const float v = values[(int64_t)p * M + m];
    const int i = indices[(int64_t)p * M + m] + row0[p];
    if (v > bv || (v == bv && i < bi)) {
      bv = v;
      bi = i;
    }
  }
  index[m] = bi;
  if (value) value[m] = bv;
}

cudaError_t launch_lse_combine(const float *parts3, int num_shards, int M, float *ce, cudaStream_t s) {
  lse_combine_kernel<<<(M + 255) / 256, 256, 0, s>>>(parts3, num_shards, M, ce);
  return cudaGetLastError();
}

cudaError_t launch_argmax_combine(const float *values, const int32_t *indices, const int32_t *row0, int num_shards,
                                  int M, int32_t *index, float *value, cudaStream_t s) {
  argmax_combine_kernel<<<(M + 255) / 256, 256, 0, s>>>(values, indices, row0, num_shards, M, index, value);
  return cudaGetLastError();
}

}  // namespace archead
