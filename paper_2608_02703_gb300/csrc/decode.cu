// Host entry points of the decode kernel (decode_kernel.cuh); the INT8
// format's instances compile here, the SC4 format's in decode_sc4.cu.
#include <algorithm>

#include "decode_kernel.cuh"

namespace archead {

int decode_num_units(const archead_pack *p, int variant) {
  return (p->num_tiles + variant_tiles(variant) - 1) / variant_tiles(variant);
}

int decode_variant_tokens(int variant) { return variant_tokens(variant); }

int decode_parts_per_unit(int variant, bool sc4) { return variant_cw(variant, sc4); }

bool decode_supported(int d_pad, int nls, int g) {
  return decode_plan(d_pad, nls, g, kDecodeMaxTokens, kDecStreamed2).stages >= 2;
}

// Up to 8 tokens: x resident in shared memory (fp16) while that leaves a ring
// of at least 96 KB; otherwise, and for 9..16 tokens, the instance that
// streams x through the ring (very wide heads: 8 tokens of d = 16384 would
// take 256 KB).
// 17..32 and 33..64 tokens take the wide instances (one launch streams the
// head once for all of them) while their ring keeps at least four stages,
// else 16-token chunks of kDecStreamed2.  More than 64 tokens run in chunks
// of 64 (kDecWide8 for every chunk, the last one included).
static bool wide_fits(int d_pad, int nls, int g, int variant) {
  return decode_plan(d_pad, nls, g, variant_tokens(variant), variant).stages >= 4;
}

// Resident x in units of two tiles: for the paper's format (measured faster
// there: 63.8 against 65.7 us at M = 1 on the Qwen3-8B head), and for INT8
// heads whose four-tile units fill the last round of blocks at least 5 %
// worse than two-tile units would (Gemma-shaped head: 77.4 against 79.3 us
// with sixteen warps of one m-tile; on the Qwen3-8B head, where both fill it
// alike, two-tile units are 2.7 % slower).
static bool half_units(const archead_pack *p) {
  if (p->d_pad % (stage_chunks(kDecResidentH) * kChunkK) != 0) return false;  // whole stages of four chunks
  if (p->sc4) return true;
  const auto fill = [&](int tiles_per_unit) {
    const int units = (p->num_tiles + tiles_per_unit - 1) / tiles_per_unit;
    const int rounds = (units + p->sm_count - 1) / p->sm_count;
    return (double)units / ((double)rounds * p->sm_count);
  };
  return fill(2) > fill(4) + 0.05;
}

int decode_variant(const archead_pack *p, int M) {
  const int d_pad = p->d_pad, nls = p->nls_dec, g = p->g;
  if (M > 32 && wide_fits(d_pad, nls, g, kDecWide8)) return kDecWide8;
  if (M > 16 && wide_fits(d_pad, nls, g, kDecWide4)) return kDecWide4;
  // Streamed x, two n-tiles: in two-tile units where d is whole four-chunk
  // stages and that ring keeps at least four stages.
  const int streamed =
      d_pad % (stage_chunks(kDecStreamedH) * kChunkK) == 0 && wide_fits(d_pad, nls, g, kDecStreamedH)
          ? kDecStreamedH
          : kDecStreamed2;
  if (M > 8) return streamed;
  const int resident = half_units(p) ? kDecResidentH : kDecResident1;
  const DecodePlan pl = decode_plan(d_pad, nls, g, M, resident);
  return pl.stages >= 2 && pl.xs_off >= (size_t)96 * 1024 ? resident : streamed;
}

// AUTO's choice for 17 to 64 tokens: true where the decode kernel is the
// faster one.  The tensor-core kernel promotes every scale group of a tile
// into fp32 registers one after the other, which takes it as long at 17 tokens
// as at 64, so it loses INT8 heads with short groups (us, decode against
// tensor-core kernel, ranks 128 + 32, 24 tokens): V = 151936, d = 4096 189
// against 433 (g = 32) and 165 / 234 (64), but 150 / 135 (128) and 159 / 109
// (256); in the paper's format, whose blocks are 512 wide, 180 / 106 even for
// g = 32.  Above 32 tokens only g = 32 stays (64 tokens, the same head: 383 /
// 443 and, g = 64, 335 / 240).  With at most a tile a multiprocessor the
// decode kernel, whose units have two or four, loses (V = 8192, d = 1024,
// g = 32: 20.5 / 16.4); beyond, the two times are estimated from the busiest
// block's tiles: us per tile and 1024 of d, per tile and per launch, fitted to
// 2936 pairs of times (13 vocabulary sizes from 16000 to 262144, d 512 to
// 32768, logits and cross entropy).  On 150 other heads, every format and
// group size, AUTO took 0.6 % longer than the faster kernel on average.
//
// A short second round of tiles costs the tensor-core kernel most on narrow
// heads, where its start is most of the time (paper's format, g = 64, d = 512,
// 32 tokens: 14.5 / 16.5 at V = 19456 to 32000, 20.5 / 18.6 at 38800).  The
// same line for longer groups would gain as much, but there the decode kernel
// is the less accurate one (relative error at d = 512: 3.9e-6 against 2.1e-6
// for INT8, g = 256; 2.0e-6 both for the paper's format, g = 64), as it is
// without rank-r branches (1.3e-6 against 4.5e-8 at d = 4096; with them, the
// bf16 split of t leaves both at 2.2e-6).
bool decode_faster(const archead_pack *p, int M, bool reduce) {
  if (p->g > 64 || p->lr == 0 || !decode_supported(p->d_pad, p->nls_dec, p->g)) return false;
  const auto rounds = [&](int units) { return (units + p->sm_count - 1) / p->sm_count; };
  const int pf_tiles = rounds(p->num_tiles);
  if (p->sc4) return M <= 32 && pf_tiles == 2 && 5 * p->num_tiles <= 8 * p->sm_count && p->d <= 768;
  const int v = decode_variant(p, M);
  if (pf_tiles < 2 || (p->g == 64 && v == kDecWide8)) return false;
  const int launches = (M + variant_tokens(v) - 1) / variant_tokens(v);
  const int dec_tiles = launches * rounds(decode_num_units(p, v)) * variant_tiles(v);
  const bool g32 = p->g == 32;
  const float k = p->d_pad / 1024.f;
  const float per_k = v == kDecWide8 ? 8.f : v == kDecWide4 ? (g32 ? 5.f : 4.f) : (g32 ? 3.2f : 2.8f);
  const float per_tile = (v == kDecWide8 ? 1.5f : 0.f) + (reduce ? (v == kDecWide8 ? 3.5f : 2.f) : 0.f);
  return 10.f * launches + dec_tiles * (per_k * k + per_tile) < 5.5f + pf_tiles * (g32 ? 11.7f : 7.3f) * k;
}

extern template cudaError_t launch_decode_fmt<true>(const DecodeParams &, int, cudaStream_t, bool);
template cudaError_t launch_decode_fmt<false>(const DecodeParams &, int, cudaStream_t, bool);

cudaError_t launch_decode(const DecodeParams &dp, int grid, cudaStream_t s, bool pdl) {
  return dp.sc4 ? launch_decode_fmt<true>(dp, grid, s, pdl) : launch_decode_fmt<false>(dp, grid, s, pdl);
}

// Opt in every instance the pack can launch: the largest token count of
// each variant needs the most shared memory.
cudaError_t prepare_decode(const archead_pack *p) {
  if (!decode_supported(p->d_pad, p->nls_dec, p->g)) return cudaSuccess;
  // For every instance some M <= 64 selects, the M that needs it most shared
  // memory (the instance can change with M on heads too wide for x of every
  // token count to stay resident).
  constexpr int kVariants = 6;
  static_assert(kDecStreamedH + 1 == kVariants, "one entry per decode instance");
  int best_m[kVariants] = {0, 0, 0, 0, 0, 0};
  size_t best_bytes[kVariants] = {0, 0, 0, 0, 0, 0};
  for (int M = 1; M <= kDecodeWideTokens; ++M) {
    const int v = decode_variant(p, M);
    const int m = std::min(M, variant_tokens(v));
    const size_t bytes = decode_plan(p->d_pad, p->nls_dec, p->g, m, v).total;
    if (v >= 0 && v < kVariants && bytes >= best_bytes[v]) best_bytes[v] = bytes, best_m[v] = m;
  }
  DecodeParams dp = decode_params(p, nullptr, kDecodeWideTokens);
  for (int v = 0; v < kVariants; ++v) {
    if (best_m[v] == 0) continue;
    dp.variant = v;
    dp.M = best_m[v];
    const cudaError_t e = launch_decode(dp, 0, nullptr, false);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace archead
