// What the backward kernels share: tile loads, the elementwise work of a tile, the order in which a key tile's steps are walked.
#pragma once
#include "tc_common.cuh"
#include "tc_launch.h"

namespace bdlm {
namespace tc {

using bf16 = __nv_bfloat16;

constexpr int TILE_BYTES = 2 * PANEL_BYTES;
// B MN-major (a [k][n] tile as loaded) with N = the head dimension
__host__ __device__ constexpr uint32_t idesc_km(int d) { return make_idesc(128, d, false, true); }

// One operand tile of head `head`: D / 64 panels of 64 columns (D = head dimension, 128 or 64).
template <int D>
__device__ __forceinline__ void tma_tile(uint32_t dst, const CUtensorMap* map, uint32_t bar, int head, int row0, int b) {
  tma_load_3d(dst, map, bar, head * D, row0, b);
  if (D == 128) tma_load_3d(dst + PANEL_BYTES, map, bar, head * D + 64, row0, b);
}

// The elementwise work of a tile, two elements per instruction where the arithmetic allows it: the compute warps are bound
// by instruction issue beside the exponential unit (L = 2048, H = 32: fused kernel 192 -> 189 us, windowed 32K 2.95 -> 2.85 ms,
// dQ pass at L = 16K, H = 8 1169 -> 1107 us; at the power cap, 32K, no change).  Scores x become P = exp2(x * scale - lse); hidden elements (bits of
// [lo, hi) clear) become zero.  nlse: minus the LSE rows in log2 units, one per element (-inf where there is no row).
template <int N>
__device__ __forceinline__ void exp_tile(uint32_t (&x)[N], uint64_t scale2, const float* nlse) {
#pragma unroll
  for (int c = 0; c < N; c += 4) {
    const ulonglong2 z = *reinterpret_cast<const ulonglong2*>(nlse + c);
    float p0, p1, p2, p3;
    unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), scale2, z.x), p0, p1);
    unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(x[c + 2]), __uint_as_float(x[c + 3])), scale2, z.y), p2, p3);
    x[c] = __float_as_uint(exp2f(p0)); x[c + 1] = __float_as_uint(exp2f(p1));
    x[c + 2] = __float_as_uint(exp2f(p2)); x[c + 3] = __float_as_uint(exp2f(p3));
  }
}
template <int N>
__device__ __forceinline__ void hide_tile(uint32_t (&x)[N], int lo, int hi) {
#pragma unroll
  for (int g = 0; g < N / 32; ++g) {
    const uint32_t seen = interval_bits(lo - 32 * g, hi - 32 * g);
#pragma unroll
    for (int e = 0; e < 32; ++e) x[32 * g + e] = (seen >> e) & 1u ? x[32 * g + e] : 0u;
  }
}
// dS = P * (dP - D) as bf16 pairs; nd: minus the D of each element.
template <int N>
__device__ __forceinline__ void ds_tile(uint32_t (&pk)[N / 2], const uint32_t (&x)[N], const uint32_t (&y)[N], const float* nd) {
#pragma unroll
  for (int c = 0; c < N; c += 4) {
    const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(nd + c);
    float d0, d1, d2, d3;
    unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])),
                           add_f32x2(pack_f32x2(__uint_as_float(y[c]), __uint_as_float(y[c + 1])), d.x)), d0, d1);
    unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(x[c + 2]), __uint_as_float(x[c + 3])),
                           add_f32x2(pack_f32x2(__uint_as_float(y[c + 2]), __uint_as_float(y[c + 3])), d.y)), d2, d3);
    pk[c / 2] = pack_bf16(d0, d1);
    pk[c / 2 + 1] = pack_bf16(d2, d3);
  }
}

// Write a thread's 128 accumulator columns (4 x 32) as bf16 to a global row, scaled.
__device__ __forceinline__ void store_row_chunk(bf16* dst, const uint32_t (&v)[32], float scale) {
#pragma unroll
  for (int e8 = 0; e8 < 4; ++e8) {
    uint4 o;
    uint32_t* po = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      po[e] = pack_bf16(__uint_as_float(v[e8 * 8 + 2 * e]) * scale, __uint_as_float(v[e8 * 8 + 2 * e + 1]) * scale);
    *reinterpret_cast<uint4*>(dst + e8 * 8) = o;
  }
}

// ---------------------------------------------------------------- steps of a key tile
struct QStep { int qs, h, q0; };

// The steps of a key tile: every (query tile, query stream, head of the group) that sees it.  Segment A holds the
// clean query tiles [a0, a1) (for a noisy key tile: the noisy ones), segment B the noisy query tiles [b0, b1) of a
// clean key tile, both in units of the step's query rows.  Segment A is walked first, then segment B, each from its
// last query tile down with all heads of the group inside a tile: CTAs that start together then meet the same
// Q / dO tiles -- and, in the fused kernel, the same dQ accumulator tiles -- at the same time, so that those stay in
// L2 between the CTAs that share them.  (Alternating the two streams tile by tile as well was measured and is
// slower: 4.7 against 3.3 ms on the sliding-window workload.)  Counters only, no division; the order is fixed, so
// dK / dV stay bitwise reproducible.
//
// When a key tile is split over a cluster (see key_unit), its steps are dealt out one by one: CTA `part` of `parts`
// takes steps part, part + parts, ... of the same order.
struct StepWalk {
  int a1, na, b1, nb, G, h_first, qs_a, rows, part, parts;
  int t, hh;   // tile counter over both segments, head within the group
  __device__ __forceinline__ int total() const { return (na + nb) * G; }
  __device__ __forceinline__ int count() const { return max(0, (total() - part + parts - 1) / parts); }
  __device__ __forceinline__ void init(int a0, int na_, int b0, int nb_, int G_, int h_first_, int qs_a_, int rows_, int part_, int parts_) {
    na = na_; nb = nb_; a1 = a0 + na_ - 1; b1 = b0 + nb_ - 1; G = G_; h_first = h_first_; qs_a = qs_a_; rows = rows_;
    part = part_; parts = parts_;
    t = 0; hh = part_;
    while (hh >= G) { hh -= G; ++t; }
  }
  __device__ __forceinline__ QStep cur() const {
    QStep s;
    s.h = h_first + hh;
    if (t < na) { s.qs = qs_a; s.q0 = (a1 - t) * rows; }
    else { s.qs = NOISY; s.q0 = (b1 - (t - na)) * rows; }
    return s;
  }
  __device__ __forceinline__ void next() {
    hh += parts;
    while (hh >= G) { hh -= G; ++t; }
  }
};


}  // namespace tc
}  // namespace bdlm
