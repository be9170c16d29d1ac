// Bandwidth-bound kernels of the BDLM attention path: the LSE merge of partial outputs
// (Eq. csbp-lse-merge over n partials, final division included) and the
// backward preprocess D_i = sum_d dO_i,d * O_i,d.
#include <type_traits>

#include "bdlm_common.cuh"

namespace bdlm {
namespace {

using bf16 = __nv_bfloat16;
constexpr int MAX_PARTIALS = 16;

struct MergeArgs {
  const void* o[MAX_PARTIALS];
  const float* lse[MAX_PARTIALS];
  int n;
};

// Eq. csbp-lse-merge for n partials at once: with m = max_j z_j and w_j = exp(z_j - m),
//   O = sum_j w_j O_j / sum_j w_j,   z = m + log sum_j w_j.
// One thread owns EPT (8 or 16) consecutive head-dim elements of one (row, head).  It first reads the row's n LSEs
// (n <= 16: they stay in registers), takes their maximum and turns them into normalised weights w_j / sum w; an empty
// partial (z_j = -inf) gets weight 0, a row whose partials are all empty gets O = 0 and z = -inf.  Then the
// partial outputs are streamed through once, four partials' loads in flight at a time, and added up with their
// weights -- no running rescale and nothing another thread could overwrite.
// NP = the number of partials rounded up to a multiple of four: the weights are a register array of that length.
template <bool F32IN, int EPT, int NP>
__global__ void __launch_bounds__(256, 3) merge_kernel(MergeArgs ma, int64_t total_chunks, int L, int H, int d,
                                                    bf16* __restrict__ o_out, float* __restrict__ lse_out) {
  constexpr int NV = F32IN ? EPT / 4 : EPT / 8;   // 16-byte vectors per thread and partial
  const int cpr = d / EPT;   // chunks per (row, head)
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total_chunks;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(idx % cpr);
    const int64_t rh = idx / cpr;
    const int h = (int)(rh % H);
    const int64_t row = rh / H;
    const int64_t bidx = row / L;
    const int i = (int)(row % L);
    const int64_t lidx = (bidx * H + h) * L + i;
    // The partial outputs do not depend on the weights: the first four partials' loads go out together with the
    // LSE loads; each later group of four is requested once the group in hand has been added up.
    uint4 cur[4][NV];
    auto request = [&](int j0, uint4 (&buf)[4][NV]) {
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        if (j0 + jj < ma.n) {
          const uint4* p = F32IN ? reinterpret_cast<const uint4*>(static_cast<const float*>(ma.o[j0 + jj]) + idx * EPT)
                                 : reinterpret_cast<const uint4*>(static_cast<const bf16*>(ma.o[j0 + jj]) + idx * EPT);
#pragma unroll
          for (int v = 0; v < NV; ++v) buf[jj][v] = p[v];
        }
      }
    };
    request(0, cur);
    float wgt[NP];
    float m = -INFINITY;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      wgt[j] = j < ma.n ? ma.lse[j][lidx] : -INFINITY;
      m = fmaxf(m, wgt[j]);
    }
    const float m_ref = (m == -INFINITY) ? 0.f : m;   // all empty: every weight becomes exp(-inf) = 0
    float wsum = 0.f;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      wgt[j] = (wgt[j] == -INFINITY) ? 0.f : expf(wgt[j] - m_ref);
      wsum += wgt[j];
    }
    const float inv = wsum > 0.f ? 1.f / wsum : 0.f;
    float acc[EPT];
#pragma unroll
    for (int e = 0; e < EPT; ++e) acc[e] = 0.f;
#pragma unroll
    for (int j0 = 0; j0 < NP; j0 += 4) {
      if (j0 >= ma.n) break;
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        if (j0 + jj >= ma.n) break;
        const float wj = wgt[j0 + jj] * inv;
        if (F32IN) {
          const float* pf = reinterpret_cast<const float*>(&cur[jj][0]);
#pragma unroll
          for (int e = 0; e < EPT; ++e) acc[e] = fmaf(wj, pf[e], acc[e]);
        } else {
          const __nv_bfloat162* p2 = reinterpret_cast<const __nv_bfloat162*>(&cur[jj][0]);
#pragma unroll
          for (int e = 0; e < EPT / 2; ++e) {
            const float2 f = __bfloat1622float2(p2[e]);
            acc[2 * e] = fmaf(wj, f.x, acc[2 * e]);
            acc[2 * e + 1] = fmaf(wj, f.y, acc[2 * e + 1]);
          }
        }
      }
      if (j0 + 4 < ma.n) request(j0 + 4, cur);
    }
#pragma unroll
    for (int v = 0; v < EPT / 8; ++v) {
      uint4 outv;
      uint32_t* ow = reinterpret_cast<uint32_t*>(&outv);
#pragma unroll
      for (int e = 0; e < 4; ++e) ow[e] = pack_bf16(acc[8 * v + 2 * e], acc[8 * v + 2 * e + 1]);
      reinterpret_cast<uint4*>(o_out + idx * EPT)[v] = outv;
    }
    if (c == 0) lse_out[lidx] = wsum > 0.f ? m + logf(wsum) : -INFINITY;
  }
}

// What the backward needs before its first key tile, for both query streams in one launch: D = sum over d of dO * O
// (fp32), and the fp32 dQ accumulators of the fused kernel set to zero.  A block takes PREP_ROWS consecutive rows of
// PREP_HEADS heads; dO and O are read as they lie ([batch, L, H, d]), the sums go through shared memory and leave as
// 128-byte runs along L of the [batch, H, L] result (written straight from the reading lanes they would be 4-byte stores
// H*4 apart).  A pure stream: bound by memory at large sizes (32K rows, H = 32: 2.15 GB in 340 us = 6.3 TB/s), by the
// number of blocks at small ones, hence the split over the heads too.
// Against one launch per stream over all heads of a row tile plus a memset: L = 2048, H = 32 (64 blocks a launch, now
// 1024) 78 -> 23 us; 32K 472 -> 340 us.
constexpr int PREP_ROWS = 32, PREP_HEADS = 4;
struct PrepArgs {
  const bf16* dout[2];
  const bf16* o[2];
  float* dsum[2];      // nullptr: the stream has no queries
  float* dq32[2];      // nullptr: nothing to zero
  int rows[2], dq32_rows[2];
  int blocks_clean, H;
};
template <int D>
__global__ void __launch_bounds__(256) bwd_prepare_kernel(const PrepArgs pa) {
  __shared__ float sums[PREP_HEADS][PREP_ROWS + 1];
  wait_for_predecessor();
  constexpr int LPR = D / 8;               // lanes per row
  constexpr int RPP = 256 / LPR;           // rows per pass of the block
  constexpr int UNROLL = 4;
  const int s = (int)blockIdx.x < pa.blocks_clean ? CLEAN : NOISY;
  auto of = [&](const auto& x) { return s == CLEAN ? x[0] : x[1]; };   // (an index computed at run time would copy the arguments to local memory)
  const int L = of(pa.rows), H = pa.H;
  int i = blockIdx.x - (s == CLEAN ? 0 : pa.blocks_clean);
  const int hgroups = (H + PREP_HEADS - 1) / PREP_HEADS, tiles = (L + PREP_ROWS - 1) / PREP_ROWS;
  const int h0 = (i % hgroups) * PREP_HEADS;   // neighbouring blocks read neighbouring heads of the same rows
  i /= hgroups;
  const int l0 = (i % tiles) * PREP_ROWS, b = i / tiles;
  const int nl = min(PREP_ROWS, L - l0), nh = min(PREP_HEADS, H - h0);
  const int64_t base = ((int64_t)b * L + l0) * H + h0;
  const int sub = threadIdx.x / LPR, c = threadIdx.x % LPR;
  const bf16 *dout = of(pa.dout), *o = of(pa.o);
  float* dq32 = of(pa.dq32);
  const int dq32_rows = of(pa.dq32_rows);
  constexpr int NROWS = PREP_ROWS * PREP_HEADS;   // r = li * PREP_HEADS + hi
#pragma unroll 1
  for (int r0 = 0; r0 < NROWS; r0 += RPP * UNROLL) {
    uint4 ua[UNROLL], ub[UNROLL];
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
      const int r = r0 + j * RPP + sub, li = r / PREP_HEADS, hi = r % PREP_HEADS;
      if (li < nl && hi < nh) {
        const int64_t at = (base + (int64_t)li * H + hi) * D + c * 8;
        ua[j] = *reinterpret_cast<const uint4*>(dout + at);
        ub[j] = *reinterpret_cast<const uint4*>(o + at);
      } else {
        ua[j] = make_uint4(0u, 0u, 0u, 0u); ub[j] = ua[j];
      }
    }
    if (r0 == 0 && dq32 != nullptr) {   // the stores go out under the first loads; the last rows' block clears the padding too
      const int nz = l0 + PREP_ROWS >= L ? dq32_rows - l0 : PREP_ROWS;
      for (int hi = 0; hi < nh; ++hi) {
        float4* z = reinterpret_cast<float4*>(dq32 + (((int64_t)b * H + h0 + hi) * dq32_rows + l0) * D);
        for (int e = threadIdx.x; e < nz * D / 4; e += 256) z[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
      const uint32_t* pa_ = reinterpret_cast<const uint32_t*>(&ua[j]);
      const uint32_t* pb_ = reinterpret_cast<const uint32_t*>(&ub[j]);
      float acc = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pa_[e]));
        const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&pb_[e]));
        acc = fmaf(x.x, y.x, fmaf(x.y, y.y, acc));
      }
#pragma unroll
      for (int sft = LPR / 2; sft > 0; sft >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, sft);
      const int r = r0 + j * RPP + sub;
      if (c == 0) sums[r % PREP_HEADS][r / PREP_HEADS] = acc;
    }
  }
  __syncthreads();
  if (threadIdx.x < NROWS) {
    const int hi = threadIdx.x / PREP_ROWS, li = threadIdx.x % PREP_ROWS;
    if (hi < nh && li < nl) of(pa.dsum)[((int64_t)b * H + h0 + hi) * L + l0 + li] = sums[hi][li];
  }
}

}  // namespace

cudaError_t launch_merge(int n, int batch, int L, int H, int d, const void* const* o_parts,
                         const float* const* lse_parts, int dtype, void* o_out, float* lse_out,
                         cudaStream_t st) {
  MergeArgs ma;
  ma.n = n;
  for (int j = 0; j < MAX_PARTIALS; ++j) {
    ma.o[j] = j < n ? o_parts[j] : nullptr;
    ma.lse[j] = j < n ? lse_parts[j] : nullptr;
  }
  // few partials: 16 elements per thread (more bytes in flight per thread); otherwise 8 (more warps per SM)
  const int ept = (d % 16 == 0 && n <= 3) ? 16 : 8;
  const int64_t total = (int64_t)batch * L * H * (d / ept);
  int64_t want = (total + 255) / 256;
  const int64_t cap = (int64_t)device_sm_count() * 16;
  int blocks = (int)(want < cap ? (want > 0 ? want : 1) : cap);
  bf16* oo = static_cast<bf16*>(o_out);
  auto go = [&](auto f32in, auto ept_c, auto np_c) {
    merge_kernel<decltype(f32in)::value, decltype(ept_c)::value, decltype(np_c)::value>
        <<<blocks, 256, 0, st>>>(ma, total, L, H, d, oo, lse_out);
  };
  auto by_np = [&](auto f32in, auto ept_c) {
    if (n <= 4) go(f32in, ept_c, std::integral_constant<int, 4>{});
    else if (n <= 8) go(f32in, ept_c, std::integral_constant<int, 8>{});
    else if (n <= 12) go(f32in, ept_c, std::integral_constant<int, 12>{});
    else go(f32in, ept_c, std::integral_constant<int, 16>{});
  };
  // (16 elements per thread only go with up to three partials, i.e. with four weights)
  if (dtype == 1) {
    if (ept == 16) go(std::true_type{}, std::integral_constant<int, 16>{}, std::integral_constant<int, 4>{});
    else by_np(std::true_type{}, std::integral_constant<int, 8>{});
  } else {
    if (ept == 16) go(std::false_type{}, std::integral_constant<int, 16>{}, std::integral_constant<int, 4>{});
    else by_np(std::false_type{}, std::integral_constant<int, 8>{});
  }
  return cudaGetLastError();
}

cudaError_t launch_bwd_prepare(const KArgs& a, float* dsum_clean, float* dsum_noisy, bool zero_dq, cudaStream_t st) {
  PrepArgs pa = {};
  float* out[2] = {dsum_clean, dsum_noisy};
  long long blocks[2] = {0, 0};
  pa.H = a.H;
  for (int s = 0; s < 2; ++s) {
    if (a.q[s] == nullptr) continue;   // a stream without queries has no D rows
    pa.dout[s] = a.dout[s]; pa.o[s] = a.o[s]; pa.dsum[s] = out[s];
    pa.dq32[s] = zero_dq ? a.dq32[s] : nullptr;
    pa.rows[s] = rows_q(a, s); pa.dq32_rows[s] = a.dq32_rows[s];
    blocks[s] = (long long)a.batch * ((pa.rows[s] + PREP_ROWS - 1) / PREP_ROWS) * ((a.H + PREP_HEADS - 1) / PREP_HEADS);
  }
  const long long n = blocks[0] + blocks[1];
  if (n == 0) return cudaSuccess;
  if (n > 0x7fffffffLL) return cudaErrorInvalidValue;
  pa.blocks_clean = (int)blocks[0];
  if (a.d == 128) bwd_prepare_kernel<128><<<(unsigned)n, 256, 0, st>>>(pa);
  else bwd_prepare_kernel<64><<<(unsigned)n, 256, 0, st>>>(pa);
  return cudaGetLastError();
}

}  // namespace bdlm
