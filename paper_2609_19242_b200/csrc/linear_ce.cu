// Token-chunked linear cross-entropy on the 5th-generation tensor cores (paper section 5, "Implementation and
// metrics": vocabulary projection + softmax cross-entropy without the logits of the whole sequence; the loss of
// Eq. bdlm-training-objective as a weighted sum of per-token negative log-likelihoods).
//
// One persistent, warp-specialised GEMM kernel C[M x N] = A . B with a contraction of K serves every matrix product
// of the path; what differs is where the operands lie and what the epilogue does with an accumulator tile:
//
//   forward            z = H W^T            epilogue: running row maximum and sum of exponentials, target logit
//   backward, chunk    z = H_c W^T          epilogue: dz = g w_t (exp(z - lse) - onehot) as bf16 into the workspace
//                      dH_c = dz W          epilogue: bf16 store
//                      dW  += dz^T H_c      epilogue: bf16 store, or fp32 accumulation over the chunks
//
// Tiles are 256 rows by at most 256 columns on a pair of CTAs, or 128 rows on one CTA (lce_rules.h), with 64-deep
// contraction steps: TMA (128-byte swizzle) fills a ring of A (16 KB) and B (up to 32 KB; of a pair each CTA loads half) tiles, one
// warp -- of a pair, that of rank 0 -- issues tcgen05.mma (M = 128 or 256, N = the tile's width, K = 16) into one of two
// 256-column accumulators in tensor memory, and four epilogue warps
// (one thread per accumulator row) drain the other one meanwhile.  An operand is either K-major (rows of the matrix = rows of
// the tile, contraction contiguous) or MN-major (rows of the matrix = contraction index, M/N contiguous; one 3-D load per tile
// where its 64-column panels are whole, a 64 x 64 box each otherwise), so W, H and dz are never transposed; W and H whose rows
// are no whole number of 128-byte lines are copied to padded rows first where that pays.  An element of a product is one
// accumulation over the whole contraction (dW: over a token chunk) whatever the tiling.
// CTAs are persistent: work items (an M tile x some N tiles) are dealt round-robin in an order that keeps the
// operand shared by concurrently running CTAs in L2.  Every wait is bounded and abortable.
#include <math.h>

#include "../../include/bdlm_linear_ce.h"
#include "lce_rules.h"
#include "tc_common.cuh"
#include "tc_launch.h"

namespace bdlm {
namespace {

using namespace tc;
using bf16 = __nv_bfloat16;

constexpr int A_BYTES = BM * BK * 2;
// PAIR: two CTAs work on a tile of 256 rows, 128 each, and each holds half of B's columns: a third less through L2 and shared
// memory per product, and the shorter stages make room for six.  The sums are the same bit for bit.  One CTA / pairs (us): 4096 x
// 2048 x 50304 forward 613 / 601, backward 2070 / 1869; 2194 x 2816 x 107056 977 / 950 and 3622 / 3236; 1531 x 1544 x 32008 171 /
// 158 and 494 / 465.  (MMAs of the pair run at the rate of one CTA's, 128 x 256 x 16 in 129 clk on each SM; what shrinks is the
// energy, at the power cap, and the load on L2.)
template <bool PAIR> struct Ring {
  static constexpr int B_BYTES = BN * BK * 2 / (PAIR ? 2 : 1), STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = PAIR ? 6 : 4;
  static constexpr int BARS = STAGES * STAGE_BYTES;
  static constexpr int SMEM = BARS + 256 + 1024;   // barriers, TMEM slot, abort flag; slack for 1024-byte alignment
};
constexpr int G_THREADS = 192;                   // warps 0-3 epilogue, warp 4 TMA, warp 5 MMA
constexpr int MN_PANEL = BK * 128;               // an MN-major panel: 64 contraction rows x 64 M/N elements

enum { EPI_LSE = 0, EPI_DZ = 1, EPI_STORE = 2, EPI_ADD = 3 };   // EPI_ADD: the two c_modes that read C first
enum { C_BF16 = 0, C_F32_STORE = 1, C_F32_ADD = 2, C_F32_ADD_TO_BF16 = 3 };

struct GemmMaps { CUtensorMap a, b; };
enum { K_MAJOR = 0, MN_PANELS = 1, MN_BOXES = 2 };

struct GemmArgs {
  int M, N, K;
  int bn;                                // width of an N tile: a multiple of 16 (of a pair 32), at most BN
  bool pair;                             // a tile of 256 rows per pair of CTAs
  int m_tiles, n_tiles, n_run, n_runs;   // an item = one M tile x n_run consecutive N tiles; n_runs = ceil(n_tiles / n_run)
  int m_inner;                           // item order: 1 = consecutive items share the N run, 0 = share the M tile
  int block;                             // and go through this many M tiles (N runs) before the next N run (M tile) begins
  int a_mn, b_mn;                        // operand layouts: K_MAJOR, MN_PANELS (one load per tile), MN_BOXES (one per 64-column panel)
  // EPI_LSE / EPI_DZ: rows are tokens row0 .. row0 + M - 1
  int row0;
  const int* labels;
  const float* weight;
  const float* lse;
  float grad;
  int run_tiles;   // N tiles per vocabulary run (a divisor of n_run)
  float* part_m;   // [vocabulary runs, ldp] running maxima (log2 units) per run
  float* part_l;   // [n_runs, ldp] sums of exponentials relative to that maximum
  float* zlab;     // [ldp] logit of the target
  int ldp;
  bf16* dz;        // EPI_DZ: [M, N] row-major, ld = ldz
  int ldz;
  // EPI_STORE
  int c_mode;
  bf16* c16; float* c32; int ldc;
};

// Loads issued by the elected lane of a converged warp (see elect_one).
__device__ __forceinline__ void tma_load_2d_e(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(elected) : "memory");
}
__device__ __forceinline__ void tma_load_panels_e(uint32_t dst, const CUtensorMap* map, uint32_t bar, int row, int panel, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {0, %3, %4}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(row), "r"(panel), "r"(elected) : "memory");
}

__device__ __forceinline__ void tma_load_2d_pair_e(uint32_t dst, const CUtensorMap* map, uint32_t peer_bar, int x, int y, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(peer_bar), "r"(x), "r"(y), "r"(elected) : "memory");
}
__device__ __forceinline__ void tma_load_panels_pair_e(uint32_t dst, const CUtensorMap* map, uint32_t peer_bar, int row, int panel, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {0, %3, %4}], [%2];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(peer_bar), "r"(row), "r"(panel), "r"(elected) : "memory");
}

// Walks the CTA's (or the pair's) tiles in the order every role uses.
struct TileWalk {
  int item, items, mt, nrun, nt, nt_end, stride;
  const GemmArgs* a;
  __device__ __forceinline__ void start(const GemmArgs& args, int first, int step) {
    a = &args; items = args.m_tiles * args.n_runs; item = first; stride = step; nt = 0; nt_end = 0;
    if (item < items) open();
  }
  __device__ __forceinline__ void open() {
    const int inner = a->m_inner ? a->m_tiles : a->n_runs, outer = a->m_inner ? a->n_runs : a->m_tiles;
    const int per_block = a->block * outer, blk = item / per_block, in_block = item - blk * per_block;
    const int width = min(a->block, inner - blk * a->block), o = in_block / width, i = blk * a->block + in_block - o * width;
    mt = a->m_inner ? i : o;
    nrun = a->m_inner ? o : i;
    nt = nrun * a->n_run;
    nt_end = min(a->n_tiles, nt + a->n_run);
  }
  __device__ __forceinline__ bool valid() const { return item < items; }
  __device__ __forceinline__ void next() {
    if (++nt < nt_end) return;
    item += stride;
    if (item < items) open();
  }
};

// Columns that the MMAs of a tile compute: the last tile of a row of tiles only those that the matrix has, in whole units of what
// the operand's layout allows (16 columns; of a pair 32, or a panel per CTA).  With D = 1544 the last of seven tiles is 8 wide.
template <bool PAIR>
__device__ __forceinline__ int mma_columns(const GemmArgs& a, int nt) {
  const int unit = PAIR ? (a.b_mn == K_MAJOR ? 32 : 128) : 16;
  return min(a.bn, (a.N - nt * a.bn + unit - 1) / unit * unit);
}

template <int EPI, bool PAIR>
__global__ void __launch_bounds__(G_THREADS, 1)
lce_gemm_kernel(const __grid_constant__ GemmMaps maps, const GemmArgs a, int* __restrict__ status) {
  constexpr int STAGES = Ring<PAIR>::STAGES, STAGE_BYTES = Ring<PAIR>::STAGE_BYTES, G_BARS = Ring<PAIR>::BARS;
  wait_for_predecessor();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;   // (the same in both CTAs of a pair)
  uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bars = base + G_BARS;
  // of a pair, full and acc_empty count in the CTA of rank 0, which issues for both; empty and acc_full are signalled to both
  const uint32_t bar_full = bars /*[STAGES]*/, bar_empty = bars + 8 * STAGES /*[STAGES]*/,
                 bar_acc_full = bars + 16 * STAGES /*[2]*/, bar_acc_empty = bars + 16 * STAGES + 16 /*[2]*/;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + G_BARS + 16 * STAGES + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + G_BARS + 16 * STAGES + 40);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = PAIR ? (int)cluster_rank() : 0;
  const int first = PAIR ? blockIdx.x >> 1 : blockIdx.x, step = PAIR ? gridDim.x >> 1 : gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar_acc_full + 8 * i, 1); mbar_init(bar_acc_empty + 8 * i, PAIR ? 8 : 128); }   // (of a pair: a warp each)
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 4) {
    if (PAIR) tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
    else tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();   // the other CTA's barriers and tensor memory are there
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const int nk = (a.K + BK - 1) / BK;

  if (warp == 4) {
    // ------------------------------------------------------------------ producer: the whole warp walks the loop, one
    // elected lane issues.  Issuing is what the products with MN-major operands were bound by (six 64-column boxes a
    // step, each from a lone lane): one load for all panels of a tile where the matrix allows it.
    const uint32_t el = elect_one();
    TileWalk w;
    w.start(a, first, step);
    int ks = 0;
    bool ok = true;
    const int bn_own = PAIR ? a.bn / 2 : a.bn;   // this CTA's columns of B
    const int stage_bytes = (A_BYTES + bn_own * BK * 2) * (PAIR ? 2 : 1);
    for (; w.valid() && ok; w.next()) {
      const int m0 = (PAIR ? 2 * w.mt + rank : w.mt) * BM, n0 = w.nt * a.bn + (PAIR ? rank * (mma_columns<PAIR>(a, w.nt) / 2) : 0);
      for (int k = 0; k < nk; ++k, ++ks) {
        const int s = ks % STAGES;
        if (ks >= STAGES) ok = mbar_wait_lean(bar_empty + 8 * s, ((ks / STAGES) - 1) & 1, abort_flag);
        if (!ok) break;
        const uint32_t sA = base + s * STAGE_BYTES, sB = sA + A_BYTES, bar = bar_full + 8 * s;
        if (el && rank == 0) mbar_expect_tx(bar, stage_bytes);
        if constexpr (PAIR) {
          const uint32_t pbar = peer_addr(bar, 0);
          if (a.a_mn == K_MAJOR) tma_load_2d_pair_e(sA, &maps.a, pbar, k * BK, m0, el);
          else if (a.a_mn == MN_PANELS) tma_load_panels_pair_e(sA, &maps.a, pbar, k * BK, m0 / 64, el);
          else {
#pragma unroll
            for (int p = 0; p < BM / 64; ++p) tma_load_2d_pair_e(sA + p * MN_PANEL, &maps.a, pbar, m0 + 64 * p, k * BK, el);
          }
          if (a.b_mn == K_MAJOR) tma_load_2d_pair_e(sB, &maps.b, pbar, k * BK, n0, el);
          else if (a.b_mn == MN_PANELS) tma_load_panels_pair_e(sB, &maps.b, pbar, k * BK, n0 / 64, el);
          else {
#pragma unroll
            for (int p = 0; p < BN / 128; ++p) if (64 * p < bn_own) tma_load_2d_pair_e(sB + p * MN_PANEL, &maps.b, pbar, n0 + 64 * p, k * BK, el);
          }
        } else {
          if (a.a_mn == K_MAJOR) tma_load_2d_e(sA, &maps.a, bar, k * BK, m0, el);
          else if (a.a_mn == MN_PANELS) tma_load_panels_e(sA, &maps.a, bar, k * BK, m0 / 64, el);
          else {
#pragma unroll
            for (int p = 0; p < BM / 64; ++p) tma_load_2d_e(sA + p * MN_PANEL, &maps.a, bar, m0 + 64 * p, k * BK, el);
          }
          if (a.b_mn == K_MAJOR) tma_load_2d_e(sB, &maps.b, bar, k * BK, n0, el);
          else if (a.b_mn == MN_PANELS) tma_load_panels_e(sB, &maps.b, bar, k * BK, n0 / 64, el);
          else {
#pragma unroll
            for (int p = 0; p < BN / 64; ++p) if (64 * p < a.bn) tma_load_2d_e(sB + p * MN_PANEL, &maps.b, bar, n0 + 64 * p, k * BK, el);
          }
        }
      }
    }
  } else if (warp == 5) {
    // ------------------------------------------------------------------ MMA issuer: the whole warp walks the loop,
    // one elected lane issues
    const uint32_t el = elect_one();
    const uint32_t a_lo0 = a.a_mn ? (((base & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(MN_PANEL >> 4) << 16)) : desc_lo_k(base);
    const uint32_t b_lo0 = a.b_mn ? ((((base + A_BYTES) & 0x3FFFFu) >> 4) | (static_cast<uint32_t>(MN_PANEL >> 4) << 16))
                                  : desc_lo_k(base + A_BYTES);
    const uint32_t a_step = a.a_mn ? 128u : 2u, b_step = a.b_mn ? 128u : 2u;   // low-word advance per 16-deep slice
    TileWalk w;
    w.start(a, first, step);
    int ks = 0, tcnt = 0;
    bool ok = true;
    for (; rank == 0 && w.valid() && ok; w.next(), ++tcnt) {
      const int buf = tcnt & 1;
      if (tcnt >= 2) {
        ok = mbar_wait_abortable(bar_acc_empty + 8 * buf, ((tcnt >> 1) - 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
      }
      const uint32_t d = tmem + buf * BN, idesc = make_idesc(PAIR ? 2 * BM : BM, mma_columns<PAIR>(a, w.nt), a.a_mn != 0, a.b_mn != 0);
      for (int k = 0; k < nk; ++k, ++ks) {
        const int s = ks % STAGES;
        ok = mbar_wait_lean(bar_full + 8 * s, (ks / STAGES) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t a_lo = a_lo0 + s * (STAGE_BYTES >> 4), b_lo = b_lo0 + s * (STAGE_BYTES >> 4);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          if (PAIR) mma_ss_pair_e(d, desc64(a_lo + kk * a_step), desc64(b_lo + kk * b_step), idesc, (k > 0 || kk > 0) ? 1u : 0u, el);
          else mma_ss_e(d, desc64(a_lo + kk * a_step), desc64(b_lo + kk * b_step), idesc, (k > 0 || kk > 0) ? 1u : 0u, el);
        if (PAIR) mma_commit_pair_e(bar_empty + 8 * s, el); else mma_commit_e(bar_empty + 8 * s, el);
      }
      if (!ok) break;
      if (PAIR) mma_commit_pair_e(bar_acc_full + 8 * buf, el); else mma_commit_e(bar_acc_full + 8 * buf, el);
    }
  } else {
    // ------------------------------------------------------------------ epilogue: one thread per accumulator row
    const int r = warp * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
    auto release = [&](int buf) {   // the accumulator's columns are read
      tc_fence_before();
      if (PAIR) {
        __syncwarp();
        if (lane == 0) mbar_arrive_peer(peer_addr(bar_acc_empty + 8 * buf, 0));
      } else {
        mbar_arrive(bar_acc_empty + 8 * buf);
      }
    };
    TileWalk w;
    w.start(a, first, step);
    int tcnt = 0;
    bool ok = true;
    // row state of the forward over a vocabulary run
    float run_m = -INFINITY, run_l = 0.f;
    for (; w.valid() && ok; w.next(), ++tcnt) {
      const int buf = tcnt & 1;
      const int m0 = (PAIR ? 2 * w.mt + rank : w.mt) * BM, n0 = w.nt * a.bn;
      const int row = m0 + r;
      const bool row_ok = row < a.M;
      const int ncols = min(a.bn, a.N - n0);        // valid columns of this tile (a multiple of 8)
      int y = -1;
      float coef = 0.f, lse2 = 0.f;
      if ((EPI == EPI_LSE || EPI == EPI_DZ) && row_ok) {
        y = a.labels[a.row0 + row];
        if (EPI == EPI_DZ) {
          const float wt = a.weight != nullptr ? a.weight[a.row0 + row] : 1.f;
          coef = y >= 0 ? a.grad * wt : 0.f;
          lse2 = a.lse[a.row0 + row] * LOG2E;
        }
      }
      if (EPI == EPI_LSE && w.nt % a.run_tiles == 0) { run_m = -INFINITY; run_l = 0.f; }
      if (EPI == EPI_ADD) {
        // The fp32 sums of the earlier token chunks are requested two 32-column chunks ahead, the first ones before the
        // wait for the accumulator: requested where they are used, their round trips to memory took longer than the
        // tile's MMAs.
        const float* src = a.c32 + (int64_t)row * a.ldc + n0;
        float4 pre[2][8];
        auto request = [&](int c, float4 (&u)[8]) {
#pragma unroll
          for (int q = 0; q < 8; ++q) if (row_ok && c * 32 + q * 4 < ncols) u[q] = __ldcs(reinterpret_cast<const float4*>(src + c * 32) + q);
        };
        auto finish = [&](int c, float4 (&u)[8]) {
          uint32_t x[32];
          tmem_ld32(tl + buf * BN + c * 32, x);
          tmem_wait_ld();
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            u[q].x += __uint_as_float(x[4 * q]); u[q].y += __uint_as_float(x[4 * q + 1]);
            u[q].z += __uint_as_float(x[4 * q + 2]); u[q].w += __uint_as_float(x[4 * q + 3]);
          }
          if (!row_ok) return;
          const int64_t off = (int64_t)row * a.ldc + n0 + c * 32;
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            if (c * 32 + q * 4 < ncols) {
              if (a.c_mode == C_F32_ADD) {
                *reinterpret_cast<float4*>(a.c32 + off + q * 4) = u[q];
                *reinterpret_cast<float4*>(a.c32 + off + q * 4 + 4) = u[q + 1];
              } else {
                *reinterpret_cast<uint4*>(a.c16 + off + q * 4) =
                    make_uint4(pack_bf16(u[q].x, u[q].y), pack_bf16(u[q].z, u[q].w), pack_bf16(u[q + 1].x, u[q + 1].y), pack_bf16(u[q + 1].z, u[q + 1].w));
              }
            }
          }
        };
        request(0, pre[0]);
        request(1, pre[1]);
        ok = mbar_wait_abortable(bar_acc_full + 8 * buf, (tcnt >> 1) & 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < BN / 32; c += 2) {   // (columns past the tile are read from tensor memory and dropped)
          finish(c, pre[0]);
          request(c + 2, pre[0]);
          finish(c + 1, pre[1]);
          request(c + 3, pre[1]);
        }
        release(buf);
        continue;
      }
      ok = mbar_wait_abortable(bar_acc_full + 8 * buf, (tcnt >> 1) & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < (a.bn + 31) / 32; ++c) {
        uint32_t x[32];
        tmem_ld32(tl + buf * BN + c * 32, x);
        tmem_wait_ld();
        const int col0 = n0 + c * 32;
        const int cvalid = ncols - c * 32;           // columns of this chunk inside the matrix (may be <= 0 or >= 32)
        // (no `continue` below: the tensor-memory loads are warp-collective, every lane takes every iteration)
        if (EPI == EPI_LSE && cvalid > 0) {
          if (cvalid < 32) {
#pragma unroll
            for (int e = 0; e < 32; ++e) if (e >= cvalid) x[e] = 0xff800000u;   // -inf beyond the vocabulary
          }
          float mx = -INFINITY;
#pragma unroll
          for (int e = 0; e < 32; ++e) mx = fmaxf(mx, __uint_as_float(x[e]));
          mx *= LOG2E;
          if (mx > run_m) { run_l *= exp2f(run_m - mx); run_m = mx; }
          const float mb = run_m == -INFINITY ? 0.f : run_m;   // (nothing but -inf so far: the sum is 0, not NaN)
          const uint64_t c2 = pack_f32x2(LOG2E, LOG2E), m2 = pack_f32x2(-mb, -mb);
          uint64_t s2 = 0;
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            float u, v;
            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(x[e]), __uint_as_float(x[e + 1])), c2, m2), u, v);
            s2 = add_f32x2(s2, pack_f32x2(exp2f(u), exp2f(v)));
          }
          float s0, s1;
          unpack_f32x2(s2, s0, s1);
          run_l += s0 + s1;
          if ((unsigned)(y - col0) < (unsigned)min(cvalid, 32)) {   // (a chunk may reach into the next tile's columns)
            float z = 0.f;
#pragma unroll
            for (int e = 0; e < 32; ++e) if (col0 + e == y) z = __uint_as_float(x[e]);
            a.zlab[a.row0 + row] = z;
          }
        } else if (EPI == EPI_DZ && cvalid > 0 && row_ok) {
          float p[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) p[e] = coef * exp2f(fmaf(__uint_as_float(x[e]), LOG2E, -lse2));
          if ((unsigned)(y - col0) < 32u) {
#pragma unroll
            for (int e = 0; e < 32; ++e) if (col0 + e == y) p[e] -= coef;
          }
          bf16* dst = a.dz + (int64_t)row * a.ldz + col0;
#pragma unroll
          for (int e8 = 0; e8 < 4; ++e8) {
            if (e8 * 8 < cvalid) {
              uint4 v;
              v.x = pack_bf16(p[e8 * 8 + 0], p[e8 * 8 + 1]); v.y = pack_bf16(p[e8 * 8 + 2], p[e8 * 8 + 3]);
              v.z = pack_bf16(p[e8 * 8 + 4], p[e8 * 8 + 5]); v.w = pack_bf16(p[e8 * 8 + 6], p[e8 * 8 + 7]);
              *reinterpret_cast<uint4*>(dst + e8 * 8) = v;
            }
          }
        } else if (EPI == EPI_STORE && cvalid > 0 && row_ok) {
          const int64_t off = (int64_t)row * a.ldc + col0;
#pragma unroll
          for (int e8 = 0; e8 < 4; ++e8) {
            if (e8 * 8 >= cvalid) break;
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(x[e8 * 8 + e]);
            if (a.c_mode != C_BF16) {
              *reinterpret_cast<float4*>(a.c32 + off + e8 * 8) = make_float4(v[0], v[1], v[2], v[3]);
              *reinterpret_cast<float4*>(a.c32 + off + e8 * 8 + 4) = make_float4(v[4], v[5], v[6], v[7]);
            } else {
              uint4 o;
              o.x = pack_bf16(v[0], v[1]); o.y = pack_bf16(v[2], v[3]); o.z = pack_bf16(v[4], v[5]); o.w = pack_bf16(v[6], v[7]);
              *reinterpret_cast<uint4*>(a.c16 + off + e8 * 8) = o;
            }
          }
        }
      }
      release(buf);
      if (EPI == EPI_LSE && ((w.nt + 1) % a.run_tiles == 0 || w.nt + 1 == a.n_tiles) && row_ok) {
        const int64_t at = (int64_t)(w.nt / a.run_tiles) * a.ldp + a.row0 + row;
        a.part_m[at] = run_m;
        a.part_l[at] = run_l;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    if (PAIR) give_up_pair(abort_flag, status, rank); else atomicExch(status, (int)BDLM_ERR_DEVICE_TIMEOUT);
  }
  if (PAIR) cluster_sync();   // no CTA leaves while the other one still signals its barriers or reads its operands
  if (warp == 4) {
    if (PAIR) tmem_dealloc_pair(tmem, 512); else tmem_dealloc(tmem, 512);
  }
}

// Combines the per-run partial (maximum, sum) pairs of every token (Eq. csbp-lse-merge's rule, in log2 units),
// writes lse and nll, and leaves one weighted partial sum of the loss per block (fixed order: reproducible).
// A block takes FIN_T tokens, eight threads share a token's runs (one thread per token left a few blocks alone with a
// hundred dependent rounds of loads when the runs are short).  A maximum of -inf is left by no run at all (sum 0) and by a run
// of NaN (sum NaN; maxima pass NaN over): both go into the sum with weight 0, so NaN stays.  The block's sum replaces its own
// first token's first partial maximum, which nobody else reads.
constexpr int FIN_T = 32;
__global__ void __launch_bounds__(256) lce_finish_kernel(float* part_m, const float* part_l,
                                                         const float* zlab, const int* __restrict__ labels,
                                                         const float* __restrict__ weight, int T, int n_runs, int ldp,
                                                         float* __restrict__ lse, float* __restrict__ nll) {
  __shared__ float sm_m[8][FIN_T], sm_l[8][FIN_T];
  wait_for_predecessor();
  const int x = threadIdx.x % FIN_T, y0 = threadIdx.x / FIN_T;
  const int t = blockIdx.x * FIN_T + x;
  float m = -INFINITY, l = 0.f;
  if (t < T) {
#pragma unroll 8
    for (int c = y0; c < n_runs; c += 8) m = fmaxf(m, part_m[(int64_t)c * ldp + t]);
    const float mb = m == -INFINITY ? 0.f : m;
#pragma unroll 8
    for (int c = y0; c < n_runs; c += 8) l += part_l[(int64_t)c * ldp + t] * exp2f(part_m[(int64_t)c * ldp + t] - mb);
  }
  sm_m[y0][x] = m; sm_l[y0][x] = l;
  __syncthreads();
  if (threadIdx.x >= FIN_T) return;
  float contrib = 0.f;
  if (t < T) {
    m = -INFINITY; l = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) m = fmaxf(m, sm_m[j][x]);
    const float mb = m == -INFINITY ? 0.f : m;
#pragma unroll
    for (int j = 0; j < 8; ++j) l += sm_l[j][x] * exp2f(sm_m[j][x] - mb);
    const float z = (m + log2f(l)) * LN2;
    const int y = labels[t];
    const float n = y >= 0 ? z - zlab[t] : 0.f;
    lse[t] = z;
    if (nll != nullptr) nll[t] = n;
    contrib = (weight != nullptr ? weight[t] : 1.f) * n;
  }
#pragma unroll
  for (int sft = FIN_T / 2; sft > 0; sft >>= 1) contrib += __shfl_xor_sync(0xffffffffu, contrib, sft);
  if (x == 0) part_m[blockIdx.x * FIN_T] = contrib;
}

__global__ void __launch_bounds__(256) lce_sum_kernel(const float* block_sums, int n, int stride, float* loss) {
  __shared__ float red[256];
  wait_for_predecessor();
  float acc = 0.f;
  for (int i = threadIdx.x; i < n; i += 256) acc += block_sums[i * stride];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = red[0];
}

// Copies W [V, D] and the tokens' h [T, D] to rows of `ld` elements (a whole number of 128-byte lines), 16 bytes per thread and
// turn; what lies past a row's D elements is never looked at.
__global__ void __launch_bounds__(256) lce_pack_kernel(const uint4* __restrict__ w, uint4* __restrict__ w_out, unsigned nw,
                                                       const uint4* __restrict__ h, uint4* __restrict__ h_out, unsigned nh,
                                                       unsigned per_row, unsigned per_row_out) {
  constexpr int U = 4;
  wait_for_predecessor();
  for (unsigned i0 = blockIdx.x * 256 * U + threadIdx.x; i0 < nw + nh; i0 += gridDim.x * 256 * U) {
    uint4 v[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const unsigned i = i0 + j * 256;
      if (i < nw) v[j] = __ldcs(w + i);
      else if (i < nw + nh) v[j] = h[i - nw];
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      unsigned i = i0 + j * 256;
      if (i >= nw + nh) break;
      uint4* dst = w_out;
      if (i >= nw) { i -= nw; dst = h_out; }
      const unsigned row = i / per_row;
      dst[(size_t)row * per_row_out + (i - row * per_row)] = v[j];
    }
  }
}

// ------------------------------------------------------------------------------------------ host
// Operand descriptions of one product: A is [M x K] (K-major) or [K x M] (MN-major) in memory, B likewise with N.
// whole: rows may be read up to the next multiple of 64 elements (a copy of our own).
struct Operand { const void* ptr; int64_t ld; int mn; bool whole; };

// How many tiles of the dimension that items walk first lie together before the other one advances: as many as keep
// their operand in L2 (126 MB, in two halves) while the other operand streams past; where a few tiles' worth is too much (dH: a
// contraction over the vocabulary), the block that lets the CTAs running together read the least of both operands.  All of them
// / blocks: T = 12288, D = 4096 (h 100 MB), V = 64000 forward 5270 / 4560 us; T = 8192, D = 4096, V = 128256 forward 6425 /
// 6000 (h 67 MB), backward 19800 / 19500; smaller ones have one block.
constexpr double L2_KEEP = 40e6;
int inner_block(const GemmArgs& a) {
  const int rows = a.pair ? 2 * BM : BM, slots = device_sm_count() / (a.pair ? 2 : 1);
  const int inner = a.m_inner ? a.m_tiles : a.n_runs;
  const double in_elems = a.m_inner ? rows : (double)a.bn * a.n_run, out_elems = a.m_inner ? (double)a.bn : rows;
  const double fit = L2_KEEP / (in_elems * a.K * 2), even = sqrt(slots * out_elems / in_elems);
  const int most = (int)(fit > even ? fit : even);
  if (inner <= most || most < 1) return inner;
  const int blocks = (inner + most - 1) / most;
  return (inner + blocks - 1) / blocks;
}

template <int EPI>
cudaError_t launch_gemm(GemmArgs a, const Operand& A, const Operand& B, cudaStream_t st, bool chained) {
  GemmMaps maps;
  auto encode = [&](CUtensorMap* m, const Operand& o, int extent, int box, int& layout) {
    if (!o.mn) { layout = K_MAJOR; return tc_make_map_2d(m, o.ptr, extent, a.K, o.ld, box); }
    if (o.whole) extent = (extent + 63) / 64 * 64;
    layout = extent % 64 == 0 ? MN_PANELS : MN_BOXES;   // (a last panel that is not whole would reach past the matrix)
    return layout == MN_PANELS ? tc_make_map_panels(m, o.ptr, a.K, extent, o.ld, BK, box / 64) : tc_make_map_2d(m, o.ptr, a.K, extent, o.ld, 64);
  };
  const bool okA = encode(&maps.a, A, a.M, BM, a.a_mn), okB = encode(&maps.b, B, a.N, a.pair ? a.bn / 2 : a.bn, a.b_mn);
  if (!okA || !okB) return cudaErrorInvalidValue;
  const int tile_rows = a.pair ? 2 * BM : BM, ctas = a.pair ? 2 : 1;
  a.m_tiles = (a.M + tile_rows - 1) / tile_rows;
  a.n_tiles = (a.N + a.bn - 1) / a.bn;
  a.n_runs = (a.n_tiles + a.n_run - 1) / a.n_run;
  int* status = device_status_ptr();
  if (status == nullptr) return cudaErrorUnknown;
  auto kern = a.pair ? lce_gemm_kernel<EPI, true> : lce_gemm_kernel<EPI, false>;
  const int smem = a.pair ? Ring<true>::SMEM : Ring<false>::SMEM;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  a.block = inner_block(a);
  const int items = a.m_tiles * a.n_runs, slots = device_sm_count() / ctas;
  const int grid = (items < slots ? items : slots) * ctas;
  return launch_chained(kern, chained, grid, G_THREADS, smem, st, ctas, maps, a, status);
}

// The forward's sums of exponentials: one running (maximum, sum) pair per token and vocabulary run, then the runs' pairs
// together (lce_finish_kernel).  Where a run ends depends on nothing but the workspace, so that a token's lse is the same bit
// for bit whatever other tokens are in the call; how many runs go into a work item is for the tiling to choose.  A run of one
// tile leaves that choice free (T = 1531, D = 1544, V = 32008: forward 196 us, with 2048 logits a run 237; T = 149, D = 224,
// V = 50912: 30 and 39) and costs 8 bytes written and read per token and 256 logits, which does not show (8192 x 4096 x
// 128256: 6.35 and 6.42 ms, inside the noise).  The smallest workspace that is accepted holds the pairs of runs of eight tiles.
constexpr int RUN_TILES = 1, RUN_TILES_LEAST = 8;

int fwd_runs(int V, int run_tiles) { return ((V + BN - 1) / BN + run_tiles - 1) / run_tiles; }
size_t align256(size_t x) { return (x + 255) / 256 * 256; }
size_t fwd_part_bytes(const bdlm_lce_params* p, int run_tiles) {
  const size_t per = align256((size_t)p->T * sizeof(float));
  return (2 * (size_t)fwd_runs(p->V, run_tiles) + 1) * per;
}
// Matrices whose rows are no whole number of 128-byte lines: every 128-byte row of a TMA box then straddles two lines,
// and the products, which live on L2 bandwidth, take half as long again or more (T = 1531, V ~ 32000: D = 1536 against
// 1544 forward 103 / 160 us, backward 346 / 600).  From PACK_*_T tokens on, W and h are copied to padded rows first
// (W of 98 MB: 35 us); the rows of dz, which is ours, are padded in any case.  Without and with the copies at D = 1544, V = 32008
// (us): forward T = 768 109 / 117, 1024 123 / 124, 1280 156 / 144; backward T = 128 225 / 233, 256 246 / 246, 384 278 / 265,
// 768 358 / 316.  Where the matrices are small (D = 264, V = 8008) the forward's copies cost 3 us at 1024 tokens.
constexpr int PACK_FWD_T = 1024, PACK_BWD_T = 384;
int64_t up64(int64_t x) { return (x + 63) / 64 * 64; }
bool packs(const bdlm_lce_params* p, int from) { return p->D % 64 != 0 && p->T >= from && ((int64_t)p->V + p->T) * (p->D / 8) < (1ll << 31); }
size_t pack_w_bytes(const bdlm_lce_params* p) { return align256((size_t)p->V * up64(p->D) * 2); }
size_t pack_bytes(const bdlm_lce_params* p) { return pack_w_bytes(p) + align256((size_t)p->T * up64(p->D) * 2); }
// Copies both to `at`; h and w become the copies.
cudaError_t pack(const bdlm_lce_params* p, char* at, Operand& h, Operand& w, cudaStream_t st) {
  const unsigned per_row = p->D / 8, nw = (unsigned)p->V * per_row, nh = (unsigned)p->T * per_row;
  uint4 *w_out = reinterpret_cast<uint4*>(at), *h_out = reinterpret_cast<uint4*>(at + pack_w_bytes(p));
  const unsigned want = (nw + nh + 1023) / 1024, cap = device_sm_count() * 8;
  lce_pack_kernel<<<want < cap ? want : cap, 256, 0, st>>>(static_cast<const uint4*>(w.ptr), w_out, nw, static_cast<const uint4*>(h.ptr), h_out, nh,
                                                           per_row, (unsigned)(up64(p->D) / 8));
  w = Operand{w_out, up64(p->D), 0, true};
  h = Operand{h_out, up64(p->D), 0, true};
  return cudaGetLastError();
}
size_t fwd_bytes(const bdlm_lce_params* p) { return fwd_part_bytes(p, RUN_TILES) + (packs(p, PACK_FWD_T) ? pack_bytes(p) : 0); }
// the smallest workspace that is accepted (with room for loss sums that now lie elsewhere: the size is an old promise)
size_t fwd_bytes_min(const bdlm_lce_params* p) {
  return fwd_part_bytes(p, RUN_TILES_LEAST) + align256(((size_t)p->T + 255) / 256 * sizeof(float));
}
int default_chunk(const bdlm_lce_params* p) {
  if (p->token_chunk > 0) return p->token_chunk;
  const int up = (p->T + 127) / 128 * 128;
  return up < 4096 ? up : 4096;
}
// The backward's workspace: dz of a chunk, the fp32 dW with several chunks, the copies of W and h.  The smallest that is
// accepted has the first two only, dz with rows of V elements.
// dH = dz W is one accumulation per element over the whole vocabulary, whatever the tile or the number of tokens, so that a
// token's dH is the same bit for bit in every call it is part of.  (Cut into pieces where its tiles do not fill the chip --
// T = 1531, D = 1544, V = 32008: 84 tiles -- forward and backward together took 674 us instead of 690, but a token's dH then
// depended on how many others there were: 3.5e-4 of its norm.)
struct BwdPlan { int64_t ldz; bool packed; size_t dw32, copies, bytes; };
BwdPlan bwd_plan(const bdlm_lce_params* p, bool least) {
  const int tc_ = default_chunk(p), chunks = (p->T + tc_ - 1) / tc_;
  BwdPlan b;
  b.ldz = least ? p->V : up64(p->V);
  b.packed = !least && packs(p, PACK_BWD_T);
  b.dw32 = align256((size_t)tc_ * b.ldz * 2);
  b.copies = b.dw32 + (chunks > 1 ? align256((size_t)p->V * p->D * sizeof(float)) : 0);
  b.bytes = b.copies + (b.packed ? pack_bytes(p) : 0);
  return b;
}

int check(const bdlm_lce_params* p) {
  if (p == nullptr) return BDLM_ERR_INVALID_ARG;
  if (p->T <= 0 || p->D <= 0 || p->V <= 0 || p->D % 8 != 0 || p->V % 8 != 0) return BDLM_ERR_INVALID_ARG;
  if (p->token_chunk < 0 || p->token_chunk % 128 != 0) return BDLM_ERR_INVALID_ARG;
  if (!(p->grad_loss == p->grad_loss) || isinf(p->grad_loss)) return BDLM_ERR_INVALID_ARG;
  return BDLM_OK;
}
bool al16(const void* x) { return (reinterpret_cast<uintptr_t>(x) & 15u) == 0; }
bool sm100() {
  int dev = 0, major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return false;
  return major == 10;
}

}  // namespace
}  // namespace bdlm

using namespace bdlm;

extern "C" {

size_t bdlm_linear_ce_workspace_bytes(const bdlm_lce_params* p, int32_t which) {
  if (check(p) != BDLM_OK) return 0;
  if (which == BDLM_LCE_WS_FWD) {
    const size_t full = fwd_bytes(p), least = fwd_bytes_min(p);
    return full > least ? full : least;
  }
  if (which == BDLM_LCE_WS_BWD) return bwd_plan(p, false).bytes;
  if (which == BDLM_LCE_WS_FWD_LEAST) return fwd_bytes_min(p);
  if (which == BDLM_LCE_WS_BWD_LEAST) return bwd_plan(p, true).bytes;
  return 0;
}

int bdlm_linear_ce_fwd(const bdlm_lce_params* p, const void* h, const void* w, const int32_t* labels,
                       const float* token_weight, float* loss, float* nll, float* lse,
                       void* workspace, size_t workspace_bytes, void* cuda_stream) {
  int rc = check(p);
  if (rc != BDLM_OK) return rc;
  const void* need[] = {h, w, labels, loss, lse, workspace};
  for (const void* x : need) if (x == nullptr) return BDLM_ERR_INVALID_ARG;
  if (!al16(h) || !al16(w) || !al16(workspace) || (reinterpret_cast<uintptr_t>(labels) & 3u) ||
      (reinterpret_cast<uintptr_t>(loss) & 3u) || (reinterpret_cast<uintptr_t>(lse) & 3u) ||
      (reinterpret_cast<uintptr_t>(nll) & 3u) || (reinterpret_cast<uintptr_t>(token_weight) & 3u))
    return BDLM_ERR_INVALID_ARG;
  if (workspace_bytes < fwd_bytes_min(p)) return BDLM_ERR_WORKSPACE_TOO_SMALL;
  if (!sm100() || !tc_encoder_available()) return BDLM_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const bool roomy = workspace_bytes >= fwd_bytes(p);
  const int run_tiles = roomy ? RUN_TILES : RUN_TILES_LEAST, runs = fwd_runs(p->V, run_tiles);
  const size_t per = align256((size_t)p->T * sizeof(float));
  char* ws = static_cast<char*>(workspace);
  GemmArgs a = {};
  a.M = p->T; a.N = p->V; a.K = p->D; a.m_inner = 1; a.run_tiles = run_tiles;
  const Tiling ta = forward_tiling(device_sm_count(), p->T, p->D, p->V, run_tiles);
  a.bn = BN; a.n_run = ta.n_run; a.pair = ta.pair;
  a.row0 = 0; a.labels = labels; a.weight = token_weight; a.ldp = (int)(per / sizeof(float));
  a.part_m = reinterpret_cast<float*>(ws);
  a.part_l = reinterpret_cast<float*>(ws + (size_t)runs * per);
  a.zlab = reinterpret_cast<float*>(ws + 2 * (size_t)runs * per);
  Operand oh{h, p->D, 0, false}, ow{w, p->D, 0, false};
  const bool packed = roomy && packs(p, PACK_FWD_T);
  if (packed && pack(p, ws + fwd_part_bytes(p, run_tiles), oh, ow, st) != cudaSuccess) return BDLM_ERR_CUDA;
  if (launch_gemm<EPI_LSE>(a, oh, ow, st, packed) != cudaSuccess) return BDLM_ERR_CUDA;
  const int blocks = (p->T + FIN_T - 1) / FIN_T;
  if (launch_chained(lce_finish_kernel, true, blocks, 256, 0, st, 1, a.part_m, a.part_l, a.zlab, labels, token_weight, p->T, runs, a.ldp, lse, nll) != cudaSuccess)
    return BDLM_ERR_CUDA;
  return launch_chained(lce_sum_kernel, true, 1, 256, 0, st, 1, a.part_m, blocks, FIN_T, loss) == cudaSuccess ? BDLM_OK : BDLM_ERR_CUDA;
}

int bdlm_linear_ce_bwd(const bdlm_lce_params* p, const void* h, const void* w, const int32_t* labels,
                       const float* token_weight, const float* lse, void* dh, void* dw,
                       void* workspace, size_t workspace_bytes, void* cuda_stream) {
  int rc = check(p);
  if (rc != BDLM_OK) return rc;
  const void* need[] = {h, w, labels, lse, dh, dw, workspace};
  for (const void* x : need) if (x == nullptr) return BDLM_ERR_INVALID_ARG;
  if (!al16(h) || !al16(w) || !al16(dh) || !al16(dw) || !al16(workspace) || (reinterpret_cast<uintptr_t>(labels) & 3u) ||
      (reinterpret_cast<uintptr_t>(lse) & 3u) || (reinterpret_cast<uintptr_t>(token_weight) & 3u))
    return BDLM_ERR_INVALID_ARG;
  const bool roomy = workspace_bytes >= bwd_plan(p, false).bytes;
  const BwdPlan plan = bwd_plan(p, !roomy);
  if (workspace_bytes < plan.bytes) return BDLM_ERR_WORKSPACE_TOO_SMALL;
  if (!sm100() || !tc_encoder_available()) return BDLM_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int T = p->T, D = p->D, V = p->V;
  const int tc_ = default_chunk(p);
  const int chunks = (T + tc_ - 1) / tc_;
  char* ws = static_cast<char*>(workspace);
  bf16* dz = static_cast<bf16*>(workspace);
  const int64_t ldz = plan.ldz;
  float* dw32 = reinterpret_cast<float*>(ws + plan.dw32);
  Operand oh{h, D, 0, false}, ow{w, D, 0, false};
  if (plan.packed && pack(p, ws + plan.copies, oh, ow, st) != cudaSuccess) return BDLM_ERR_CUDA;
  auto mn = [](Operand o) { o.mn = 1; return o; };
  for (int ci = 0; ci < chunks; ++ci) {
    const int t0 = ci * tc_, rows = (T - t0) < tc_ ? (T - t0) : tc_;
    Operand oh_c = oh;
    oh_c.ptr = static_cast<const bf16*>(oh.ptr) + (size_t)t0 * oh.ld;
    const Operand odz{dz, ldz, 0, roomy};
    // dz of the chunk: logits again, softmax minus one-hot in the epilogue
    GemmArgs a = {};
    const Tiling ta = choose_tiling(device_sm_count(), rows, V, D, 128, 1, MAX_RUN, EPI_CLK_DZ, 0);
    a.M = rows; a.N = V; a.K = D; a.bn = ta.bn; a.n_run = ta.n_run; a.pair = ta.pair; a.m_inner = 1;
    a.row0 = t0; a.labels = labels; a.weight = token_weight; a.lse = lse; a.grad = p->grad_loss;
    a.dz = dz; a.ldz = (int)ldz;
    if (launch_gemm<EPI_DZ>(a, oh_c, ow, st, ci > 0 || plan.packed) != cudaSuccess) return BDLM_ERR_CUDA;
    // dH of the chunk = dz W   (contraction over the vocabulary; W as it lies is the MN-major B operand)
    GemmArgs b = {};
    const Tiling tb = choose_tiling(device_sm_count(), rows, D, V, 64, 1, 1, EPI_CLK_STORE, 1);
    b.M = rows; b.N = D; b.K = V; b.bn = tb.bn; b.n_run = 1; b.pair = tb.pair; b.m_inner = 1;
    b.c_mode = C_BF16; b.c16 = static_cast<bf16*>(dh) + (size_t)t0 * D; b.ldc = D;
    if (launch_gemm<EPI_STORE>(b, odz, mn(ow), st, true) != cudaSuccess) return BDLM_ERR_CUDA;
    // dW += dz^T H_c   (contraction over the chunk's tokens; both operands MN-major)
    GemmArgs c = {};
    const Tiling tw = choose_tiling(device_sm_count(), V, D, rows, 128, 1, 1, EPI_CLK_STORE, 1);
    c.M = V; c.N = D; c.K = rows; c.bn = tw.bn; c.n_run = 1; c.pair = tw.pair; c.m_inner = 0;
    c.c16 = static_cast<bf16*>(dw); c.c32 = dw32; c.ldc = D;
    c.c_mode = chunks == 1 ? C_BF16 : (ci == 0 ? C_F32_STORE : (ci + 1 < chunks ? C_F32_ADD : C_F32_ADD_TO_BF16));
    const Operand A = mn(odz), B = mn(oh_c);
    const bool adds = c.c_mode == C_F32_ADD || c.c_mode == C_F32_ADD_TO_BF16;
    if ((adds ? launch_gemm<EPI_ADD>(c, A, B, st, true) : launch_gemm<EPI_STORE>(c, A, B, st, true)) != cudaSuccess) return BDLM_ERR_CUDA;
  }
  return BDLM_OK;
}

}  // extern "C"
