// Backward on pairs of CTAs for head dimension 128: dK, dV and dQ in one kernel (or dK and dV alone, see DQ).
//
// A unit is two neighbouring 128-key tiles of one KV head, one per CTA of a cluster of two; the pair walks every 128-row query
// tile that sees either of them (all heads of the group, clean then noisy queries).  Every product is one tcgen05.mma of the
// pair (cta_group::2), issued by the CTA of rank 0:
//   S^T = K Q^T, dP^T = V dO^T     M = 256 keys, N = 128 queries; each CTA holds 64 of the query rows of Q and dO
//   dV += P^T dO, dK += dS^T Q     M = 256 keys, N = 128; each CTA holds 64 of the head dimension's columns; A in tensor memory
//   dQ^T = K^T dS^T                M = 128 (head dimension, 64 per CTA), N = 128 queries, contraction over the 256 keys
// dQ^T is what the pair is for: its sum runs over both key tiles before it leaves the SM, so half as many bytes go through the
// fp32 reductions into the dQ accumulators per product (4 of the 41 ms that the one-CTA kernel takes at 32K, H = 32 / 8, are
// these reductions), and every product reads half of its B operand from shared memory.  Each CTA holds K^T of both tiles for
// its half of the head dimension and dS^T of both tiles for its half of the queries.
//   tensor memory  [0,128) S^T; P^T as bf16 pairs at [0,32) and [64,96)   [128,256) dP^T; dS^T as bf16 pairs at [128,192),
//                  dQ^T at [192,256)   [256,384) dV   [384,512) dK
//   shared memory  K, V, K^T of both tiles, dS^T (32 KB each), three 16 KB operand buffers, the half of dS^T on its way to the
//                  other CTA (16 KB), dQ staging (2 x 16 KB)
// The order of the products in step i: dV(i), S^T(i+1), dQ^T(i-1), dK(i), dP^T(i+1).  dQ^T runs a step late, over columns of
// dP^T(i) that the compute warps have read by then, so that dS^T has a step's time to get to the other CTA.
//   compute      exponentials, then dS = P (dP - D), 64 query columns of a key row per thread; dS^T goes to tensor memory,
//                where dK reads it
//   move         four warps copy dS^T from tensor memory to shared memory; what the other CTA needs goes on from there as bulk
//                copies (stores straight into the other CTA's shared memory took 2500 clk a step)
//   read-out     four warps take dQ^T to two staging tiles, one reduction each
// Against the one-CTA kernel: 3340 clk per 128 x 128 tile pair instead of 3700; 32K, H = 32 / 8 (at the power cap) 40.8 ->
// 37.8 ms for the whole backward, 2 x 8K, H = 16 / 4 2.98 -> 2.85 ms.  What bounds a step: the chain dV(i), S^T(i+1), exponentials
// (1024 + 1700 clk and the signals between them) and, at the power cap, energy.  Handing P^T over in halves was slower (two more
// waits of the issuing warp; 38.2 ms), so were read-out tiles of 32 queries and dS^T stored by the compute warps (40.4 ms).
// The accumulators of dQ lie in blocks of 64 rows, each as two [64 rows x 64] halves of the head dimension.
#include <type_traits>

#include "tc_bwd_common.cuh"

namespace bdlm {
namespace {

using namespace tc;

struct PairMaps {
  CUtensorMap q[2], dout[2];     // boxes of 64 rows: this CTA's rows of a query tile
  CUtensorMap qc[2], doutc[2];   // boxes of 128 rows: its columns
  CUtensorMap k[2], v[2];
  CUtensorMap dk[2], dv[2];      // boxes of 32 rows: what a warp stores
};

constexpr int D = 128;
constexpr int HT = 64;
constexpr int HPANEL_BYTES = HT * 128;
constexpr int BP_K = 0, BP_V = TILE_BYTES, BP_KT = 2 * TILE_BYTES, BP_DS = 3 * TILE_BYTES;
constexpr int BP_OPER = 4 * TILE_BYTES;             // three 16 KB buffers for Q and dO by rows and by columns, in turn
constexpr int BP_SEND = BP_OPER + 3 * PANEL_BYTES;  // the half of dS^T that the other CTA needs, on its way there
constexpr int BP_STG = BP_SEND + PANEL_BYTES;
constexpr int STG_BYTES = HT * HT * 4;              // [64 queries x 64] fp32, one per half of the queries
// The products read Q and dO in the order dO's columns (dV of step i), Q's rows (S^T of i + 1), Q's columns (dK of i), dO's rows
// (dP^T of i + 1), so the use that stands at place p of step i has number 4 i + p and buffer (4 i + p) mod 3 = (i + p) mod 3; it
// is loaded when the use three before it has completed.
__device__ __forceinline__ int oper_buf(int n) { return n % 3; }
constexpr int BP_ARR = BP_STG + 2 * STG_BYTES;       // lse_s[2][128], d_s[2][128]
constexpr int BP_BARS = BP_ARR + 2048;
constexpr int BP_SMEM = BP_BARS + 256;
// warps 0-7 compute, 8 TMA, 9 MMA issue (rank 0), 10 LSE / D rows, 11 idle, 12-15 dQ read-out, 16-19 dS^T to shared memory
// (without dQ: 0-10 and one idle)
__host__ __device__ constexpr int bp_threads(bool dq) { return dq ? 640 : 384; }
// 256 x 136 + 128 x (40 + 88 + 80) = 640 x 96, without dQ 256 x 200 + 128 x 104 = 384 x 168
__host__ __device__ constexpr int bp_regs_compute(bool dq) { return dq ? 136 : 200; }
__host__ __device__ constexpr int bp_regs_misc(bool dq) { return dq ? 40 : 104; }
constexpr int BP_REGS_READ = 88, BP_REGS_MOVE = 80;
constexpr uint32_t IDESC_S = make_idesc(256, 128, false, false), IDESC_ACC = make_idesc(256, 128, false, true),
                   IDESC_DQT = make_idesc(128, 128, true, true);
__host__ __device__ constexpr uint32_t koff_h(int kk) { return (kk >> 2) * (HPANEL_BYTES >> 4) + (kk & 3) * 2; }   // K-major slice of a 64-row tile

// DQ = false: dK and dV only (the dK/dV pass of the two-pass backward), the same sums as tc_dkdv_kernel.  A step is then bound by
// the same chain; L = 16384, H = 8 / 8: two-pass backward 3239 -> 3177 us.
template <bool TR, bool DQ>
__global__ void __launch_bounds__(bp_threads(DQ), 1)
tc_bwd_pair_kernel(const __grid_constant__ PairMaps maps, const KArgs a, const TileGrid tg, int* __restrict__ status) {
  wait_for_predecessor();
  extern __shared__ __align__(1024) uint8_t sm[];
  const uint32_t base = smem_u32(sm);
  const uint32_t sK = base + BP_K, sV = base + BP_V, sKT = base + BP_KT, sDS = base + BP_DS, sOP = base + BP_OPER,
                 sSEND = base + BP_SEND, sSTG = base + BP_STG;
  float* lse_s = reinterpret_cast<float*>(sm + BP_ARR);   // [2][128], minus the LSE in log2 units
  float* d_s = lse_s + 256;                               // [2][128], minus D
  const uint32_t bars = base + BP_BARS;
  // rank 0's only, counted in both CTAs: all that a product waits for, one barrier each, because every wait of the issuing warp
  // costs it about as much as three MMAs.  Phase i:
  const uint32_t bar_kv = bars;             // K, V, K^T; dO's rows of step 0
  const uint32_t bar_go_s = bars + 8;       // S^T(i): Q's rows
  const uint32_t bar_go_dv = bars + 16;     // dV(i): P^T(i); dO's columns
  const uint32_t bar_go_dk = bars + 24;     // dK(i): dS^T(i) in tensor memory; Q's columns
  const uint32_t bar_go_dp = bars + 32;     // dP^T(i+1): dS^T(i) and dQ^T(i-1) read out of the columns that it takes; dO's rows
  const uint32_t bar_go_dq = bars + 40;     // dQ^T(i): dP^T(i+1) read out of the columns that it takes; dS^T(i) in shared memory
  // in both: the products' completion
  const uint32_t bar_st = bars + 48, bar_dpt = bars + 56, bar_dqf = bars + 64, bar_doc_e = bars + 72, bar_qc_e = bars + 80, bar_done = bars + 88;
  // each CTA's own
  const uint32_t bar_rows_full = bars + 96 /*[2]*/, bar_rows_empty = bars + 112 /*[2]*/, bar_dpl = bars + 128, bar_dsl = bars + 136, bar_rx = bars + 144;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + BP_BARS + 160);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + BP_BARS + 168);

  const int rank = (int)cluster_rank();
  int bx, hk, bz;
  tile_grid_decode(tg, blockIdx.x >> 1, bx, hk, bz);
  const int ks = bz & 1, b = bz >> 1;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int L = rows_k(a, ks), M = a.M;
  const int pair_row = bx * 2 * TILE;
  if (pair_row >= L || a.dk[ks] == nullptr) return;   // both CTAs
  const int k0_row = pair_row + rank * TILE;          // this CTA's first key in memory
  const bool two = pair_row + TILE < L;               // an odd last tile: rank 1 has no key, all it computes is masked out
  const bool own = rank == 0 || two;
  const int k0a = ks == CLEAN ? clean_key_pos(a, pair_row) : pair_row;
  const int k0b = !two ? k0a : ks == CLEAN ? clean_key_pos(a, pair_row + TILE) : pair_row + TILE;
  const int k0 = rank == 0 ? k0a : k0b;               // its position

  // query tiles that see a key of the pair: segment A (clean queries; noisy ones for noisy keys), then segment B (noisy queries
  // of clean keys), for each head of the group; where the two key tiles' intervals differ, their hull
  int tA0 = 0, nA = 0, tB0 = 0, nB = 0;
  if (ks == CLEAN) {
    auto hull = [&](int qs, int& t0, int& n) {
      if (a.q[qs] == nullptr) return;
      int lo_a, hi_a, lo_b, hi_b, tmp;
      visible_queries_of_clean_key(a, qs, k0a, lo_a, tmp);
      visible_queries_of_clean_key(a, qs, k0a + TILE - 1, tmp, hi_a);
      visible_queries_of_clean_key(a, qs, k0b, lo_b, tmp);
      visible_queries_of_clean_key(a, qs, k0b + TILE - 1, tmp, hi_b);
      int lo = 0, hi = 0;
      if (hi_a > lo_a && hi_b > lo_b) { lo = min(lo_a, lo_b); hi = max(hi_a, hi_b); }
      else if (hi_a > lo_a) { lo = lo_a; hi = hi_a; }
      else if (hi_b > lo_b) { lo = lo_b; hi = hi_b; }
      if (hi > lo) { t0 = lo / TILE; n = (hi + TILE - 1) / TILE - t0; }
    };
    hull(CLEAN, tA0, nA);
    hull(NOISY, tB0, nB);
  } else {
    const int lo = (pair_row / M) * M, hi = min(L, ((pair_row + (two ? 2 : 1) * TILE - 1) / M + 1) * M);
    tA0 = lo / TILE; nA = (hi + TILE - 1) / TILE - tA0;
  }
  StepWalk walk;
  walk.init(tA0, nA, tB0, nB, a.G, hk * a.G, ks == NOISY ? NOISY : CLEAN, TILE, 0, 1);
  const int nsteps = walk.count();

  if (threadIdx.x == 0) {
    if (base & 1023u) *abort_flag = 1; else *abort_flag = 0;   // swizzled tiles need a 1024-byte aligned base
    // (a warp of each role of both CTAs counts once, the loads of both CTAs with rank 0's arrival)
    mbar_init(bar_kv, 1); mbar_init(bar_go_s, 1); mbar_init(bar_go_dv, 16 + 1); mbar_init(bar_go_dk, 16 + 1);
    mbar_init(bar_go_dp, DQ ? 8 + 8 + 1 : 1); mbar_init(bar_go_dq, 16 + 8 + 2);
    mbar_init(bar_st, 1); mbar_init(bar_dpt, 1); mbar_init(bar_dqf, 1); mbar_init(bar_doc_e, 1); mbar_init(bar_qc_e, 1); mbar_init(bar_done, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(bar_rows_full + 8 * i, 1); mbar_init(bar_rows_empty + 8 * i, 8); }
    mbar_init(bar_dpl, 8); mbar_init(bar_dsl, 8); mbar_init(bar_rx, 1);
    fence_mbar_init();
  }
  if (warp == 8) tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // the other CTA's barriers and tensor memory are there
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);   // (the whole of it: the same address in both CTAs)
  const bool bad_base = (*abort_flag != 0);

  if (bad_base) {
    // fall through to the common exit
  } else if (warp >= 8 && warp < 12) {
    reg_dec<bp_regs_misc(DQ)>();
    if (warp == 8) {
      // ------------------------------------------------------------------ TMA loads of this CTA's share, counted by rank 0's
      // barriers
      if (lane == 0 && nsteps > 0) {
        const uint32_t r_kv = peer_addr(bar_kv, 0);
        auto expect = [&](uint32_t bar, int bytes) { if (rank == 0) mbar_expect_tx(bar, 2 * bytes); };   // both CTAs' loads
        auto load_rows = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, const QStep& s) {
          const uint32_t rbar = peer_addr(bar, 0);
          tma_load_3d_pair(dst, map, rbar, s.h * D, s.q0 + rank * HT, b);
          tma_load_3d_pair(dst + HPANEL_BYTES, map, rbar, s.h * D + 64, s.q0 + rank * HT, b);
        };
        auto load_cols = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, const QStep& s) {
          tma_load_3d_pair(dst, map, peer_addr(bar, 0), s.h * D + rank * 64, s.q0, b);
        };
        expect(bar_kv, (DQ ? 3 : 2) * TILE_BYTES + PANEL_BYTES);
        for (int p = 0; p < 2; ++p) {
          tma_load_3d_pair(sK + p * PANEL_BYTES, &maps.k[ks], r_kv, hk * D + 64 * p, k0_row, b);
          tma_load_3d_pair(sV + p * PANEL_BYTES, &maps.v[ks], r_kv, hk * D + 64 * p, k0_row, b);
          if (DQ) tma_load_3d_pair(sKT + p * PANEL_BYTES, &maps.k[ks], r_kv, hk * D + 64 * rank, pair_row + p * TILE, b);
        }
        // (numbers: dOc(i) 4 i, Qr(i) 4 i - 3, Qc(i) 4 i + 2, dOr(i) 4 i - 1)
        auto buf = [&](int i, int p) { return sOP + oper_buf(i + p) * PANEL_BYTES; };
        auto load_qr = [&](int i, const QStep& s) { expect(bar_go_s, PANEL_BYTES); load_rows(buf(i, 0), &maps.q[s.qs], bar_go_s, s); };
        auto load_doc = [&](int i, const QStep& s) { expect(bar_go_dv, PANEL_BYTES); load_cols(buf(i, 0), &maps.doutc[s.qs], bar_go_dv, s); };
        auto load_qc = [&](int i, const QStep& s) { expect(bar_go_dk, PANEL_BYTES); load_cols(buf(i, 2), &maps.qc[s.qs], bar_go_dk, s); };
        auto load_dor = [&](int i, const QStep& s) {
          if (i > 0) expect(bar_go_dp, PANEL_BYTES);
          load_rows(buf(i, 2), &maps.dout[s.qs], i > 0 ? bar_go_dp : bar_kv, s);
        };
        QStep s0 = walk.cur(), s1 = s0;
        load_qr(0, s0);
        load_dor(0, s0);
        walk.next();
        bool ok = mbar_wait_abortable(bar_st, 0, abort_flag);
        if (ok) load_doc(0, s0);
        if (ok && nsteps > 1) {   // (its buffer is free from the start, its barrier only now)
          s1 = walk.cur();
          load_qr(1, s1);
          walk.next();
        }
        ok = ok && mbar_wait_abortable(bar_dpt, 0, abort_flag);
        if (ok) load_qc(0, s0);
        for (int i = 0; i + 1 < nsteps && ok; ++i) {   // s1: step i + 1
          ok = mbar_wait_abortable(bar_doc_e, i & 1, abort_flag);
          if (!ok) break;
          load_dor(i + 1, s1);
          ok = mbar_wait_abortable(bar_st, (i + 1) & 1, abort_flag);
          if (!ok) break;
          load_doc(i + 1, s1);
          QStep s2 = s1;
          if (i + 2 < nsteps) {
            s2 = walk.cur();
            walk.next();
            ok = mbar_wait_abortable(bar_qc_e, i & 1, abort_flag);
            if (!ok) break;
            load_qr(i + 2, s2);
          }
          ok = mbar_wait_abortable(bar_dpt, (i + 1) & 1, abort_flag);
          if (!ok) break;
          load_qc(i + 1, s1);
          s1 = s2;
        }
        if (DQ && ok && rank == 0) mbar_arrive(bar_go_dp);   // in place of another step's load: dQ^T of the last step waits for it
      }
    } else if (warp == 9) {
      // ------------------------------------------------------------------ MMA issue for both CTAs: the whole warp walks the
      // loop, one elected lane issues (see elect_one)
      if (rank == 0 && nsteps > 0) {
        const uint32_t el = elect_one();
        long long w_dv = 0, w_s = 0, w_dk = 0, w_dp = 0, w_dq = 0;
        const long long t_begin = tick<TR>();
        const uint32_t k_lo = desc_lo_k(sK), v_lo = desc_lo_k(sV), kt_lo = desc_lo_mn(sKT), ds_lo = desc_lo_mn(sDS);
        const uint32_t op_k = desc_lo_k(sOP), op_mn = desc_lo_mn(sOP);   // an operand buffer as K-major B / MN-major B
        auto go = [&](uint32_t bar, int i, long long& acc) { return mbar_wait_timed<TR>(bar, i & 1, abort_flag, acc); };
        auto issue_st = [&](int b3) {   // b3: i mod 3
          tc_fence_after();
          const uint32_t qr_lo = op_k + b3 * (PANEL_BYTES >> 4);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) mma_ss_pair_e(tmem, desc64(k_lo + koff(kk)), desc64(qr_lo + koff_h(kk)), IDESC_S, kk > 0, el);
          mma_commit_pair_e(bar_st, el);
        };
        auto issue_dpt = [&](int b3) {
          tc_fence_after();
          const uint32_t dor_lo = op_k + b3 * (PANEL_BYTES >> 4);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) mma_ss_pair_e(tmem + 128, desc64(v_lo + koff(kk)), desc64(dor_lo + koff_h(kk)), IDESC_S, kk > 0, el);
          mma_commit_pair_e(bar_dpt, el);
        };
        auto issue_dqt = [&]() {
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 16; ++kk)
            mma_ss_pair_e(tmem + 192, desc64(kt_lo + moff(kk)), desc64(ds_lo + moff(kk)), IDESC_DQT, kk > 0, el);
          mma_commit_pair_e(bar_dqf, el);
        };
        bool ok = go(bar_kv, 0, w_s) && go(bar_go_s, 0, w_s);
        if (ok) {
          issue_st(0);
          issue_dpt(2);
        }
        int b0 = 0, b1 = 1, b2 = 2;   // i, i + 1, i + 2 mod 3
        for (int i = 0; i < nsteps && ok; ++i) {
          const uint32_t acc = i > 0 ? 1u : 0u;
          const bool more = i + 1 < nsteps;
          ok = go(bar_go_dv, i, w_dv);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_ts_pair_e(tmem + 256, tmem + (kk >> 2) * 64 + (kk & 3) * 8, desc64(op_mn + b0 * (PANEL_BYTES >> 4) + moff(kk)), IDESC_ACC, kk == 0 ? acc : 1u, el);
          mma_commit_pair_e(bar_doc_e, el);
          if (more) {   // over P^T(i): its reader, dV(i), is ahead in the pipe
            ok = go(bar_go_s, i + 1, w_s);
            if (!ok) break;
            issue_st(b1);
          }
          if (DQ && i > 0) {
            ok = go(bar_go_dq, i - 1, w_dq);
            if (!ok) break;
            issue_dqt();
          }
          ok = go(bar_go_dk, i, w_dk);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_ts_pair_e(tmem + 384, tmem + 128 + kk * 8, desc64(op_mn + b2 * (PANEL_BYTES >> 4) + moff(kk)), IDESC_ACC, kk == 0 ? acc : 1u, el);
          mma_commit_pair_e(bar_qc_e, el);
          if (DQ || more) ok = go(bar_go_dp, i, w_dp);
          if (!ok) break;
          if (more) issue_dpt(b0);   // i + 3
          const int t = b0;
          b0 = b1; b1 = b2; b2 = t;
        }
        if (DQ && ok) {
          ok = go(bar_go_dq, nsteps - 1, w_dq);
          if (ok) issue_dqt();
        }
        mma_commit_pair_e(bar_done, el);
        if (!ok) {   // tensor memory is given back below: not before the MMAs already issued have landed (bounded)
          const long long t0 = clock64();
          while (!mbar_try_wait(bar_done, 0) && clock64() - t0 < WAIT_LIMIT_TICKS) {}
        }
        if (lane == 0) {
          trace_add(a.trace, 16 + 8, tick<TR>() - t_begin); trace_add(a.trace, 16 + 9, w_dv); trace_add(a.trace, 16 + 10, w_dp);
          trace_add(a.trace, 16 + 11, w_dk); trace_add(a.trace, 16 + 12, w_dq); trace_add(a.trace, 16 + 7, w_s);
        }
      }
    } else if (warp == 10) {
      // ------------------------------------------------------------------ the LSE and D rows of a step, fetched one step ahead
      auto fetch_rows = [&](const QStep& s, float4& z, float4& dd) {
        const int Lq = rows_q(a, s.qs);
        const int64_t row0 = ((int64_t)b * a.H + s.h) * Lq + s.q0;
        if ((Lq & 3) == 0 && s.q0 + TILE <= Lq) {
          z = reinterpret_cast<const float4*>(a.lse[s.qs] + row0)[lane];
          dd = reinterpret_cast<const float4*>(a.dsum[s.qs] + row0)[lane];
        } else {   // a tile that runs past the end of the tensor (or rows that are not 16-byte aligned): P = 0 and D = 0 there
          float zz[4], ds[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const bool in = s.q0 + 4 * lane + e < Lq;
            zz[e] = in ? a.lse[s.qs][row0 + 4 * lane + e] : INFINITY;
            ds[e] = in ? a.dsum[s.qs][row0 + 4 * lane + e] : 0.f;
          }
          z = make_float4(zz[0], zz[1], zz[2], zz[3]);
          dd = make_float4(ds[0], ds[1], ds[2], ds[3]);
        }
      };
      float4 z_next = make_float4(0.f, 0.f, 0.f, 0.f), d_next = z_next;
      if (nsteps > 0) fetch_rows(walk.cur(), z_next, d_next);
      for (int i = 0; i < nsteps; ++i) {
        const int sr = i & 1;
        walk.next();
        const float4 z = z_next, dd = d_next;
        if (i + 1 < nsteps) fetch_rows(walk.cur(), z_next, d_next);
        bool ok = i < 2 || mbar_wait_abortable(bar_rows_empty + 8 * sr, ((i >> 1) - 1) & 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        float4 z2;
        z2.x = isfinite(z.x) ? z.x * -LOG2E : -INFINITY; z2.y = isfinite(z.y) ? z.y * -LOG2E : -INFINITY;
        z2.z = isfinite(z.z) ? z.z * -LOG2E : -INFINITY; z2.w = isfinite(z.w) ? z.w * -LOG2E : -INFINITY;
        reinterpret_cast<float4*>(lse_s + sr * 128)[lane] = z2;
        reinterpret_cast<float4*>(d_s + sr * 128)[lane] = make_float4(-dd.x, -dd.y, -dd.z, -dd.w);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_rows_full + 8 * sr);
      }
    } else if (DQ && lane == 0) {
      // ------------------------------------------------------------------ the rows of dS^T(i) that the other CTA has copied
      // here are complete: told rank 0
      const uint32_t r_go_dq = peer_addr(bar_go_dq, 0);
      for (int i = 0; i < nsteps; ++i) {
        mbar_expect_tx(bar_rx, PANEL_BYTES);
        if (!mbar_wait_abortable(bar_rx, i & 1, abort_flag)) break;
        mbar_arrive_peer_smem(r_go_dq);
      }
    }
  } else if (DQ && warp >= 16) {
    // ------------------------------------------------------------------ dS^T out of tensor memory, where dK reads it, into the
    // shared memory of the CTAs whose dQ^T needs it: columns 0-63 (queries) to rank 0, 64-127 to rank 1; a lane is a key.  Not
    // done by the compute warps: their 64 columns each took 850 of 4000 clk per step.
    reg_dec<BP_REGS_MOVE>();
    const int r = (warp & 3) * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t r_go_dp = peer_addr(bar_go_dp, 0), r_go_dq = peer_addr(bar_go_dq, 0);
    const uint32_t send_src = sSEND + (warp & 3) * 4096, send_dst = peer_addr(sDS + rank * PANEL_BYTES + (warp & 3) * 4096, rank ^ 1),
                   send_bar = peer_addr(bar_rx, rank ^ 1);
    for (int i = 0; i < nsteps; ++i) {
      bool ok = mbar_wait_abortable(bar_dsl, i & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      uint32_t v[2][32];   // what has to be sent, what stays
      tmem_ld32(tl + 128 + 32 * (rank ^ 1), v[0]); tmem_ld32(tl + 128 + 32 * rank, v[1]);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_peer(r_go_dp);   // dP^T(i+1) may go over it
      // the tiles are free once dQ^T(i-1) has read dS^T(i-1) in both CTAs
      ok = i == 0 || mbar_wait_abortable(bar_dqf, (i - 1) & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint8_t* row = sm + (half == 0 ? BP_SEND : BP_DS + rank * PANEL_BYTES) + r * 128;
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
          *reinterpret_cast<uint4*>(row + ((c8 ^ (r & 7)) << 4)) = make_uint4(v[half][4 * c8], v[half][4 * c8 + 1], v[half][4 * c8 + 2], v[half][4 * c8 + 3]);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (half == 0) bulk_copy_peer(send_dst, send_src, 4096, send_bar);   // this warp's 32 rows
          else mbar_arrive_peer_smem(r_go_dq);
        }
      }
    }
  } else if (DQ && warp >= 12) {
    // ------------------------------------------------------------------ dQ read-out: warps 12, 13 the first 64 queries of the
    // step, 14, 15 the other 64; a lane is a head-dimension index of this CTA's half
    reg_dec<BP_REGS_READ>();
    const int j = (warp >> 1) & 1, dd = (warp & 1) * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t r_go_dp = peer_addr(bar_go_dp, 0);
    if (lane == 0 && nsteps > 0) mbar_arrive_peer(r_go_dp);   // dP^T(1) waits for no dQ^T
    const bool leader = (warp & 1) == 0 && lane == 0;
    float* sg = reinterpret_cast<float*>(sm + BP_STG + j * STG_BYTES) + dd;
    bool ok = true;
    long long w_dqf = 0, c_ro = 0;
    for (int i = 0; i < nsteps; ++i) {
      const QStep st = walk.cur();
      walk.next();
      // after a failed wait the warp still meets the other at the named barrier, then both leave together
      if (ok) {
        ok = mbar_wait_timed<TR>(bar_dqf, i & 1, abort_flag, w_dqf);
        ok = __all_sync(0xffffffffu, ok);
      }
      const long long t0 = tick<TR>();
      uint32_t v[2][32];   // the whole tile into registers first: dP^T of the step after next gets its columns back at once
      if (ok) {
        tc_fence_after();
        tmem_ld32(tl + 192, v[0]); tmem_ld32(tl + 224, v[1]);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_peer(r_go_dp);
      }
      if (leader) bulk_wait_read0();   // the last step's reduction has read the staging tile
      asm volatile("bar.sync %0, 64;" ::"r"(1 + j) : "memory");
      if (ok) {
#pragma unroll
        for (int e = 0; e < HT; ++e) sg[e * HT] = __uint_as_float(v[e >> 5][e & 31]);
        fence_async_smem();
      }
      // the second meeting also takes the decision to leave, for all 64 threads at once
      uint32_t leave;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.b32 q, %1, 0;\n\t"
          "bar.red.or.pred p, %2, 64, q;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(leave) : "r"(*abort_flag), "r"(1 + j) : "memory");
      if (leave) break;
      if (leader && st.q0 + j * HT < a.dq32_rows[st.qs]) {
        float* dst = a.dq32[st.qs] + (((int64_t)b * a.H + st.h) * a.dq32_rows[st.qs] + st.q0 + j * HT) * D + rank * (HT * HT);
        bulk_reduce_add_f32(dst, sSTG + j * STG_BYTES, STG_BYTES);
        bulk_commit();
      }
      c_ro += tick<TR>() - t0;
    }
    if (leader) {
      bulk_wait_all();
      if (j == 0 && rank == 0) { trace_add(a.trace, 16 + 14, w_dqf); trace_add(a.trace, 16 + 15, c_ro); }
    }
  } else {
    // ------------------------------------------------------------------ compute: warpgroup w has queries 64 w .. of every step
    reg_inc<bp_regs_compute(DQ)>();
    const int w = warp >> 2;
    const int r = (warp & 3) * 32 + lane;                      // TMEM lane = key row of the tile
    const int j = k0 + r;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const int c0 = 64 * w;
    const uint32_t r_go_dv = peer_addr(bar_go_dv, 0), r_go_dk = peer_addr(bar_go_dk, 0), r_go_dq = peer_addr(bar_go_dq, 0);
    // query rows that see key j, per query stream (section 3.2 read from the key's side), and the bounds inside
    // which a step needs no masking: every key row of this tile sees all of its queries
    int vqc_lo = 0, vqc_hi = 0, vqn_lo = 0, vqn_hi = 0, fullc_lo = 0, fullc_hi = 0, fulln_lo = 0, fulln_hi = 0;
    if (own) {
      if (ks == CLEAN) {
        int tmp;
        if (a.q[CLEAN] != nullptr) {
          visible_queries_of_clean_key(a, CLEAN, j, vqc_lo, vqc_hi);
          visible_queries_of_clean_key(a, CLEAN, k0 + TILE - 1, fullc_lo, tmp);
          visible_queries_of_clean_key(a, CLEAN, k0, tmp, fullc_hi);
        }
        if (a.q[NOISY] != nullptr) {
          visible_queries_of_clean_key(a, NOISY, j, vqn_lo, vqn_hi);
          visible_queries_of_clean_key(a, NOISY, k0 + TILE - 1, fulln_lo, tmp);
          visible_queries_of_clean_key(a, NOISY, k0, tmp, fulln_hi);
        }
      } else {
        vqn_lo = (j / M) * M; vqn_hi = vqn_lo + M;
        fulln_lo = ((k0 + TILE - 1) / M) * M; fulln_hi = (k0 / M) * M + M;
      }
    }
    const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2);
    bool ok = true;
    long long w_st = 0, w_dpt = 0, w_dsf = 0, c_exp = 0, c_ds = 0;
    const long long t_begin = tick<TR>();
    for (int i = 0; i < nsteps; ++i) {
      const QStep st = walk.cur();
      walk.next();
      const bool need_mask = (st.qs == CLEAN) ? (st.q0 < fullc_lo || st.q0 + TILE > fullc_hi)
                                              : (st.q0 < fulln_lo || st.q0 + TILE > fulln_hi);
      const int sr = i & 1;
      ok = mbar_wait_timed<TR>(bar_rows_full + 8 * sr, (i >> 1) & 1, abort_flag, w_st);
      ok = ok && mbar_wait_timed<TR>(bar_st, i & 1, abort_flag, w_st);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const long long t0 = tick<TR>();
      uint32_t x[64];
      {
        uint32_t (*c)[32] = reinterpret_cast<uint32_t (*)[32]>(x);
        tmem_ld32(tl + c0, c[0]); tmem_ld32(tl + c0 + 32, c[1]);
        tmem_wait_ld();
      }
      // (no branch between the exponentials and the packing of an unmasked tile, so that they overlap)
      auto p_tile = [&](auto masked) {
        const int lo = (st.qs == CLEAN ? vqc_lo : vqn_lo) - st.q0 - c0, hi = (st.qs == CLEAN ? vqc_hi : vqn_hi) - st.q0 - c0;   // visible columns of this thread's key row
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t (&xh)[32] = reinterpret_cast<uint32_t (&)[32]>(x[32 * half]);
          exp_tile<32>(xh, scale2, lse_s + sr * 128 + c0 + 32 * half);
          if (decltype(masked)::value) hide_tile<32>(xh, lo - 32 * half, hi - 32 * half);
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) pk[e] = pack_bf16(__uint_as_float(xh[2 * e]), __uint_as_float(xh[2 * e + 1]));
          tmem_st16(tl + c0 + 16 * half, pk);
        }
        tmem_wait_st();
      };
      if (need_mask) p_tile(std::true_type{}); else p_tile(std::false_type{});
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_peer(r_go_dv);
      const long long t1 = tick<TR>();
      c_exp += t1 - t0;

      ok = mbar_wait_timed<TR>(bar_dpt, i & 1, abort_flag, w_dpt);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const long long t2 = tick<TR>();
      uint32_t pk[2][16];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t y[32];
        tmem_ld32(tl + 128 + c0 + 32 * half, y);
        tmem_wait_ld();
        if (half == 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {   // the other warpgroup's dS^T and dQ^T go over columns of this one's dP^T
            mbar_arrive(bar_dpl);
            if (DQ && i > 0) mbar_arrive_peer(r_go_dq);
          }
        }
        ds_tile<32>(pk[half], reinterpret_cast<const uint32_t (&)[32]>(x[32 * half]), y, d_s + sr * 128 + c0 + 32 * half);
      }
      ok = mbar_wait_timed<TR>(bar_dpl, i & 1, abort_flag, w_dsf);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      tmem_st32(tl + 128 + 32 * w, reinterpret_cast<const uint32_t (&)[32]>(pk));
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) { mbar_arrive_peer(r_go_dk); if (DQ) mbar_arrive(bar_dsl); mbar_arrive(bar_rows_empty + 8 * sr); }   // this warp is done with the stage's LSE / D rows
      c_ds += tick<TR>() - t2;
    }
    if (DQ && ok && lane == 0 && nsteps > 0) mbar_arrive_peer(r_go_dq);   // dQ^T of the last step waits for no dP^T
    if (warp == 0 && lane == 0 && rank == 0) {
      trace_add(a.trace, 16 + 0, nsteps); trace_add(a.trace, 16 + 1, w_st); trace_add(a.trace, 16 + 2, w_dpt);
      trace_add(a.trace, 16 + 3, w_dsf); trace_add(a.trace, 16 + 4, c_exp); trace_add(a.trace, 16 + 5, c_ds);
      trace_add(a.trace, 16 + 6, tick<TR>() - t_begin);
    }
    // epilogue: warpgroup 0 writes dV, warpgroup 1 writes dK (scaled)
    if (ok && nsteps > 0) {
      ok = mbar_wait_abortable(bar_done, 0, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
    }
    if (ok) {
      tc_fence_after();
      // through the buffers of K and V, which nothing reads any more, and TMA stores of a warp's 32 rows (rows past the end of
      // the tensor are not written).  Stored by rows from registers this took 6700 of a unit's 21000 clk outside its steps.
      const CUtensorMap* map = w == 0 ? &maps.dv[ks] : &maps.dk[ks];
      const uint32_t at = base + (w == 0 ? BP_K : BP_V) + (warp & 3) * 4096;
      const float sc = (w == 0) ? 1.f : a.scale;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        uint32_t pk[32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t v[32];
          if (nsteps > 0) { tmem_ld32(tl + 256 + w * 128 + p * 64 + c * 32, v); tmem_wait_ld(); }
          else {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = 0u;
          }
#pragma unroll
          for (int e = 0; e < 16; ++e) pk[c * 16 + e] = pack_bf16(__uint_as_float(v[2 * e]) * sc, __uint_as_float(v[2 * e + 1]) * sc);
        }
        const uint32_t panel = at + p * PANEL_BYTES;
        uint8_t* row = sm + (panel - base) + lane * 128;
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
          *reinterpret_cast<uint4*>(row + ((c8 ^ (lane & 7)) << 4)) = make_uint4(pk[4 * c8], pk[4 * c8 + 1], pk[4 * c8 + 2], pk[4 * c8 + 3]);
        fence_async_smem();
        __syncwarp();
        if (lane == 0 && k0_row + r < L) {
          tma_store_3d(map, panel, hk * D + p * 64, k0_row + r, b);
          bulk_commit();
        }
      }
      if (lane == 0) bulk_wait_all();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) give_up_pair(abort_flag, status, rank);
  cluster_sync();   // no CTA leaves while the other one still writes to its shared memory or signals its barriers
  if (warp == 8) tmem_dealloc_pair(tmem, 512);
}

}  // namespace

template <bool DQ>
static cudaError_t launch_pair(const KArgs& a, cudaStream_t st, bool chained) {
  PairMaps maps;
  for (int s = 0; s < 2; ++s) {
    // a stream that is left out gets the other stream's tensors as placeholders: its maps are never used
    const int sq = a.q[s] != nullptr ? s : 1 - s;
    const int sk = a.k[s] != nullptr ? s : CLEAN;
    if (!tc_make_map(&maps.q[s], a.q[sq], a.H, rows_q(a, sq), a.batch, HT, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.dout[s], a.dout[sq], a.H, rows_q(a, sq), a.batch, HT, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.qc[s], a.q[sq], a.H, rows_q(a, sq), a.batch, TILE, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.doutc[s], a.dout[sq], a.H, rows_q(a, sq), a.batch, TILE, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.k[s], a.k[sk], a.Hkv, rows_k(a, sk), a.batch, TILE, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.v[s], a.v[sk], a.Hkv, rows_k(a, sk), a.batch, TILE, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.dk[s], a.dk[sk], a.Hkv, rows_k(a, sk), a.batch, 32, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.dv[s], a.dv[sk], a.Hkv, rows_k(a, sk), a.batch, 32, D)) return cudaErrorInvalidValue;
  }
  int* status = device_status_ptr();
  if (status == nullptr) return cudaErrorUnknown;
  TileGrid tg = {(max(a.L, a.k[NOISY] != nullptr ? a.Ln : 0) + 2 * TILE - 1) / (2 * TILE), a.Hkv, a.batch * 2, 0, 1};
  tg.tile_major = pairs_tile_major_pay(bwd_sizes(a), device_sm_count(), DQ) ? 1 : 0;
  const long long blocks = 2LL * tile_grid_blocks(tg);
  if (blocks == 0 || blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto kern = a.trace ? tc_bwd_pair_kernel<true, DQ> : tc_bwd_pair_kernel<false, DQ>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BP_SMEM);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, chained, (unsigned)blocks, bp_threads(DQ), BP_SMEM, st, 2, maps, a, tg, status);
}

cudaError_t launch_tc_bwd_pair(const KArgs& a, bool dq, cudaStream_t st, bool chained) {
  return dq ? launch_pair<true>(a, st, chained) : launch_pair<false>(a, st, chained);
}

}  // namespace bdlm
