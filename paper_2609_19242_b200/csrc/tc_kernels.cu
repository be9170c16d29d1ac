// BDLM attention on the 5th-generation tensor cores (tcgen05): Q.K^T and P.V are issued as
// tcgen05.mma with operands staged in shared memory by TMA (128-byte swizzle) and fp32
// accumulators in tensor memory; the online softmax runs in registers, one thread per query
// row.  The tile schedule enumerates only the key tiles a query tile can see (Algorithm 1:
// clean-prefix tiles, then the noisy-diagonal tiles); no mask is materialised.
#include "fwd_issue.h"
#include "tc_common.cuh"
#include "tc_launch.h"

namespace bdlm {
namespace {

using namespace tc;
using bf16 = __nv_bfloat16;

struct FwdMaps {
  CUtensorMap q[2], k[2], v[2], o[2];
};

// ---------------------------------------------------------------- host: tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace

namespace {
EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) p = nullptr;
    if (q != cudaDriverEntryPointSuccess) p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

}  // namespace

bool tc_encoder_available() { return encode_fn() != nullptr; }

// [batch, L, heads, d] bf16 viewed as 3-D (heads*d, L, batch); box = 64 columns x `rows` rows.
// Encoding a map costs the host a microsecond or two and a call needs six to eight of them, which shows at sizes
// where a whole step takes a few milliseconds; a training loop passes the same tensors again and again, so each host
// thread keeps the maps it encoded last in a small direct-mapped table keyed by (address, shape, box).  A map is a
// plain 128-byte value that describes addresses and strides only, so a copy of it is as good as a fresh encode.
bool tc_make_map(CUtensorMap* m, const void* ptr, int heads_in, int L, int batch, int rows, int d) {
  const int heads = heads_in * (d / 64);   // in units of 64-column panels: the map only knows the row length
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr || ptr == nullptr) return false;
  struct Entry { const void* ptr; int heads, L, batch, rows; bool valid; CUtensorMap map; };
  constexpr int kEntries = 64;
  thread_local Entry cache[kEntries] = {};
  const uint64_t key = (reinterpret_cast<uint64_t>(ptr) >> 8) * 0x9E3779B97F4A7C15ull + (uint64_t)rows * 0x632BE59BD9B4E019ull +
                       (uint64_t)L * 31 + (uint64_t)heads;
  Entry& e = cache[(key >> 32) % kEntries];
  if (e.valid && e.ptr == ptr && e.heads == heads && e.L == L && e.batch == batch && e.rows == rows) {
    *m = e.map;
    return true;
  }
  cuuint64_t gdim[3] = {(cuuint64_t)heads * 64, (cuuint64_t)L, (cuuint64_t)batch};
  cuuint64_t gstride[2] = {(cuuint64_t)heads * 64 * 2, (cuuint64_t)L * heads * 64 * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  e.ptr = ptr; e.heads = heads; e.L = L; e.batch = batch; e.rows = rows; e.map = *m; e.valid = true;
  return true;
}

bool tc_make_map_2d(CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr || ptr == nullptr) return false;
  cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstride, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tc_make_map_panels(CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows, int box_panels) {
  EncodeTiledFn fn = encode_fn();
  if (fn == nullptr || ptr == nullptr || cols % 64 != 0) return false;
  cuuint64_t gdim[3] = {64, (cuuint64_t)rows, (cuuint64_t)cols / 64};
  cuuint64_t gstride[2] = {(cuuint64_t)ld * 2, 128};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)box_panels};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), gdim, gstride, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {
// ---------------------------------------------------------------- forward kernel
constexpr uint32_t IDESC_QK = make_idesc(128, 128, false, false);
constexpr int TILE_BYTES = 2 * PANEL_BYTES;   // 128 x 128 bf16

// Key tiles visible from a run of query rows: a clean segment then a noisy segment, each a run
// of 128-key tiles starting at the first visible key; scalars only (no indexed arrays).
struct TileSched {
  int lo0, lo1, nt0, nt1, lo_last0, lo_last1, hi_first0, hi_first1;
  // key tiles seen by the query rows [q0, q_last]: the visible interval of a row moves up with the row, so the
  // first row gives the lower end and the last row the upper end
  __device__ __forceinline__ void init(int qs, int q0, int q_last, const KArgs& a) {
    int lo_f, hi_f, lo_l, hi_l;
    visible_interval(a, qs, 0, q0, lo_f, hi_f);
    visible_interval(a, qs, 0, q_last, lo_l, hi_l);
    lo0 = lo_f; lo_last0 = lo_l; hi_first0 = hi_f; nt0 = hi_l > lo_f ? (hi_l - lo_f + TILE - 1) / TILE : 0;
    visible_interval(a, qs, 1, q0, lo_f, hi_f);
    visible_interval(a, qs, 1, q_last, lo_l, hi_l);
    lo1 = lo_f; lo_last1 = lo_l; hi_first1 = hi_f; nt1 = hi_l > lo_f ? (hi_l - lo_f + TILE - 1) / TILE : 0;
  }
  // a tile needs per-element masking unless every one of the query rows sees all of its 128 keys
  __device__ __forceinline__ bool need_mask(int ks, int k0) const {
    return ks == 0 ? (k0 < lo_last0 || k0 + TILE > hi_first0) : (k0 < lo_last1 || k0 + TILE > hi_first1);
  }
};

// ---------------------------------------------------------------- forward, warp-specialised
// A unit is one 128-row query tile of TWO query heads of the same KV group (same stream, same rows, so
// the same key tiles and the same masks).  Warp 8 loads Q of both heads once and streams K/V tiles through
// a 2-stage ring; warp 9 issues tcgen05.mma (QK^T from shared memory, PV with P as a TMEM operand: the whole
// warp walks the loop, one elected lane issues); warps 0-7 run the online softmax, one warpgroup per head and
// one thread per query row: the thread holds the tile's 128 scores in registers (one pass over S, no exchange
// between threads).  While one head's warpgroup is in its
// exponentials the tensor core runs the other head's P V and next Q K^T.  P (bf16) overwrites the first 64 of
// the S columns it was computed from; O is rescaled only when the running maximum grew by more than 2^8 (the
// stale maximum is exact in the final LSE and normalisation).
// With an odd number of query heads per KV head (PAIRQ) the two warpgroups take two consecutive query tiles of
// ONE head instead: the unit walks the union of their key tiles (the later tile's list contains the earlier
// one's except for noisy diagonal tiles), a tile that one of them does not see at all is masked out for it
// like any other hidden key, and a second tile past the end of the tensor stays masked and is not written.
// TMEM columns: [0,128) S/P head A   [128,256) S/P head B   [256,384) O head A   [384,512) O head B
//
// A CTA works on one unit after another: the grid has a CTA per unit, and a running CTA takes over the next one that
// has not started (cluster launch control), so the start order still decides who goes first.  Tensor memory,
// barriers and the K/V ring carry over, the next unit's Q is loaded once the last Q K^T has read the old one, its first
// Q K^T runs under the previous unit's last P V and output, and O leaves through a 4 KB staging tile per warp and
// TMA stores.  With one unit per CTA, 16k of the 43k clk of a 1024-key window's unit were not tile work: set-up
// 2k, first scores 4.5k, 16-byte row stores 3.9k (each a memory line of its own), exit and start of the next CTA 4.2k.
// Forward: L = 2048, H = 32 82 -> 69 us, windowed 32K 1.46 -> 1.26 ms, 2 x 8K, H = 16 1.05 -> 1.01 ms, 32K 15.0 -> 14.7 ms.
constexpr int FWDR_THREADS = 384;                            // 8 softmax warps, producer warp, MMA warp, two idle ones
constexpr int FWDR_REGS_SOFTMAX = 224, FWDR_REGS_REST = 56;  // 256 x 224 + 128 x 56 = 384 x 168, what the block is launched with
constexpr int FWDR_STG = 6 * TILE_BYTES;                     // after Q (2 tiles) and the K/V ring (2 stages x 2 tiles)
constexpr int FWDR_STG_WARP = 32 * 128;                      // per softmax warp: 32 rows x 64 columns of O
constexpr int FWDR_BARS = FWDR_STG + 8 * FWDR_STG_WARP;
constexpr int FWDR_SMEM = FWDR_BARS + 512 + 1024;

// What a CTA knows about a unit; written to shared memory by the producer, two slots in turn.
struct FwdUnit {
  int more;                // 0: no unit left
  int qs, b, h0, q0;
  TileSched sch;
};
constexpr int FWD_UNIT_BYTES = 64;
static_assert(sizeof(FwdUnit) <= FWD_UNIT_BYTES, "unit slot");

// What fwd_issue_loop works with: the issuing warp's waits and instructions, as closures over the kernel's state.
template <class U, class Q, class K, class V, class P, class QK, class PV, class O, class KV>
struct IssueOps { U& next_unit; Q& q_full; K& k_full; V& v_full; P& p_full; QK& qk; PV& pv; O& o_done; KV& kv_done; };

// D = head dimension (128 or 64).  With D = 64 a tile is one 64-column panel: the second panel of every shared-memory
// tile stays unused, Q K^T contracts over four k-slices and P V produces 64 output columns.
template <bool TR, bool PAIRQ, int D>
__global__ void __launch_bounds__(FWDR_THREADS, 1)
tc_fwdr_kernel(const __grid_constant__ FwdMaps maps, const KArgs a, const TileGrid tg, int* __restrict__ status) {
  constexpr uint32_t IDESC_PV = make_idesc(128, D, false, true);
  constexpr int OPER_BYTES = TILE_BYTES * D / 128;   // bytes TMA delivers per operand tile
  // warpgroup w works on head h0 + w * HSTEP, query rows q0 + w * QSTEP ...
  constexpr int HSTEP = PAIRQ ? 0 : 1, QSTEP = PAIRQ ? TILE : 0, QROWS = PAIRQ ? 2 * TILE : TILE;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t sQ = base, sK0 = base + 2 * TILE_BYTES;   // stage s: K at sK0 + s*2*TILE, V after it
  const uint32_t bars = base + FWDR_BARS;
  const uint32_t bar_q = bars, bar_k_full = bars + 8 /*[2]*/, bar_v_full = bars + 24 /*[2]*/, bar_kv_empty = bars + 40 /*[2]*/,
                 bar_s = bars + 56 /*[2]*/, bar_o = bars + 72 /*[2]*/, bar_p = bars + 88 /*[head][key half]*/,
                 bar_q_empty = bars + 120, bar_unit_full = bars + 128 /*[2]*/, bar_unit_empty = bars + 144 /*[2]*/,
                 bar_clc = bars + 160, bar_drain = bars + 168, clc_slot = bars + 176;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + FWDR_BARS + 192);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + FWDR_BARS + 200);
  auto unit_slot = [&](int k) { return reinterpret_cast<FwdUnit*>(sm + FWDR_BARS + 256 + (k & 1) * FWD_UNIT_BYTES); };
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp index, provably uniform

  auto tile_ks = [](const TileSched& sch, int t) { return t < sch.nt0 ? 0 : 1; };
  auto tile_k0 = [](const TileSched& sch, int t) { return t < sch.nt0 ? sch.lo0 + t * TILE : sch.lo1 + (t - sch.nt0) * TILE; };

  // The producer starts loading as soon as the barriers are set up; everyone else also needs tensor memory.
  if (warp == 8) {
    if (lane == 0) {
      mbar_init(bar_q, 1); mbar_init(bar_q_empty, 1); mbar_init(bar_clc, 1); mbar_init(bar_drain, 1);
      for (int i = 0; i < 2; ++i) {
        mbar_init(bar_k_full + 8 * i, 1); mbar_init(bar_v_full + 8 * i, 1); mbar_init(bar_kv_empty + 8 * i, 1);
        mbar_init(bar_s + 8 * i, 1); mbar_init(bar_o + 8 * i, 1);
        mbar_init(bar_p + 16 * i, 128); mbar_init(bar_p + 16 * i + 8, 128);
        mbar_init(bar_unit_full + 8 * i, 1); mbar_init(bar_unit_empty + 8 * i, 9);   // read by the MMA warp and 8 softmax warps
      }
      *abort_flag = 0;
      fence_mbar_init();
      fence_async_smem();   // this thread issues its first loads without a block barrier in between
    }
    __syncwarp();
    asm volatile("barrier.cta.arrive 1, 384;" ::: "memory");
  } else {
    if (warp == 9) tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
    tc_fence_before();
    asm volatile("barrier.cta.sync 1, 384;" ::: "memory");
    tc_fence_after();
  }

  if (warp >= 8) {
    reg_dec<FWDR_REGS_REST>();
    if (warp == 8) {
      // ------------------------------------------------------------------ producer
      if (lane == 0) {
        const bool two = a.q[CLEAN] != nullptr && a.q[NOISY] != nullptr;
        int index = blockIdx.x, g = 0, n_units = 0, n_q = 0, n_clc = 0;   // g: K/V tiles loaded so far
        bool ok = true, asked = false;
        // The next unit is asked for three K/V tiles before the end of this one, and answered while those are loaded.  Asked
        // for at the start of a unit, the next one would be taken long before it can begin: of 256 units on 148 SMs the
        // heaviest, which start first, would take the second ones too (H = 8 / 1: L = 4096 87 us, now 65; L = 8192, H = 4 / 1
        // 158, now 115; with one unit per CTA 72 and 131).
        auto ask = [&]() { clc_request(clc_slot, bar_clc); asked = true; };
        while (ok) {
          int bx, by, bz;
          tile_grid_decode(tg, index, bx, by, bz);
          const int qs = two ? bz & 1 : (a.q[CLEAN] != nullptr ? CLEAN : NOISY), b = two ? bz >> 1 : bz;
          const int h0 = PAIRQ ? by : by * 2, hk = h0 / a.G;
          const int q0 = (tg.nx - 1 - bx) * QROWS;   // the last query tile sees the most keys: started first
          const int Lq = rows_q(a, qs);
          if (q0 >= Lq) {
            ask();
          } else {
            TileSched sch;
            sch.init(qs, q0, min(q0 + QROWS, Lq) - 1, a);
            if (n_units >= 2) ok = mbar_wait_abortable(bar_unit_empty + 8 * (n_units & 1), ((n_units >> 1) - 1) & 1, abort_flag);
            if (!ok) break;
            FwdUnit* slot = unit_slot(n_units);
            slot->more = 1; slot->qs = qs; slot->b = b; slot->h0 = h0; slot->q0 = q0; slot->sch = sch;
            mbar_arrive(bar_unit_full + 8 * (n_units & 1));
            ++n_units;
            const int nt = sch.nt0 + sch.nt1;
            if (nt > 0) {
              if (n_q > 0) ok = mbar_wait_abortable(bar_q_empty, (n_q - 1) & 1, abort_flag);
              if (!ok) break;
              ++n_q;
              mbar_expect_tx(bar_q, 2 * OPER_BYTES);
              tma_load_3d(sQ, &maps.q[qs], bar_q, h0 * D, q0, b);
              if (D == 128) tma_load_3d(sQ + PANEL_BYTES, &maps.q[qs], bar_q, h0 * D + 64, q0, b);
              // (rows past the end of the tensor are filled with zeros)
              tma_load_3d(sQ + TILE_BYTES, &maps.q[qs], bar_q, (h0 + HSTEP) * D, q0 + QSTEP, b);
              if (D == 128) tma_load_3d(sQ + TILE_BYTES + PANEL_BYTES, &maps.q[qs], bar_q, (h0 + HSTEP) * D + 64, q0 + QSTEP, b);
            }
            if (nt == 0) ask();
            for (int t = 0; t < nt; ++t, ++g) {
              const int s = g & 1;
              if (t == max(nt - 3, 0)) ask();
              if (g >= 2) ok = mbar_wait_abortable(bar_kv_empty + 8 * s, ((g >> 1) - 1) & 1, abort_flag);
              if (!ok) break;
              const int ks = tile_ks(sch, t), k0 = tile_k0(sch, t);
              const uint32_t dK = sK0 + s * 2 * TILE_BYTES, dV = dK + TILE_BYTES;
              mbar_expect_tx(bar_k_full + 8 * s, OPER_BYTES);
              const int krow = ks == CLEAN ? clean_key_row(a, k0) : k0;   // where the tile's first key is stored
              tma_load_3d(dK, &maps.k[ks], bar_k_full + 8 * s, hk * D, krow, b);
              if (D == 128) tma_load_3d(dK + PANEL_BYTES, &maps.k[ks], bar_k_full + 8 * s, hk * D + 64, krow, b);
              mbar_expect_tx(bar_v_full + 8 * s, OPER_BYTES);
              tma_load_3d(dV, &maps.v[ks], bar_v_full + 8 * s, hk * D, krow, b);
              if (D == 128) tma_load_3d(dV + PANEL_BYTES, &maps.v[ks], bar_v_full + 8 * s, hk * D + 64, krow, b);
            }
            if (!ok) break;
          }
          ok = mbar_wait_abortable(bar_clc, n_clc & 1, abort_flag);
          if (!ok) break;
          asked = false;
          ++n_clc;
          const bool more = clc_answer(clc_slot, index);
          if (!more) break;
          fence_async_smem();   // the answer has been read before the next request may overwrite it
        }
        if (!ok) {   // leaving early: not before the answer and the loads on their way have landed (bounded)
          const long long t0 = clock64();
          auto landed = [&](uint32_t bar, int parity) { while (!mbar_try_wait(bar, parity) && clock64() - t0 < WAIT_LIMIT_TICKS) {} };
          if (asked) landed(bar_clc, n_clc & 1);
          if (n_q > 0) landed(bar_q, (n_q - 1) & 1);
          for (int i = max(g - 2, 0); i < g; ++i) { landed(bar_k_full + 8 * (i & 1), (i >> 1) & 1); landed(bar_v_full + 8 * (i & 1), (i >> 1) & 1); }
        }
        if (ok && n_units >= 2) ok = mbar_wait_abortable(bar_unit_empty + 8 * (n_units & 1), ((n_units >> 1) - 1) & 1, abort_flag);
        if (ok) {
          unit_slot(n_units)->more = 0;
          mbar_arrive(bar_unit_full + 8 * (n_units & 1));
        }
      }
    } else if (warp == 9) {
      // ------------------------------------------------------------------ MMA issuer
      // the whole warp walks fwd_issue_loop; one elected lane issues (see elect_one).  The lanes vote on every wait, so that
      // they leave together after one that failed in any of them.  (A vote is a few clocks of a tile's 2900; predicating the
      // issue on a lane's own waits instead took the operands off the uniform datapath: 8 to 15 % of the forward.)  Tile
      // counts are broadcast so that the loop is provably uniform.
      const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);   // broadcast: provably warp-uniform
      const uint32_t el = elect_one();
      const uint32_t qa_lo = desc_lo_k(sQ);
      const uint32_t k_lo0 = desc_lo_k(sK0), v_lo0 = desc_lo_mn(sK0 + TILE_BYTES);
      int n_units = 0;
      long long w_p = 0, w_v = 0, w_k = 0;
      auto arrived = [&](uint32_t bar, int parity, long long& acc) { return __all_sync(0xffffffffu, mbar_wait_timed<TR>(bar, parity, abort_flag, acc)) != 0; };
      auto next_unit = [&]() {
        if (!__all_sync(0xffffffffu, mbar_wait_abortable(bar_unit_full + 8 * (n_units & 1), (n_units >> 1) & 1, abort_flag))) return FWD_UNIT_FAILED;
        const volatile FwdUnit* u = unit_slot(n_units);
        const int n = __shfl_sync(0xffffffffu, u->more ? u->sch.nt0 + u->sch.nt1 : FWD_NO_UNIT, 0);
        if (lane == 0) mbar_arrive(bar_unit_empty + 8 * (n_units & 1));
        ++n_units;
        return n;
      };
      auto q_full = [&](int n) { return arrived(bar_q, n & 1, w_k); };
      auto k_full = [&](int g) { return arrived(bar_k_full + 8 * (g & 1), (g >> 1) & 1, w_k); };
      auto v_full = [&](int g) { return arrived(bar_v_full + 8 * (g & 1), (g >> 1) & 1, w_v); };
      // (P: bf16 pairs at columns [0,32) and [32,64) of the head's S region)
      auto p_full = [&](int head, int half, int g) { return arrived(bar_p + 16 * head + 8 * half, g & 1, w_p); };
      auto qk = [&](int head, int g, bool last_of_q) {
        tc_fence_after();
        gemm_ss_e<D / 16>(tmem + 128 * head, qa_lo + head * TILE_LO, k_lo0 + (g & 1) * 2 * TILE_LO, IDESC_QK, 0u, el);
        mma_commit_e(bar_s + 8 * head, el);
        if (last_of_q) mma_commit_e(bar_q_empty, el);
      };
      // O += P V over key half j of the tile: four k-slices of 16 keys
      auto pv = [&](int head, int j, int g, uint32_t acc_first) {
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_ts_e(tmem + 256 + 128 * head, tmem + 128 * head + (4 * j + kk) * 8, desc64(v_lo0 + (g & 1) * 2 * TILE_LO + moff(4 * j + kk)),
                   IDESC_PV, kk == 0 ? acc_first : 1u, el);
      };
      auto o_done = [&](int head) { mma_commit_e(bar_o + 8 * head, el); };
      auto kv_done = [&](int g) { mma_commit_e(bar_kv_empty + 8 * (g & 1), el); };
      const long long tm0 = tick<TR>();
      IssueOps<decltype(next_unit), decltype(q_full), decltype(k_full), decltype(v_full), decltype(p_full), decltype(qk), decltype(pv),
               decltype(o_done), decltype(kv_done)> ops = {next_unit, q_full, k_full, v_full, p_full, qk, pv, o_done, kv_done};
      if (!fwd_issue_loop(ops)) {   // tensor memory is given back below: not before the MMAs already issued have landed (bounded)
        mma_commit_e(bar_drain, el);
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_drain, 0) && clock64() - t0 < WAIT_LIMIT_TICKS) {}
      }
      if (lane == 0) {
        trace_add(a.trace, 8, tick<TR>() - tm0); trace_add(a.trace, 9, w_p); trace_add(a.trace, 10, w_v); trace_add(a.trace, 11, w_k);
      }
    } else if (lane < 2 && warp == 10) {
      prefetch_tmap(&maps.k[lane]); prefetch_tmap(&maps.v[lane]); prefetch_tmap(&maps.o[lane]);
    }
  } else {
    // ------------------------------------------------------------------ softmax: one warpgroup per head, one thread per query row
    reg_inc<FWDR_REGS_SOFTMAX>();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const int w = warp >> 2;
    const int r = (warp & 3) * 32 + lane;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + lane_base + w * 128;          // this row's 128 score columns
    const uint32_t tO = tmem + lane_base + 256 + w * 128;    // and its 128 output columns
    const uint32_t stg = base + FWDR_STG + warp * FWDR_STG_WARP;
    bool ok = true;
    int g = 0;   // tiles done so far
    long long w_s = 0, c_ld = 0, c_max = 0, c_exp = 0;
    const long long t_begin = tick<TR>();
    for (int k = 0; ok; ++k) {
      ok = mbar_wait_abortable(bar_unit_full + 8 * (k & 1), (k >> 1) & 1, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const FwdUnit un = *unit_slot(k);
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_unit_empty + 8 * (k & 1));
      if (!un.more) break;
      const TileSched sch = un.sch;
      const int qs = un.qs, b = un.b, nt = sch.nt0 + sch.nt1;
      const int Lq = rows_q(a, qs), row = un.q0 + w * QSTEP + r, h = un.h0 + w * HSTEP;
      const bool row_ok = row < Lq;                            // PAIRQ: the second tile may lie past the end
      int rlo0 = 0, rhi0 = 0, rlo1 = 0, rhi1 = 0;
      if (row_ok) {
        visible_interval(a, qs, 0, row, rlo0, rhi0);
        visible_interval(a, qs, 1, row, rlo1, rhi1);
      }
      float m_ref = -INFINITY, l = 0.f;
      for (int t = 0; t < nt; ++t, ++g) {
        const int ks = tile_ks(sch, t), k0 = tile_k0(sch, t);
        ok = mbar_wait_timed<TR>(bar_s + 8 * w, g & 1, abort_flag, w_s);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const bool need_mask = sch.need_mask(ks, k0) || un.q0 + QROWS > Lq;   // rows past the end of the tensor see nothing
        const int vlo = (ks == 0 ? rlo0 : rlo1) - k0, vhi = (ks == 0 ? rhi0 : rhi1) - k0;
        // the whole row of the tile in registers: one pass over S.  The softmax warps are bound by instruction issue and
        // by the exponential unit, so the arithmetic is packed two to an instruction where it can be (scaling, sums,
        // three-input maxima) and hidden keys are cleared by bit masks: 3330 -> 2900 clk per key tile of two heads,
        // 5750 -> 3900 for a masked first one; forward at L = 2048, H = 32: 88.8 -> 82.1 us, windowed 32K layer
        // 1.57 -> 1.46 ms.  Long sequences run into the power cap: 32K 15.2 -> 15.0 ms.
        const long long tp0 = tick<TR>();
        uint32_t v[128];
        {
          uint32_t (*c)[32] = reinterpret_cast<uint32_t (*)[32]>(v);
          tmem_ld32(tS, c[0]); tmem_ld32(tS + 32, c[1]); tmem_ld32(tS + 64, c[2]); tmem_ld32(tS + 96, c[3]);
          tmem_wait_ld();
        }
        const long long tp1 = tick<TR>();
        if (need_mask) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {   // -inf on hidden keys: one bit per key, so an element costs one test and one select
            const uint32_t seen = interval_bits(vlo - 32 * j, vhi - 32 * j);
#pragma unroll
            for (int e = 0; e < 32; ++e) v[32 * j + e] = (seen >> e) & 1u ? v[32 * j + e] : 0xff800000u;
          }
        }
        float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          mx0 = max3(mx0, __uint_as_float(v[e]), __uint_as_float(v[e + 1]));
          mx1 = max3(mx1, __uint_as_float(v[32 + e]), __uint_as_float(v[33 + e]));
          mx2 = max3(mx2, __uint_as_float(v[64 + e]), __uint_as_float(v[65 + e]));
          mx3 = max3(mx3, __uint_as_float(v[96 + e]), __uint_as_float(v[97 + e]));
        }
        const float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * a.scale_log2;
        const float m_new = fmaxf(m_ref, mx);
        const bool grow = m_new > m_ref + 8.0f;
        if (__any_sync(0xffffffffu, grow)) {
          const float mb_new = (m_new == -INFINITY) ? 0.f : m_new;
          const float corr = exp2f(m_ref - mb_new);
          m_ref = m_new;
          l *= corr;
          if (t > 0) {
            ok = mbar_wait_abortable(bar_o + 8 * w, (g - 1) & 1, abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              uint32_t o[32];
              tmem_ld32(tO + c * 32, o);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * corr);
              tmem_st32(tO + c * 32, o);
            }
          }
        }
        const float mb = (m_ref == -INFINITY) ? 0.f : m_ref;
        const long long tp2 = tick<TR>();
        // p = exp2(s * scale - m) (exp2(-inf) = 0 on hidden keys); bf16 pairs over the first 64 columns
        uint64_t ps0 = 0, ps1 = 0;
        const uint64_t sc2 = pack_f32x2(a.scale_log2, a.scale_log2), nm2 = pack_f32x2(-mb, -mb);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t pk[32];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            if (half == 1 && e == 4) {   // the first half's store has landed by now: hand it over without stalling for it
              tmem_wait_st();
              tc_fence_before();
              mbar_arrive(bar_p + 16 * w);
            }
            const int c = 64 * half + 4 * e;
            float p0, p1, p2, p3;
            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])), sc2, nm2), p0, p1);
            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])), sc2, nm2), p2, p3);
            p0 = exp2f(p0); p1 = exp2f(p1); p2 = exp2f(p2); p3 = exp2f(p3);
            ps0 = add_f32x2(ps0, pack_f32x2(p0, p1));
            ps1 = add_f32x2(ps1, pack_f32x2(p2, p3));
            pk[2 * e] = pack_bf16(p0, p1);
            pk[2 * e + 1] = pack_bf16(p2, p3);
          }
          tmem_st32(tS + 32 * half, pk);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar_p + 16 * w + 8);
        float l0, l1;
        unpack_f32x2(add_f32x2(ps0, ps1), l0, l1);
        l += l0 + l1;
        c_ld += tp1 - tp0; c_max += tp2 - tp1; c_exp += tick<TR>() - tp2;
      }
      if (TR && warp == 0 && lane == 0) trace_add(a.trace, 0, nt);
      if (ok && nt > 0) {
        ok = mbar_wait_abortable(bar_o + 8 * w, (g - 1) & 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
      }
      if (!ok) break;
      // O leaves 64 columns at a time: TMEM -> registers -> the warp's staging tile -> TMA store of its 32 rows.  (The next
      // unit's P V may overwrite O once this thread has handed over the next P, i.e. after it has read O here.)
      tc_fence_after();
      const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll 1
      for (int c = 0; c < D / 64; ++c) {
        uint32_t pk[32];
        if (nt > 0) {
          uint32_t o[64];
          uint32_t (*oc)[32] = reinterpret_cast<uint32_t (*)[32]>(o);
          tmem_ld32(tO + c * 64, oc[0]); tmem_ld32(tO + c * 64 + 32, oc[1]);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e) pk[e] = pack_bf16(__uint_as_float(o[2 * e]) * inv, __uint_as_float(o[2 * e + 1]) * inv);
        } else {
#pragma unroll
          for (int e = 0; e < 32; ++e) pk[e] = 0u;
        }
        if (lane == 0) bulk_wait_read0();   // the store before this one has read the staging tile
        __syncwarp();
        uint8_t* mine = sm + FWDR_STG + warp * FWDR_STG_WARP + lane * 128;
#pragma unroll
        for (int c8 = 0; c8 < 8; ++c8)
          *reinterpret_cast<uint4*>(mine + ((c8 ^ (lane & 7)) << 4)) = make_uint4(pk[4 * c8], pk[4 * c8 + 1], pk[4 * c8 + 2], pk[4 * c8 + 3]);
        fence_async_smem();
        __syncwarp();
        if (lane == 0 && row < Lq) {   // lane 0 has the warp's first row; rows past the end are clipped
          tma_store_3d(&maps.o[qs], stg, h * D + c * 64, row, b);
          bulk_commit();
        }
      }
      if (row_ok) a.lse[qs][((int64_t)b * a.H + h) * Lq + row] = l > 0.f ? (m_ref + log2f(l)) * LN2 : -INFINITY;
    }
    if (lane == 0) bulk_wait_all();
    if (warp == 0 && lane == 0) { trace_add(a.trace, 1, w_s); trace_add(a.trace, 6, tick<TR>() - t_begin);
      trace_add(a.trace, 3, c_ld); trace_add(a.trace, 4, c_max); trace_add(a.trace, 5, c_exp); }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicExch(status, (int)BDLM_ERR_DEVICE_TIMEOUT);
  if (warp == 9) tmem_dealloc(*tmem_slot, 512);
}

}  // namespace

// Row counts need not be multiples of the 128-row tile: TMA fills the rows of a tile that lie past the end of a tensor
// with zeros, the masks never show a key past the end, and rows past the end are neither read from the per-row arrays
// nor written.  Only the gathered K/V order keeps its own rule (chunks of a multiple of 128 rows: checked at the boundary).
bool tc_rows_ok(const KArgs& a) {
  if (a.L <= 0) return false;
  if (a.q[CLEAN] != nullptr && a.Lqc <= 0) return false;
  if (a.q[NOISY] != nullptr && a.Ln <= 0) return false;
  return true;
}

bool tc_fwd_supported(const KArgs& a) {
  return (a.d == 128 || a.d == 64) && tc_rows_ok(a) && encode_fn() != nullptr;
}

template <int D>
static cudaError_t launch_tc_fwd_d(const KArgs& a, cudaStream_t st) {
  FwdMaps maps;
  for (int s = 0; s < 2; ++s) {
    // a stream that is left out gets the other stream's tensors as placeholders: its maps are never used
    const int sq = a.q[s] ? s : 1 - s;
    if (!tc_make_map(&maps.q[s], a.q[sq], a.H, rows_q(a, sq), a.batch, TILE, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.o[s], a.o[sq], a.H, rows_q(a, sq), a.batch, 32, D)) return cudaErrorInvalidValue;
    const int sk = (s == NOISY && (a.q[NOISY] == nullptr || a.Ln == 0 || !a.diag)) ? CLEAN : s;
    if (!tc_make_map(&maps.k[s], a.k[sk], a.Hkv, rows_k(a, sk), a.batch, TILE, D)) return cudaErrorInvalidValue;
    if (!tc_make_map(&maps.v[s], a.v[sk], a.Hkv, rows_k(a, sk), a.batch, TILE, D)) return cudaErrorInvalidValue;
  }
  const int qrows = max(a.q[CLEAN] != nullptr ? a.Lqc : 0, a.q[NOISY] != nullptr ? a.Ln : 0);
  const int streams = (a.q[CLEAN] != nullptr) + (a.q[NOISY] != nullptr);
  int* status = device_status_ptr();
  if (status == nullptr) return cudaErrorUnknown;
  cudaError_t e;
  if (a.G % 2 == 0) {   // two heads of one KV group per CTA, one softmax warpgroup per head
    auto kern = a.trace ? tc_fwdr_kernel<true, false, D> : tc_fwdr_kernel<false, false, D>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FWDR_SMEM);
    if (e != cudaSuccess) return e;
    const TileGrid tg = make_tile_grid((qrows + TILE - 1) / TILE, a.H / 2, a.batch * streams);
    if (tile_grid_blocks(tg) == 0) return cudaErrorInvalidValue;
    kern<<<tile_grid_blocks(tg), FWDR_THREADS, FWDR_SMEM, st>>>(maps, a, tg, status);
    return cudaGetLastError();
  }
  // odd group size: two consecutive query tiles of one head per CTA
  auto kern = a.trace ? tc_fwdr_kernel<true, true, D> : tc_fwdr_kernel<false, true, D>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FWDR_SMEM);
  if (e != cudaSuccess) return e;
  const TileGrid tg = make_tile_grid(((qrows + TILE - 1) / TILE + 1) / 2, a.H, a.batch * streams);
  if (tile_grid_blocks(tg) == 0) return cudaErrorInvalidValue;
  kern<<<tile_grid_blocks(tg), FWDR_THREADS, FWDR_SMEM, st>>>(maps, a, tg, status);
  return cudaGetLastError();
}

cudaError_t launch_tc_fwd(const KArgs& a, cudaStream_t st) {
  return a.d == 64 ? launch_tc_fwd_d<64>(a, st) : launch_tc_fwd_d<128>(a, st);
}

}  // namespace bdlm
