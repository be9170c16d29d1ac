// Rules on sizes that choose how a call is launched.  Plain C++, so that a host program can ask them as well.
#pragma once

#include <algorithm>

namespace bdlm {

// What a backward call looks like to the rules below.
struct BwdSizes {
  int batch, L, Lqc, cq_pos0, Ln;   // clean keys, clean query rows (0: none) from this position on, noisy rows (0: none)
  int Hkv, G, window, kv_chunk_len;
};

// Whether the units of a launch start tile-major (see TileGrid).  A stack (one head of one batch element and stream; ny nz of
// them) has nx units; work grows by one from the lightest unit up to `heavy` (nx without a window) and stays there; `at_once`
// units run at one time.  Tile-major when the heaviest unit takes more than 1 / ratio of the launch's ideal duration.
inline bool tile_major_pays(int nx, int ny, int nz, double heavy, int at_once, double ratio) {
  const double stack = heavy * nx - heavy * (heavy - 1) / 2;
  return heavy * ratio * at_once > stack * ny * nz;
}
constexpr double ORDER_RATIO = 5;   // one CTA per tile: 10 SMs > ny nz (nx + 1)

// Pairs of CTAs (backward): half as many units at once, each of 256 keys.  Measured x-fastest / tile-major, sustained at the
// power cap (us), by 2 ny nz stack / heavy (= ny nz (nx + 1) without a window), which is compared with 2 ratio SMs / 2:
//                                         fused              dK/dV alone
//    720   L = 11264, H = 32 / 8           5155 / 5114        3700 / 3531
//    784   L = 12288, H = 8 / 8            1552 / 1526        1113 / 1079
//    888   3 x 9216, H = 12 / 4            4005 / 4001        2845 / 2747
//    928   2 x 7168, H = 32 / 8            4433 / 4616        3103 / 3044
//    976   L = 15360, H = 8 / 8            2290 / 2329        1653 / 1652
//    984   3 x 10240, H = 12 / 4           4831 / 4865        3457 / 3348
//   1040   L = 16384, H = 8 / 8            2561 / 2628        1844 / 1880
//   1200   3 x 6144, H = 32 / 8            4982 / 5541        3447 / 3494
//   1312   2 x 10240, H = 32 / 8           8404 / 9151        5966 / 6051
//    555   L = 8192, H = 32 / 8, window 7500    2980 / 2836        2112 / 1935
//    618   L = 8192, H = 32 / 8, window 6500    2807 / 2783        1977 / 1888
//    640   L = 12000, H = 16 / 4, window 3500   1674 / 1810        1113 / 1201
//    699   L = 8192, H = 32 / 8, window 5200    2567 / 2640        1801 / 1751
//    768   L = 8192, H = 32 / 8, window 4096    2271 / 2448        1563 / 1562
//    912   L = 12288, H = 32 / 8, window 10000  5797 / 6026        4204 / 4119
//   1036   L = 12288, H = 32 / 8, window 8000   5323 / 5838        3775 / 3814
//   1280   2 x 12000, H = 16 / 4, window 3500   3296 / 3773        2232 / 2330
// The fused kernel turns earlier than dK/dV alone, and under a window earlier still: its dQ accumulators leave L2 when the tiles of
// all heads run together, while neighbouring tiles of one head complete them (3 x 6144, H = 32 / 8: one CTA per tile 5107).
// Tiles are counted over the clean keys: noisy ones have a few steps each.  With 32 query heads or more the fused kernel counts the
// longer of the two streams, as its accumulators then need the other order all the more (blocks without clean queries, fused,
// x-fastest / tile-major: L = 9984, 19712 rows, H = 24 / 8 3147 / 3094; L = 12288, 32768 rows, H = 32 / 8 8228 / 8660; L = 8192,
// 20480 rows, H = 64 / 8 7814 / 8316).
inline bool pairs_tile_major_pay(const BwdSizes& z, int sms, bool dq) {
  const int keys = dq && z.Hkv * z.G * z.batch >= 32 ? std::max(z.L, z.Ln) : z.L, nx = (keys + 255) / 256;
  const double band = z.window > 0 ? z.window / 256.0 + 1 : nx, heavy = band < nx ? band : nx;
  return tile_major_pays(nx, z.Hkv, 2 * z.batch, heavy, sms / 2, !dq ? 20.0 / 3 : heavy < nx ? 4.2 : 6);
}

// How many CTAs share a clean key tile (1, 2 or 4), from two estimates in steps of STEP_ROWS query rows: `heavy` for the
// first clean key tile and `mean` per SM; with a prefix table the blocks are taken to be spread evenly over the keys.
// A launch cannot end before its heaviest CTA, so a split pays when that is well above the mean; below, longest-first
// start order fills the chip and the exchange of the partial tiles (about 4 steps per CTA) is a loss.  Clusters of four
// only reach 132 of the 148 SMs.  Fused backward with 1 / 2 / 4 CTAs per tile (us, all kernels of the call):
//   L = 2048, H = 32 / 8        heavy 1.9 means    386 /  308 /  343
//   L = 1024, H = 32 / 8        heavy 3.4 means    236 /  176 /  174
//   L = 8192, H = 8 / 1         heavy 4.4 means   2097 / 1098 /  740
//   L = 16384, H = 8 / 1        heavy 2.3 means   4284 / 2717 / 2919
//   L = 4096, H = 32 / 8        heavy 1.06 means   914 /  920 / 1050
//   L = 8192, H = 32 / 8        heavy 0.55 means  2755 / 3122 / 4237
// and at the thresholds:
//   L = 4096, H = 32 / 8        heavy 1.09 means   806 /  798 /  972
//   L = 3584, H = 32 / 8        heavy 1.23 means   682 /  639 /  790
//   L = 3072, H = 32 / 8        heavy 1.42 means   571 /  470 /  585
//   L = 1536, H = 32 / 8        heavy 2.64 means   248 /  151 /  174
//   L = 14336, H = 8 / 1        heavy 2.60 means  3789 / 2302 / 2195
//   L = 12288, H = 8 / 1        heavy 3.02 means  3193 / 1844 / 1625
//   L = 1280, H = 32 / 8        heavy 3.08 means   200 /  123 /  138
//   2 x 1024, H = 16 / 8, window 256   1.35 means, 28 steps: 74 / 82 / 121 (few steps: the estimate is rough there)
// Under MIN_HEAVY steps the exchange eats what the split gives (L = 256: 37 / 36 / 36).
constexpr int TILE_KEYS = 128, STEP_ROWS = 64;
constexpr double MIN_HEAVY = 24, SPLIT_2 = 1.2, SPLIT_4 = 3.0;
struct KeyLoad { double heavy, mean, total; };   // steps of STEP_ROWS query rows: of the first clean key tile, per SM, of all clean key tiles of a KV head
inline KeyLoad key_load(const BwdSizes& z, int sms) {
  const double W = z.window > 0 ? z.window : 0;
  double heavy = 0, total = 0;
  for (int noisy = 0; noisy <= 1; ++noisy) {
    const int rows = noisy ? z.Ln : z.Lqc;
    if (rows == 0) continue;
    const double nq = (rows + STEP_ROWS - 1) / STEP_ROWS;
    const double seen = noisy ? 0.5 * z.L : z.cq_pos0 + 0.5 * z.Lqc;   // keys a query sees on average
    heavy += W > 0 ? std::min(nq, (W + TILE_KEYS) / STEP_ROWS + 1) : nq;
    total += nq * ((W > 0 ? std::min(W, seen) : seen) / TILE_KEYS + 1);
  }
  total *= z.G;
  return {heavy * z.G, total * z.Hkv * z.batch / sms, total};
}
inline int split_key_tiles(const KeyLoad& l) {
  if (l.heavy < MIN_HEAVY || l.heavy < SPLIT_2 * l.mean) return 1;
  return l.heavy < SPLIT_4 * l.mean ? 2 : 4;
}

// Where clean K/V lie in chunks of an odd number of tiles, every other boundary between chunks falls into a pair, and its two tiles
// are neighbours in memory but stand anywhere: the pair walks the queries between their positions for both, although only one of
// them is seen by those.  How many tiles that is cannot be read from the sizes; for an all-gather of zigzag shards (chunk r next
// to chunk n - 1 - r) a query at position x of the sequence lies between the two with probability 2 min(x, 1 - x).  Clean queries
// count by where they stand, noisy ones as spread evenly (a half).  Weighed with APART: chunks slow one CTA per tile, too.  Calls
// without noisy queries bear more of it.  Fused backward, H = 32 / 8, zigzag, one CTA per tile / pairs (us), by the whole extra
// over the tiles there are; "run": a rank's clean queries alone, "blocks": with its blocks:
//   0.36    L = 32768, chunks of 1 tile                    49340 / 57010
//   0.17    L = 8064, 3 tiles                               3405 /  3489
//   0.145   L = 16128, 3 tiles                             10740 / 11350
//   0.130   L = 32640, 3 tiles                             46710 / 46830
//   0.116   L = 11264, 11 tiles, blocks                     1023 /  1047
//   0.097   L = 16000, 5 tiles                             10520 / 10640
//   0.093   L = 22528, 11 tiles, blocks                     1922 /  1880
//   0.082   L = 26624, 13 tiles, blocks                     2315 /  2248
//   0.080   L = 16128, 7 tiles                             10570 / 10440
//   0.065   L = 32256, 7 tiles                             43380 / 41420
//   0.22    L = 14336, 7 tiles, run                          329 /   328
//   0.14    L = 22528, 11 tiles, run                         732 /   719
//   0.12    L = 26624, 13 tiles, run                         991 /   966
constexpr double APART = 0.7;
inline double pairs_apart(const BwdSizes& z) {
  const int n = z.kv_chunk_len > 0 && z.kv_chunk_len / TILE_KEYS % 2 == 1 ? z.L / z.kv_chunk_len : 0;
  auto below = [](double x) { return x < 0.5 ? x * x : 0.5 - (1 - x) * (1 - x); };   // integral of 2 min(x, 1 - x)
  const double x0 = (double)z.cq_pos0 / z.L, x1 = (double)(z.cq_pos0 + z.Lqc) / z.L;
  const double between = (below(x1) - below(x0)) * z.L + 0.5 * z.Ln;   // query rows
  return APART * (n / 2) * z.G * between / TILE_KEYS;
}

// Whether pairs of CTAs (tc_bwd_pair_kernel) take the call: head dimension 128, key tiles not shared (a pair has two of them), and
// enough work for what a pair does more.  In 128 x 128 tiles: its two key tiles see one query tile more in their hull than each by
// itself wherever a query stream's limit passes them, noisy key tiles two (half as much again, as measured, for masking them),
// and a unit's start and end cost it 3.6 tiles more than two CTAs'.  Fused backward, one CTA per tile / pairs (us, whole
// call), by that extra over the tiles there are:
//   0.015   L = 32768, H = 32 / 8                  40770 / 37860
//   0.040   L = 12288, H = 32 / 8                   6400 /  6070
//   0.051   L = 16384, H = 8 / 8                    2690 /  2640
//   0.059   2 x 8192, H = 16 / 4                    2980 /  2850
//   0.059   L = 32768, H = 32 / 8, window 4096     11540 / 11010
//   0.078   L = 6144, H = 32 / 8                    1760 /  1730
//   0.093   L = 5120, H = 32 / 8                    1230 /  1220
//   0.100   L = 8192, H = 16 / 16                   1523 /  1540
//   0.115   2 x 4096, H = 32 / 8                    1690 /  1710
//   0.115   L = 32768, H = 32 / 8, window 2048      6390 /  6550
//   0.132   3 x 6144, H = 8 / 8                     1367 /  1399
constexpr double PAIR_EXTRA = 0.09, PAIR_EXTRA_APART_RUN = 0.15, PAIR_MASKED = 1.5, PAIR_UNIT = 3.6;
inline bool pairs_pay(const BwdSizes& z, const KeyLoad& l) {
  const double tiles = l.total * STEP_ROWS / TILE_KEYS, pairs_c = z.Lqc / 256.0, pairs_n = z.Ln / 256.0;
  const double extra = PAIR_MASKED * z.G * (pairs_c + 3 * pairs_n) + PAIR_UNIT * (z.L / 256.0 + pairs_n);
  return extra <= PAIR_EXTRA * tiles && extra + pairs_apart(z) <= (z.Ln == 0 ? PAIR_EXTRA_APART_RUN : PAIR_EXTRA) * tiles;
}

}  // namespace bdlm
