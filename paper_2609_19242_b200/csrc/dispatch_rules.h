// Rules on sizes that choose how a call is launched.  Plain C++, so that a host program can ask them as well.
#pragma once

namespace bdlm {

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
inline bool pairs_tile_major_pay(int nx, int ny, int nz, int window, int sms, bool dq) {
  const double keys = window > 0 ? window / 256.0 + 1 : nx, heavy = keys < nx ? keys : nx;
  return tile_major_pays(nx, ny, nz, heavy, sms / 2, !dq ? 20.0 / 3 : heavy < nx ? 4.2 : 6);
}

}  // namespace bdlm
