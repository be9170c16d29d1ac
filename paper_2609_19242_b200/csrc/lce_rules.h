// How the loss head's products are cut into tiles.  Plain C++, so that a host program can ask the rules as well.
#pragma once

namespace bdlm {

constexpr int BM = 128, BN = 256, BK = 64;   // rows of a CTA's tile, most columns, depth of a contraction step
constexpr int MAX_RUN = 8;                   // most N tiles per work item of the forward and of dz

// Clocks of an epilogue per 32 columns.  Rough, but they decide only where the contraction is short: 8 x 350 clk for a tile
// against 512 per 64-deep step of its MMAs, which run under it.
constexpr int EPI_CLK_LSE = 350, EPI_CLK_DZ = 500, EPI_CLK_STORE = 300;

// How a product is cut into tiles: with fixed 256-column tiles and runs of eight, a ragged or small product leaves a
// part of the chip idle (T = 1531, D = 1544, V = 32008: 192 forward items on 148 SMs, dH 84 tiles, the last of every
// seven 8 columns wide).  The width of an N tile and the number of tiles per item are chosen for the shortest launch: rounds
// of items per SM times the clocks of one item.  A 16-deep slice of an M = 128 MMA takes bn / 2 clk, and no less than its
// operands need from shared memory at 128 bytes per clk.  A narrower tile or fewer tiles have to promise 5 %: the count knows
// nothing of L2 or power.  No choice changes a bit of a result.
//   pairs     where rows in units of 256 fill the chip as well (a lone CTA's tiling has to promise 5 %) and the contraction has
//             six steps or more: shorter ones are bound by the epilogue and the start (us, one CTA / pairs: T = 1000, D = 256,
//             V = 32000 forward 34.9 / 36.8, backward 159 / 168; dW of 400 tokens, D = 2048, V = 50304, seven steps: the
//             backward 431 / 415; of 300, five steps: 296 / 295)
//   forward   256 columns, where its vocabulary runs end; 1 to 8 tiles per item, see forward_tiling
//   dz        128 to 256 columns in steps of 16 (of a pair 32); 1 to 8 tiles per item.  T = 1531, D = 1544, V = 32008: 275 -> 188 us
//   dH, dW    256 columns where the matrix has them (their B operand lies MN-major; dH at T = 4096, D = 4096: 5.7 ms with 240
//             or 192 columns against 3.4: its panels then start off the 128-byte lines, or a tile's rows off the 512 bytes they
//             share), unless dH's tiles leave SMs idle: then 64 columns or more (min_bn = 64; V = 32008: T = 1531, D = 1536
//             backward 415 -> 380 us, T = 384, D = 1544 305 -> 264; T = 149, D = 224, V = 50912 280 -> 208)
//             Matrices of 129 to 240 columns in one round of items: one CTA's MMAs cover them in units of 16, a pair's in units of
//             128 (dW, pairs / one CTA, whole backward: 2609 x 224 x 4488 53.1 / 50.0 us, 11177 x 224 x 5192 220 / 209, 4096 x 144 x
//             8000 92.2 / 89.5; in more rounds memory bounds them: 3000 x 176 x 30000 266.5 / 268.4)
constexpr int PAIR_DEPTH = 6;
struct Tiling { int bn, n_run; bool pair; };
inline Tiling choose_tiling(int sms, int M, int N, int K, int min_bn, int min_run, int max_run, int epi_per_32, int b_mn) {
  const int nk = (K + BK - 1) / BK;
  Tiling best = {BN, max_run, false};
  double t_best = 1e300;
  for (int pair = nk >= PAIR_DEPTH; pair >= 0; --pair) {
    const int rows = pair ? 2 * BM : BM, slots = sms / (pair + 1);
    const long long m_tiles = (M + rows - 1) / rows;
    const int least = pair && b_mn && min_bn < 128 ? 128 : min_bn;   // (half of an MN-major tile is whole panels)
    const int unit = b_mn ? least : pair ? 32 : 16;
    const bool few = b_mn && least < 128 && m_tiles * ((N + BN - 1) / BN) < slots;
    for (int bn = BN; bn >= least; bn -= unit) {
      if (bn > least && bn - unit >= N) continue;           // a whole unit wider than the matrix
      if (b_mn && bn < BN && N > bn && !few) break;
      const long long n_tiles = (N + bn - 1) / bn;
      // the columns that MMAs compute: of a lone tile wider than the matrix those that its layout's units cover
      const int cover = pair ? (b_mn ? 128 : 32) : 16;
      const bool narrow = bn == BN && n_tiles == 1 && m_tiles <= slots;
      const int cols = narrow ? (N + cover - 1) / cover * cover : bn;
      const double oper = 32 + (pair ? bn / 8 : bn / 4), slice = cols / 2 > oper ? cols / 2 : oper;
      const double epi = (double)epi_per_32 * ((bn + 31) / 32);
      const double mma = nk * (BK / 16) * slice;
      const double tile = mma > epi ? mma : epi;
      for (int run = max_run; run >= min_run; run /= 2) {
        const long long items = m_tiles * ((n_tiles + run - 1) / run);
        const double t = (double)((items + slots - 1) / slots) * (run < n_tiles ? run : n_tiles) * tile + epi;
        if (t < 0.95 * t_best) { t_best = t; best = {bn, run, pair != 0}; }
      }
    }
  }
  return best;
}

// The forward: items of one tile where the contraction has DEEP steps or more, the token tiles share W's and there are ROUNDS rounds of
// items.  The tiles of an item share nothing on chip, and the CTAs that run together read the same few W tiles only while they keep
// step, which eight deep tiles in a row do not: 8192 x 4096 x 128256 reads 8.6 GB from memory with items of eight, 5.6 with items of
// one.  Items of eight / one, on pairs (us): 8192 x 4096 x 128256 6450 / 5960; 12288 x 4096 x 64000 4890 / 4465; 4096 x 4096 x
// 128256 3058 / 2957; 8192 x 1280 x 50304 742 / 728; 8192 x 1024 x 50304 591 / 588; 8192 x 768 x 50304 450 / 449; shorter ones are
// bound by the epilogue, and all CTAs on the same W tile at once cost more there: 8192 x 512 x 50304 339 / 349, 2048 x 384 x 128256
// 211 / 218.  In few rounds the last one counts, which choose_tiling weighs (items of two / one: 123 x 1048 x 49664 37 / 40, 137 x
// 4000 x 20272 54 / 58).
constexpr int DEEP = 16, ROUNDS = 4;
inline Tiling forward_tiling(int sms, int T, int D, int V, int run_tiles) {
  const long long items = (long long)((T + 2 * BM - 1) / (2 * BM)) * ((V + BN - 1) / BN);
  const bool one = (D + BK - 1) / BK >= DEEP && T > 2 * BM && items >= ROUNDS * (sms / 2);
  return choose_tiling(sms, T, V, D, BN, run_tiles, one ? run_tiles : MAX_RUN, EPI_CLK_LSE, 0);
}

}  // namespace bdlm
