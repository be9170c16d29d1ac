// Asks the rules that choose a launch: the first argument names the rule, the others are its sizes.  Prints the answer.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "dispatch_rules.h"
#include "lce_rules.h"

using namespace bdlm;

int main(int argc, char** argv) {
  auto num = [&](int i) { return i + 2 < argc ? std::atoi(argv[i + 2]) : 0; };
  const char* rule = argv[1];
  if (!std::strcmp(rule, "order")) std::printf("%d\n", tile_major_pays(num(0), num(1), num(2), num(0), num(3), ORDER_RATIO));
  else if (!std::strcmp(rule, "order_pairs")) {
    const BwdSizes z = {num(0), num(1), num(2), num(3), num(4), num(5), num(6), num(7), num(8)};
    std::printf("%d %d\n", pairs_tile_major_pay(z, num(9), true), pairs_tile_major_pay(z, num(9), false));
  }
  else if (!std::strcmp(rule, "pairs")) {
    const BwdSizes z = {num(0), num(1), num(2), num(3), num(4), num(5), num(6), num(7), num(8)};
    const KeyLoad load = key_load(z, num(9));
    std::printf("%d %d\n", split_key_tiles(load), pairs_pay(z, load));
  } else if (!std::strcmp(rule, "lce_forward")) {
    const Tiling t = forward_tiling(num(4), num(0), num(1), num(2), num(3));
    std::printf("%d %d %d\n", t.bn, t.n_run, t.pair);
  } else if (!std::strcmp(rule, "lce_dw")) {
    const Tiling t = choose_tiling(num(3), num(2), num(1), num(0), 128, 1, 1, EPI_CLK_STORE, 1);
    std::printf("%d %d\n", t.bn, t.pair);
  } else return 1;
}
