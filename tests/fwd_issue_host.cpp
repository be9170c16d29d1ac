// Runs the forward's issuing loop with stand-ins for its waits and instructions.  Reads units (their tile counts) from the
// arguments; the first is the index of the wait that fails (-1: none).  Prints one letter per event, for the test to judge.
#include <cstdio>
#include <cstdlib>

#include "fwd_issue.h"

struct Ops {
  int fail, units, at = 0, waits = 0;
  char** tiles;
  bool wait(char c) {
    std::putchar(c);
    return waits++ != fail;
  }
  int next_unit() {
    if (!wait('u')) return bdlm::FWD_UNIT_FAILED;
    return at < units ? std::atoi(tiles[at++]) : bdlm::FWD_NO_UNIT;
  }
  bool q_full(int) { return wait('q'); }
  bool k_full(int) { return wait('k'); }
  bool v_full(int) { return wait('v'); }
  bool p_full(int, int, int) { return wait('p'); }
  void qk(int head, int, bool last_of_q) { std::putchar("ST"[head]); if (last_of_q) std::putchar('E'); }
  void pv(int head, int, int, unsigned acc) { std::putchar(acc ? "AB"[head] : "YZ"[head]); }
  void o_done(int head) { std::putchar("OP"[head]); }
  void kv_done(int) { std::putchar('K'); }
};

int main(int argc, char** argv) {
  Ops op;
  op.fail = std::atoi(argv[1]);
  op.units = argc - 2;
  op.tiles = argv + 2;
  const bool done = bdlm::fwd_issue_loop(op);
  std::printf("\n%d\n", done ? 1 : 0);
}
