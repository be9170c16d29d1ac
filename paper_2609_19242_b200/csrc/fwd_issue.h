// The order in which the forward's issuing warp waits, issues and commits, apart from how it does so: the kernel supplies the
// waits and the instructions, a host program can supply stand-ins.
//
// Per tile g of a unit with nt key tiles: O += P V for both heads (a and b = 0 and 1), each in two halves of the keys, and
// between them the scores of the next tile.  A wait answers false when it has run out in any lane; nothing is issued or waited
// for after that, and the caller gives up.
#pragma once

#ifdef __CUDACC__
#define BDLM_ISSUE_FN __device__ __forceinline__
#else
#define BDLM_ISSUE_FN inline
#endif

namespace bdlm {

constexpr int FWD_NO_UNIT = -1, FWD_UNIT_FAILED = -2;

// Ops:  int next_unit()                 tiles of the next unit (0: it sees no key), or one of the two codes above
//       bool q_full(n), k_full(g), v_full(g), p_full(head, half, g)
//       void qk(head, g, last_of_q)     scores of tile g, committed; last_of_q: Q is free after them (second head only)
//       void pv(head, half, g, acc)     acc: add to O (0 for the first tile of a unit)
//       void o_done(head), kv_done(g)   commits
// True: every unit is done.  False: a wait has failed.
template <class Ops>
BDLM_ISSUE_FN bool fwd_issue_loop(Ops& op) {
  int nt = 0, g = 0, n_q = 0;   // g: tiles done so far, n_q: units whose Q has been waited for
  while (nt >= 0) {
    if (nt == 0) {   // the first unit, and after units that see no key: nothing in flight to overlap with
      nt = op.next_unit();
      if (nt == FWD_UNIT_FAILED) return false;
      if (nt <= 0) continue;
      if (!op.q_full(n_q) || !op.k_full(g)) return false;
      ++n_q;
      op.qk(0, g, false);
      op.qk(1, g, nt == 1);
    }
    int nt_next = 0;
    for (int t = 0; t < nt; ++t, ++g) {
      const unsigned acc = t > 0 ? 1u : 0u;
      // head a: P arrives in two halves of the keys, so P V over the first 64 keys runs while the softmax is still in the
      // exponentials of the rest
      if (!op.p_full(0, 0, g) || !op.v_full(g)) return false;
      op.pv(0, 0, g, acc);
      if (!op.p_full(0, 1, g)) return false;
      op.pv(0, 1, g, 1u);
      op.o_done(0);
      // the next tile's scores: this unit's, or the first of the next unit (whose Q has been loaded meanwhile).
      // Only one unit ahead: the one after it is announced when the softmax warps have left this one, and they
      // still wait for head b's P V below.
      bool more = t + 1 < nt, q_done = t + 2 == nt;   // q_done: they are the last that read Q
      if (!more) {
        nt_next = op.next_unit();
        if (nt_next == FWD_UNIT_FAILED) return false;
        if (nt_next > 0) {
          if (!op.q_full(n_q)) return false;
          ++n_q;
          more = true;
          q_done = nt_next == 1;
        }
      }
      if (more) {
        if (!op.k_full(g + 1)) return false;
        op.qk(0, g + 1, false);
      }
      // head b
      if (!op.p_full(1, 0, g)) return false;
      op.pv(1, 0, g, acc);
      if (!op.p_full(1, 1, g)) return false;
      op.pv(1, 1, g, 1u);
      op.o_done(1);
      op.kv_done(g);
      if (more) op.qk(1, g + 1, q_done);
    }
    nt = nt_next;
  }
  return true;
}

}  // namespace bdlm
