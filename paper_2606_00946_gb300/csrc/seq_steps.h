// Which named barriers the warps of a sequential-commit CTA meet on at which
// step, as plain functions that k_route_seq calls and a host check walks
// through (tests/test_seq_steps.py explores every order the warps can take).
//
// For n requests the scoring warps take steps 0 .. n (step s decides request
// s - 1 and scores request s; step n only decides), the lookup warps steps
// -1 .. n - 2 (step s prepares request s + 1), the inserting warps steps 0 .. n
// (step s inserts request s - 1).  A named barrier counts arrivals and knows no
// request, so every barrier is used again only by warps that an earlier wait
// holds back until everyone has left its last use.
#pragma once

#if defined(__CUDACC__)
#define LS_SEQ_FN __host__ __device__ __forceinline__ constexpr
#else
#define LS_SEQ_FN inline constexpr
#endif

namespace ls {
namespace seq {

// Request s is looked up: the lookup warps arrive at the end of their step
// s - 1, the scoring warps wait in step s < n.
LS_SEQ_FN int bar_looked_up(int s) { return 2 + (s & 1); }

// The inserting warps are through their step s (they have taken the decision
// on request s - 1, and its keys are in): they arrive in step s, the scoring
// warps wait in step s + 2, the last one (n) included: their arrival at
// bar_bids_insert there must not meet that of step n - 2, which inserting warps
// may still be on their way to.  With it three uses of a barrier are apart: an
// inserting warp arrives for step s + 3 only after that step's bids, told by
// scoring warps that have waited for step s.
LS_SEQ_FN int bar_inserted(int s) { return 4 + s % 3; }
LS_SEQ_FN bool waits_inserted(int s, int n) { return s >= 2 && s <= n; }  // scoring warps, step s
LS_SEQ_FN bool tells_inserted(int s, int n) { return s + 2 <= n; }        // inserting warps, step s

// The bids for request s - 1 are in: the scoring warps arrive in step s, the
// lookup warps wait in their step s.
LS_SEQ_FN int bar_bids_look() { return 7; }
LS_SEQ_FN bool tells_look(int s, int n) { return s > 0 && s + 1 < n; }

// The same for the inserting warps, steps 1 to n.
LS_SEQ_FN int bar_bids_insert(int s) { return 8 + (s & 1); }

}  // namespace seq
}  // namespace ls
