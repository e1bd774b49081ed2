// pass_plan.cuh -- how a call of n steps is cut into passes (host code only).
//
// A pass reads one state buffer and writes the other, so the buffer that holds the state after a call
// depends on the number of passes.  A captured call is replayed from the buffer it was captured on:
// it advances the state again only if the state is back there, which takes an even number of
// passes.  Where the number is a matter of speed alone (the register-tile passes, the deeper default
// passes, the multi-step BGK passes), it is therefore even in a captured call, and has the parity of
// the plain cut -- ceil(n / depth) passes, for BGK n -- in every later call of that handle, so that
// calls between replays leave the state in the buffer where the plain cut would.
#pragma once
#include <stdint.h>

namespace sslbm {

enum { kAnyParity = -1, kEvenPasses = 0, kOddPasses = 1 };

// Passes of at most `depth` steps that cover n: the fewest, one more where their number has to be
// odd or even (a single step is one pass).
inline int64_t pass_count(int64_t n, int depth, int parity) {
  const int64_t p = (n + depth - 1) / depth;
  return parity != kAnyParity && (p & 1) != parity && p < n ? p + 1 : p;
}

// Required parity of a call's passes: `captured` is whether this call is being captured, `was_captured`
// whether an earlier one of the handle was; depth: that of the plain cut.
inline int pass_parity(int64_t n, int depth, bool captured, bool was_captured) {
  if (captured) return kEvenPasses;
  return was_captured ? (int)(((n + depth - 1) / depth) & 1) : kAnyParity;
}

// Depth of the next of the pipeline passes that cover n steps: passes deeper than depth are taken
// whole, where they leave at least three steps or none; else the n steps are cut into passes whose
// depths differ by at most one (100 steps at depth 7: 10 of 7 and 5 of 6), rather than full passes and
// a shallow remainder, which runs at a lower rate per step.  parity: of the passes that remain.
inline int next_pass_depth(int64_t n, int depth, int deep, int parity) {
  if (deep > depth && ((n == deep && parity != kEvenPasses) || n >= deep + 3)) return deep;
  const int64_t passes = pass_count(n, depth, parity);
  return (int)((n + passes - 1) / passes);
}

// Parity of the passes that remain after one more.
inline int flip_parity(int parity) { return parity == kAnyParity ? parity : 1 - parity; }

}  // namespace sslbm
