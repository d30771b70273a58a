// Constants of one axis for the warp-level line solves (lines.cuh), shared with
// the host.  Element type E of the solve; positions past the line are zero.
#pragma once

namespace bfv {

struct LineTab {
  const void *inv, *mul;  // [T * m][S] of every position (0 past the line)
  const void *wt;         // [log2 T][2][T][S] scan weights: forward, the product of mul over
                          // chunks t - 2^k + 1 .. t; backward, over t .. t + 2^k - 1
  int n, T, m;            // T chunks (a power of two) of m positions
};

// T chunks (a power of two, at most 32) of at most maxm positions; T = 0: n is too long.
inline int line_chunks(int n, int maxm) {
  int T = 1;
  while (T < 32 && T * maxm < n) T *= 2;
  return T * maxm >= n ? T : 0;
}

}  // namespace bfv
