// Warp-level line solves in registers, for fields that stay in L2.
//
// A warp takes an item of 32/T adjacent lines, each cut into T chunks of m
// positions (T a power of two, m <= MAXM): lane t*(32/T) + l holds chunk t of
// line l.  Its positions are all loaded at once (one round of L2 latency),
// solved in registers, and stored; carries cross the chunks by shuffles, so an
// item needs neither shared memory nor a CTA barrier, and warps hide one
// another's latency.  Lanes without a line, and positions past a line's end,
// have zero values and zero coefficients.
//
// The recurrences (App. A) run twice in either direction: from a zero carry for
// the chunk's end value, then from the true carry.  The end values meet in a Kogge-Stone scan over the chunks,
// weighted with products of mul that the host forms in FP64.
//
// The field is read through L1, where the lanes of neighbouring items (a CTA
// takes consecutive ones) share sectors; the caller's barrier between sweeps
// acquires what other SMs wrote.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lines_args.h"

namespace bfv {

// Dirichlet values of a lane's line: which of its positions take the value.
template <typename E>
struct ItemDir {
  bool on;    // the line's substrate is flagged
  bool face;  // the whole line lies on a face of the other axes
  E val;
  __device__ __forceinline__ bool at(int j, int n) const {
    return on && (face || j == 0 || j == n - 1);
  }
};

// Solve one item.  p: position 0 of the lane's chunk (element stride ps); len:
// its positions (0: none); lo: its first position; s: its substrate.  prep(v)
// may change the loaded values before the solve.
template <typename E, int MAXM, typename Prep>
__device__ __forceinline__ void solve_item(E *p, long long ps, int len, int lo, int s, int lane,
                                           const LineTab &tb, int S, const ItemDir<E> &before,
                                           const ItemDir<E> &after, Prep &&prep) {
  const unsigned FULL = 0xffffffffu;
  const int n = tb.n, T = tb.T, m = tb.m, lpw = 32 / T, t = lane / lpw;
  E v[MAXM], mu[MAXM];
#pragma unroll
  for (int i = 0; i < MAXM; i++) v[i] = i < len ? p[i * ps] : E(0);
  const E *const t_inv = static_cast<const E *>(tb.inv) + (size_t)lo * S + s;
  const E *const t_mul = static_cast<const E *>(tb.mul) + (size_t)lo * S + s;
#pragma unroll
  for (int i = 0; i < MAXM; i++) mu[i] = i < m ? __ldg(t_mul + i * S) : E(0);
  prep(v);
  if (__any_sync(FULL, before.on)) {
#pragma unroll
    for (int i = 0; i < MAXM; i++)
      if (i < len && before.at(lo + i, n)) v[i] = before.val;
  }
  E g = E(0);
#pragma unroll
  for (int i = 0; i < MAXM; i++)
    if (i < m) {
      v[i] *= __ldg(t_inv + i * S);
      g = fma(mu[i], g, v[i]);
    }
  const E *const w = static_cast<const E *>(tb.wt) + (size_t)t * S + s;
  const int TS = T * S;
  for (int k = 0, dd = 1; dd < T; dd <<= 1, k++) {
    const E o = __shfl_up_sync(FULL, g, dd * lpw);
    if (t >= dd) g = fma(__ldg(w + 2 * k * TS), o, g);
  }
  g = __shfl_up_sync(FULL, g, lpw);
  if (t == 0) g = E(0);
#pragma unroll
  for (int i = 0; i < MAXM; i++)
    if (i < m) {
      g = fma(mu[i], g, v[i]);
      v[i] = g;
    }
  E x = E(0);
#pragma unroll
  for (int i = MAXM - 1; i >= 0; i--)
    if (i < m) x = fma(mu[i], x, v[i]);
  for (int k = 0, dd = 1; dd < T; dd <<= 1, k++) {
    const E o = __shfl_down_sync(FULL, x, dd * lpw);
    if (t + dd < T) x = fma(__ldg(w + (2 * k + 1) * TS), o, x);
  }
  x = __shfl_down_sync(FULL, x, lpw);
  if (t == T - 1) x = E(0);
#pragma unroll
  for (int i = MAXM - 1; i >= 0; i--)
    if (i < m) {
      x = fma(mu[i], x, v[i]);
      v[i] = x;
    }
  if (__any_sync(FULL, after.on)) {
#pragma unroll
    for (int i = 0; i < MAXM; i++)
      if (after.at(lo + i, n)) v[i] = after.val;
  }
#pragma unroll
  for (int i = 0; i < MAXM; i++)
    if (i < len) p[i * ps] = v[i];
}

// Where a lane's chunk of an item lies.
struct ItemLane {
  long long base;  // element offset of position 0 of the line
  long long ps;    // element stride between positions
  int s, lo, len;
  int row;         // x: the line's row
  bool face;       // the whole line lies on a face of the two other axes
};
__device__ __forceinline__ ItemLane item_lane(int axis, int item, int lane, const LineTab &tb,
                                              int nx, int ny, int nz, int S, int lines) {
  ItemLane L;
  const int lpw = 32 / tb.T, t = lane / lpw, line = item * lpw + (lane - t * lpw);
  const bool active = line < lines;
  const int q = active ? line : 0, rowlen = nx * S;
  L.lo = t * tb.m;
  L.len = active ? max(0, min(tb.m, tb.n - L.lo)) : 0;
  L.row = 0;
  if (axis == 0) {
    L.row = q / S;
    L.s = q - L.row * S;
    const int z = L.row / ny, y = L.row - z * ny;
    L.face = y == 0 || y == ny - 1 || z == 0 || z == nz - 1;
    L.base = (long long)L.row * rowlen + L.s;
    L.ps = S;
  } else if (axis == 1) {
    const int z = q / rowlen, c = q - z * rowlen, x = c / S;
    L.s = c - x * S;
    L.face = x == 0 || x == nx - 1 || z == 0 || z == nz - 1;
    L.base = (long long)z * ny * rowlen + c;
    L.ps = rowlen;
  } else {
    const int v = q / S, y = v / nx, x = v - y * nx;
    L.s = q - v * S;
    L.face = x == 0 || x == nx - 1 || y == 0 || y == ny - 1;
    L.base = q;
    L.ps = (long long)rowlen * ny;
  }
  return L;
}

// The source update of an x item's lines from the entries e0..e1 of its rows (sorted by element,
// unique).  row_first: first element of the item's first row.
//
// Few entries: on the values in registers; the lanes read the entries and hand each to the lane
// that holds its element (first: the chunk's position 0 from row_first).  An entry takes about
// 0.24 us, one after the other.
constexpr int kFewSources = 4;
template <typename E, int MAXM>
__device__ __forceinline__ void item_sources(E (&v)[MAXM], long long e0, long long e1,
                                             long long row_first, int first, int len, int S,
                                             int lane, const int64_t *elem, const E *alpha,
                                             const E *scale) {
  const unsigned FULL = 0xffffffffu;
  const long long e = e0 + lane;
  // the entry's place relative to the item's first row (a field has fewer than 2^31 elements)
  const int el = e < e1 ? (int)(__ldg(elem + e) - row_first) : -1;
  const E al = e < e1 ? __ldg(alpha + e) : E(0), sc = e < e1 ? __ldg(scale + e) : E(0);
  const int cnt = (int)(e1 - e0);
  for (int j = 0; j < cnt; j++) {
    const int off = __shfl_sync(FULL, el, j) - first;  // from the chunk's position 0
    const E a = __shfl_sync(FULL, al, j), c = __shfl_sync(FULL, sc, j);
    int pos = off / S;
    if (off < 0 || off != pos * S || pos >= len) pos = -1;
    // one update whatever the position: an FP64 instruction costs its 64 cycles also in
    // lanes that discard the result
    E x = E(0);
#pragma unroll
    for (int i = 0; i < MAXM; i++)
      if (i == pos) x = v[i];
    x = (x + a) * c;
#pragma unroll
    for (int i = 0; i < MAXM; i++)
      if (i == pos) v[i] = x;
  }
}

// More: in the field, 32 entries at a time; the item then loads its values again.  (It has loaded
// them before it knows the count, so that few entries cost no round trip: waiting for the count
// first took 0.17 us a step of 50^3.)  Items of one row share its entries; each takes those of its
// own lines line0 .. line0 + lpw - 1.  Agents in every voxel, one after the other and so: 50^3 60.1
// and 22.3 us a step, x 4 138 and 45.0, 100^3 316 and 73.3, 12^3 48.0 and 14.5; 12500 agents in 50^3
// 23.9 and 19.8, 2000 20.1 and 19.8.
template <typename E>
__device__ __forceinline__ void item_sources_in_field(E *field, long long e0, long long e1,
                                                      long long row_first, int rowlen, int row0,
                                                      int line0, int lpw, int S, int lane,
                                                      const int64_t *elem, const E *alpha,
                                                      const E *scale) {
  for (long long e = e0 + lane; e < e1; e += 32) {
    const int off = (int)(__ldg(elem + e) - row_first);
    const int line = (row0 + off / rowlen) * S + off % S - line0;
    if (line < 0 || line >= lpw) continue;
    E *const q = field + row_first + off;
    *q = (*q + __ldg(alpha + e)) * __ldg(scale + e);
  }
  __syncwarp();  // the lanes that load the elements see the update
}

}  // namespace bfv
