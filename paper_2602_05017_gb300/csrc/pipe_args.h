// Arguments of the persistent TMA-pipelined sweep kernel (pipe.cuh).
#pragma once
#include <stdint.h>

#include "internal.h"

namespace bfv {

// A tile is cw "columns" (independent lines) x n positions along the axis,
// cw = 32, or 24 (y/z) or 16 for lines too long for two stages of 32 columns.
//
// The field's rows (fixed y, z: rowlen = nx*S elements) start gpitch elements
// apart in global memory: gpitch = rowlen, or rowlen rounded up to 16 bytes for
// a row-padded copy of a field whose rows are not 16-byte multiples (TMA copies
// need 16-byte aligned rows); the padding elements are carried along untouched.
//
//   mode 0 (x-sweep): a column is one (row, substrate) pair of
//     rows_per_tile = floor(cw/S) consecutive rows (y, z); the rows (gpitch
//     elements each) are staged with one cp.async.bulk each, issued by the
//     lanes of the producer warp, into shared memory at a padded `pitch`
//     (elements) chosen on the host so that the lanes of a warp hit different
//     banks; element (column c, position x) sits at (c/S)*pitch + x*S + c%S.
//   mode 1 / 2 (y- / z-sweep): a column is one of cw consecutive (x, s)
//     entries of a row (mode 1) or entries of a plane, C = ny*gpitch
//     including any padding (mode 2); the tile [n][cw] is staged with
//     cp.async.bulk.tensor boxes of box_rows x cw; element (c, j) sits at
//     j*cw + c.
//
// Tile k of a CTA is tile blockIdx.x + k*gridDim.x of ntiles.
//
// The consumers work on pairs of columns (packed FP32 pairs), so the constants
// come as pairs too: one class per pair of substrates that occurs -- S even:
// (2c, 2c+1), S odd: (c, c+1 mod S), S = 1: (0, 0).  AxisTab::tabT holds, in
// pairs (pipe_tab_pairs of them):
//   constants   [classes][4]              interior inv' and mul; c_hi, c_lo
//   inv', mul   [2][classes][npad]        of every position of every chunk (0 past the line);
//               `split` (odd S only): single values [2][S][npad], half as many
//   weights     [classes][W * chunks per warp][kWtN]  products of mul over whole chunks of
//               the chunk's warp (1 for chunks past the line):
//               kWtF0 this chunk; kWtF1 it and the one before; kWtFx all before it;
//               kWtB1 it and the one after; kWtBx all after it
//   pw          [classes][W]              all of a warp's chunks
enum { kWtF0, kWtF1, kWtFx, kWtB1, kWtBx, kWtN };
#if defined(__CUDACC__)
#define BFV_HD __host__ __device__
#else
#define BFV_HD
#endif
// Chunks of a tile that a consumer warp holds: its 12 or 16 column pairs side by side take half
// a warp, 8 a quarter.
BFV_HD constexpr int pipe_chunks_per_warp(int cw) { return cw == 16 ? 4 : 2; }
BFV_HD constexpr int pipe_classes(int S) { return S > 1 && S % 2 == 0 ? S / 2 : S; }
// (two pairs past a multiple of 16: neighbouring classes start in other banks, 16-byte aligned)
BFV_HD constexpr int pipe_npad(int n) { return (n + 15) / 16 * 16 + 2; }
// maxm: positions of a chunk.
BFV_HD constexpr int pipe_tab_pairs(int maxm, int S, int W, int chunks_per_warp, bool split) {
  return pipe_classes(S) * (4 + (split ? 1 : 2) * pipe_npad(W * chunks_per_warp * maxm) +
                            W * chunks_per_warp * kWtN + W);
}
// The chunk capacity compiled with `split` coefficients (tiles of 32 and 16 columns), for substrate
// counts whose pairs repeat every coefficient.
constexpr int kSplitMaxm = 24;
BFV_HD constexpr bool pipe_can_split(int64_t S) { return S > 1 && S % 2 == 1; }
// Registers of a thread of chunk capacity maxm (the chunk pair takes 2 maxm): 96, 128 and 168
// hold the solve with few or no spills, and the warps an SM then has room for (its four register files
// take whole warps) -- also the largest CTA.
BFV_HD constexpr int pipe_regs(int maxm) { return maxm <= 16 ? 96 : maxm <= 24 ? 128 : 168; }
BFV_HD constexpr int pipe_sm_warps(int maxm) { return 4 * (16384 / (pipe_regs(maxm) * 32)); }

struct PipeArgs {
  int mode, n, S, nx, ny, nz;
  int cw;  // columns per tile: 32, 24 or 16
  int split;
  int64_t ntiles;
  // mode 1 / 2
  int64_t C;
  int tiles_per_plane, nplanes, box_rows, nbox;
  // mode 0
  int rows_per_tile, rowlen, pitch;
  int gpitch;  // elements between consecutive rows of the field (rowlen, or padded)
  int64_t nrows;
  void *field;
  // ring of stages
  int stages;
  int64_t stage_elems;
  AxisTab tab;
  int k0;  // positions k0 .. n-2 have the interior coefficients
  int flags;
  // mode 0: sources (CSR over rows) and the Dirichlet application before the solve
  const int64_t *src_row_off, *src_elem;
  const int2 *src_rowcol;  // (row, position in the row) of each entry
  const void *src_alpha, *src_scale;
  int has_src;
  int prep_warp;  // mode 0: a warp of its own applies Src and B before the solve (1) or none (0)
  const uint8_t *dir_on;
  const void *dir_val;
  int *status;
  int overlap;  // host only: launch with programmatic serialisation
};

}  // namespace bfv
