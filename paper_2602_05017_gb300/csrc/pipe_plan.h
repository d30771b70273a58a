// Tile shapes of the pipelined sweep (pipe.cuh): host arithmetic only, no CUDA calls.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

#include "pipe_args.h"

namespace bfv {

struct PipeShape {
  int T = 1, m = 1, maxm = 16;  // chunks of a line, positions of a chunk, its capacity
  int cw = 32, W = 1;           // columns per tile (32, or 24 or 16 for long lines); consumer warps
  int split = 0;                // coefficients per substrate instead of per pair (pipe_args.h)
  int box_rows = 0, nbox = 0, rows_per_tile = 0, pitch = 0;
  int stages = 0, ctas = 1;     // ctas: per SM
  int64_t stage_elems = 0, ntiles = 0;
  size_t smem = 0;
};
struct PipeKnobs {
  // asked-for chunk length and columns per tile (0: the planner's): the chunk capacity that holds it
  // or the largest of the axis and width, and the planner's own choice where those do not fit
  int chunk = 0, cw = 0;
  int ns = 4;             // most ring stages per CTA
};

// Shared-memory wavefronts of one warp access of the pipelined x tile at row
// pitch `pitch` (elements): lane l reads column pair l % (cw/2) of its chunk, m
// positions from the next lane group's, as pipe.cuh does -- S = 1: four
// consecutive positions of a row, S = 2: two positions of both substrates, even
// S: a pair of substrates, else one column.  The hardware serves 128 bytes of
// lanes at a time; a group of lanes costs the most distinct words in one bank.
inline int x_tile_wavefronts(int64_t pitch, int S, int cw, int m, size_t esz) {
  const bool wide = S == 1 || S == 2;
  const bool even = S == 2 || S == 4 || S == 8;
  const int width = (int)esz * (wide ? 4 : even ? 2 : 1);  // bytes a lane reads
  const int pw = cw / 2, per = std::max(1, std::min(32, 128 / width)), ncol = cw / S * S;
  int total = 0;
  for (int g = 0; g < 32; g += per) {
    std::vector<int64_t> words[32];
    size_t worst = 0;
    for (int l = g; l < std::min(32, g + per); l++) {
      int c = S == 1 ? l % pw : 2 * (l % pw);
      if (c >= ncol) c = 0;
      const int64_t byte = ((c / S) * pitch + c % S + (int64_t)(l / pw) * m * S) * (int64_t)esz;
      for (int64_t w = byte / 4; w <= (byte + width - 1) / 4; w++) {
        std::vector<int64_t> &v = words[w & 31];
        if (std::find(v.begin(), v.end(), w) == v.end()) v.push_back(w);
        worst = std::max(worst, v.size());
      }
    }
    total += (int)worst;
  }
  return total;
}

// Axis 0 (x), 1 (y) or 2 (z) of a field whose rows (nx*S elements of esz bytes) start gp elements
// apart, in tiles of cw columns and chunks of `maxm` positions: false when the warps of a tile
// exceed a CTA, a copy would be unaligned or a ring of two stages does not fit beside the constants.
inline bool pipe_shape_of(int axis, int64_t nx, int64_t ny, int64_t nz, int64_t S, size_t esz,
                          int64_t gp, int ns_most, int cw, int maxm, bool split, PipeShape &p) {
  const int n = (int)(axis == 0 ? nx : axis == 1 ? ny : nz);
  const int cpw = pipe_chunks_per_warp(cw);
  const int extra = axis == 0 ? 2 : 1;  // warps besides the consumers: producer (+ preparer)
  PipeShape q;
  q.cw = cw;
  q.split = split;
  q.m = q.maxm = maxm;
  q.T = (n + maxm - 1) / maxm;
  q.W = (q.T + cpw - 1) / cpw;
  if (q.W + extra > pipe_sm_warps(maxm)) return false;
  if (axis == 0) {
    if ((gp * (int64_t)esz) % 16 != 0 || S > cw) return false;
    if (ny * nz > (int64_t)0x7fffffff) return false;  // the kernel tracks rows in 32 bits
    q.rows_per_tile = (int)(cw / S);
    // the staged rows: gp elements each (a 16-byte multiple), at a shared-memory pitch in
    // elements that keeps every row 16-byte aligned
    const int align = (int)(16 / esz);
    int best = 1 << 30;
    for (int64_t pitch = gp; pitch <= gp + 64; pitch += align) {
      const int d = x_tile_wavefronts(pitch, (int)S, cw, q.m, esz);
      if (d < best) {
        best = d;
        q.pitch = (int)pitch;
      }
    }
    q.stage_elems = (int64_t)q.rows_per_tile * q.pitch;
    q.ntiles = (ny * nz + q.rows_per_tile - 1) / q.rows_per_tile;
  } else {
    const int64_t C = axis == 1 ? nx * S : ny * gp;
    const int nplanes = axis == 1 ? (int)nz : 1;
    // the map's stride between a line's positions must be a 16-byte multiple: y: the row
    // pitch gp; z: the plane, C = ny * gp (the inner extent C of a y map need not be)
    const int64_t lstride = axis == 1 ? gp : C;
    if ((lstride * (int64_t)esz) % 16 != 0 || C > (int64_t)0x7fffffff || nplanes > 65535)
      return false;
    // boxes of at most 256 rows; a tensor copy's shared-memory destination must be
    // 128-byte aligned, so box_rows * cw * esz is rounded up to a 128-byte multiple (rows
    // past the line's end are filled with zeros on load and skipped on store)
    q.nbox = (n + 255) / 256;
    const int rgran = cw == 24 ? (int)(16 / esz) : std::max(1, (int)(128 / ((size_t)cw * esz)));
    q.box_rows = ((n + q.nbox - 1) / q.nbox + rgran - 1) / rgran * rgran;
    if (((size_t)q.box_rows * cw * esz) % 128 != 0 || q.box_rows > 256) return false;
    q.stage_elems = (int64_t)q.nbox * q.box_rows * cw;
    q.ntiles = (int64_t)nplanes * ((C + cw - 1) / cw);
    if (q.ntiles > (int64_t)0x7fffffff) return false;  // tiles are indexed in 32 bits
  }
  const size_t stage = (size_t)q.stage_elems * esz;
  const size_t tab = (size_t)pipe_tab_pairs(maxm, (int)S, q.W, cpw, split) * 8 + 16;  // + alignment
  // carry exchange [2][W][32 / cpw] pairs; mbarriers: full, done, ready per stage, at most 8 stages
  const size_t scratch = 2 * (size_t)q.W * (32 / cpw) * 8 + 3 * 8 * 8;
  // As many CTAs per SM as the registers take, while each keeps three stages (256 positions:
  // two CTAs of 9 warps); else one with as many stages as fit.
  const int most = std::max(2, std::min(ns_most, 8));
  for (int c = std::max(1, pipe_sm_warps(maxm) / (q.W + extra)); c >= 1 && !q.stages; c--) {
    const size_t room = std::min(kMaxDynamicSmem, (kMaxDynamicSmem + 1024) / c - 1024);
    for (int ns = most; ns >= (c > 1 ? std::min(3, most) : 2) && !q.stages; ns--)
      if (ns * stage + tab + scratch <= room) {
        q.stages = ns;
        q.ctas = c;
      }
  }
  if (!q.stages) return false;
  q.smem = q.stages * stage + tab + scratch;
  p = q;
  return true;
}

// The shape of an axis; false when none fits (the other kernels then have to solve it).
//
// Tiles of 32 columns when a ring of two stages of them fits, else of 24 (y, z) or 16 (long
// lines), in chunks of exactly the capacity, the shortest whose warps fit in a CTA (the last chunk
// is shorter; positions past the line's end have zero coefficients).  48 positions (y/z) keep long
// lines on tiles of 32 or 24 columns: z sweeps read one tile row per plane, and with 16 columns,
// 64 bytes, a 1200 x 400 x 900 x 2 sweep ran at 2.5 TB/s (with 24 at 3.7).
//
// Where those rings do not fit -- an odd substrate count stages every coefficient twice -- any
// width with any capacity, and last the coefficients per substrate, which stage half as much and
// cost a ragged chunk twice the loads and the moves that pair them.
inline bool pipe_shape(int axis, int64_t nx, int64_t ny, int64_t nz, int64_t S, size_t esz,
                       int64_t gp, const PipeKnobs &knobs, PipeShape &p) {
  auto compiled = [&](int cw, int maxm) {
    return maxm == 48 ? axis != 0 && cw != 16 : cw != 24;
  };
  auto fits = [&](int cw, int maxm, bool split) {
    return pipe_shape_of(axis, nx, ny, nz, S, esz, gp, knobs.ns, cw, maxm, split, p);
  };
  const int n = (int)(axis == 0 ? nx : axis == 1 ? ny : nz), extra = axis == 0 ? 2 : 1;
  for (int cw : {32, 24, 16}) {
    if (knobs.cw && cw != knobs.cw) continue;
    for (int target : {16, 24, 48}) {
      int maxm = target;
      if (knobs.chunk > 0) {
        maxm = cw == 24 ? 48 : knobs.chunk <= 16 ? 16 : knobs.chunk <= 24 ? 24 : 48;
        if (!compiled(cw, maxm)) maxm = cw == 24 ? 48 : 24;
      }
      const int cpw = pipe_chunks_per_warp(cw), T = (n + maxm - 1) / maxm;
      if (!compiled(cw, maxm) || (T + cpw - 1) / cpw + extra > pipe_sm_warps(maxm)) continue;
      if (fits(cw, maxm, false)) return true;
      break;
    }
  }
  if (knobs.chunk > 0 || knobs.cw) {
    PipeKnobs own;
    own.ns = knobs.ns;
    return pipe_shape(axis, nx, ny, nz, S, esz, gp, own, p);
  }
  for (int cw : {32, 24, 16})
    for (int maxm : {16, 24, 48})
      if (compiled(cw, maxm) && fits(cw, maxm, false)) return true;
  for (int cw : {32, 16})
    if (pipe_can_split(S) && fits(cw, kSplitMaxm, true)) return true;
  return false;
}

}  // namespace bfv
