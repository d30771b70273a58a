// Persistent, TMA-pipelined sweep kernel for sm_103a (x, y and z sweeps).
//
// The arithmetic is the plain kernels' of sweeps.cuh -- partitioned Thomas of
// Algorithm 1 on the App. A system, FP32 in defect-correction form -- on tiles
// of CW independent lines ("columns") x n positions that move through a ring
// of shared-memory stages.  CW = 32 normally; 24 (y/z) or 16 for lines so long
// that two stages of 32 columns do not fit:
//
//   warp 0 (producer): TMA loads of tile k+NS-1 (cp.async.bulk.tensor boxes
//     for y/z tiles, issued by lane 0; one cp.async.bulk per row for x tiles,
//     the rows spread over the 32 lanes) completing on mbarrier `full`; once
//     the consumers have written tile k back into its stage (mbarrier `done`),
//     the bulk store of that tile; the stage is reloaded after the store has
//     finished reading it;
//   warp 1 (preparer, x tiles with a source update or a Dirichlet application
//     before the solve): applies them in shared memory to each tile once it
//     has landed -- running ahead of the consumers, who solve earlier tiles --
//     and arrives on mbarrier `ready`, which the consumers then wait for
//     instead of `full`;
//   the next W warps (consumers): each thread holds one chunk (MAXM positions)
//     of a PAIR of columns in registers and works on both with packed FP32
//     instructions; a warp holds two chunks (CW = 16: four) of the tile's CW/2
//     pairs (CW = 24: four lanes of each chunk's sixteen idle).  Carries cross a warp by shuffles and the CTA through shared memory,
//     between two named barriers per tile that only consumers join.
//
// What bounds it.  One column per thread, coefficients and carry weights read
// from shared memory at every position and a guard on every ragged position
// took 27 issued instructions per element and left the sweep waiting on them:
// 0.51 ms a sweep at 400^3 x 4 (4.0 TB/s).  Pairs halve the instructions,
// chunks whose coefficients have reached their interior values (all but the
// first one or two and the last of a line) read none, and running the
// recurrences again from the true carry replaces the correction passes: 16
// instructions per element, all warps of the CTA counted.  Chunks are short (16
// positions) because the four dependent chains per tile are the remaining
// latency.  Measured, x / y / z of 400^3 x 4 with 1M agents: 0.540 / 0.506 / 0.513
// ms before, 0.37 / 0.32 / 0.39 after (HBM copy rate: 0.306); the z sweep's rows
// are 128 bytes, a plane apart.
//
// The grid is persistent (tiles strided by gridDim.x), so loads of later
// tiles overlap the solve and the store of earlier ones.  The constants are
// staged once per CTA.
//
// Every mbarrier wait is bounded (mbar_wait_bounded): on a timeout the status
// word is set, the consumers agree to stop at the first carry barrier, which
// ANDs every consumer's wait outcome (no named barrier is left waiting), and
// the producer drains (bounded) the loads still in flight before the CTA exits.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "pipe_args.h"
#include "sweeps.cuh"

namespace bfv {

// Field storage H and arithmetic E: the same type, or 16-bit storage (bf16,
// fp16) with FP32 arithmetic -- values are widened on their way from the
// staged tile into registers and rounded to nearest on their way back.
template <typename E, typename H>
__device__ __forceinline__ E widen(H v) {
  if constexpr (std::is_same<H, __nv_bfloat16>::value) return __bfloat162float(v);
  else if constexpr (std::is_same<H, __half>::value) return __half2float(v);
  else return v;
}
template <typename H, typename E>
__device__ __forceinline__ H narrow(E v) {
  if constexpr (std::is_same<H, __nv_bfloat16>::value) return __float2bfloat16_rn(v);
  else if constexpr (std::is_same<H, __half>::value) return __float2half_rn(v);
  else return v;
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int c0, int c1,
                                            int c2, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, int c0, int c1, int c2,
                                             const void *src) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
          map),
      "r"(c0), "r"(c1), "r"(c2), "r"(smem_addr(src))
      : "memory");
}
__device__ __forceinline__ void bulk_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// Barrier 1 over the consumer warps only.  The non-.aligned form, after a
// __syncwarp: lanes may reach it from divergent code (ragged tiles), and the
// compiler does not treat an asm barrier as a reconvergence point.
__device__ __forceinline__ void consumers_sync(int nthreads) {
  __syncwarp();
  asm volatile("barrier.cta.sync 1, %0;" ::"r"(nthreads) : "memory");
}
// Barrier 1 over the consumers with an AND of `ok` (uniform result).
__device__ __forceinline__ bool consumers_all(bool ok, int nthreads) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)ok), "r"(nthreads)
      : "memory");
  return r != 0;
}

// Two FP32 values in one 64-bit register pair: every arithmetic instruction of
// the solve works on two columns at once (fma.rn.f32x2 and friends, sm_100+;
// each half rounds as the scalar instruction would).
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Let the stream's next kernel be scheduled, then wait for the one before this (both no-ops
// unless the launches ask for programmatic serialisation).
__device__ __forceinline__ void grid_dependency_sync() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// A thread's two columns of a staged tile, positions ps elements apart.
//   PAIR: the columns are neighbours (c, c + 1) at an even offset: one access
//         of two elements per position;
//   VEC > 1: VEC consecutive positions arrive in one access per column
//         (x tiles of one substrate: the two columns are rows) or for the pair
//         (x tiles of two);
//   otherwise two scalar accesses per position.
template <typename H, int PS, bool PAIR, int VEC>
struct ColPair {
  H *p0, *p1;  // position 0 of the thread's chunk in either column (PAIR: p1 unused)
  int ps_rt;
  __device__ __forceinline__ int ps() const { return PS > 0 ? PS : ps_rt; }
  __device__ __forceinline__ f2 one(int i) const {  // any position
    if constexpr (PAIR) {
      return load2(p0 + i * ps());
    } else {
      return f2_pack(widen<float>(p0[i * ps()]), widen<float>(p1[i * ps()]));
    }
  }
  __device__ __forceinline__ void put(int i, f2 v, bool st0, bool st1) const {
    if constexpr (PAIR) {  // (both columns are in the tile: st0 == st1)
      if (st0) store2(p0 + i * ps(), v);
    } else {
      const float2 x = f2_unpack(v);
      if (st0) p0[i * ps()] = narrow<H>(x.x);
      if (st1) p1[i * ps()] = narrow<H>(x.y);
    }
  }
  // positions i .. i+VEC-1, i a multiple of VEC (and the chunk start too)
  __device__ __forceinline__ void block(int i, f2 (&d)[VEC]) const {
    if constexpr (VEC == 1) {
      d[0] = one(i);
    } else if constexpr (PAIR) {  // PS == 2, VEC == 2
      float x[4];
      load4(p0 + i * 2, x);
      d[0] = f2_pack(x[0], x[1]);
      d[1] = f2_pack(x[2], x[3]);
    } else {  // PS == 1, VEC == 4
      float x[4], y[4];
      load4(p0 + i, x);
      load4(p1 + i, y);
#pragma unroll
      for (int k = 0; k < 4; k++) d[k] = f2_pack(x[k], y[k]);
    }
  }
  __device__ __forceinline__ void put_block(int i, const f2 (&d)[VEC], bool st0, bool st1) const {
    if constexpr (VEC == 1) {
      put(i, d[0], st0, st1);
    } else if constexpr (PAIR) {
      const float2 a = f2_unpack(d[0]), b = f2_unpack(d[1]);
      store4(p0 + i * 2, a.x, a.y, b.x, b.y);
    } else {
      float2 a[4];
#pragma unroll
      for (int k = 0; k < 4; k++) a[k] = f2_unpack(d[k]);
      store4(p0 + i, a[0].x, a[1].x, a[2].x, a[3].x);
      store4(p1 + i, a[0].y, a[1].y, a[2].y, a[3].y);
    }
  }

 private:
  static __device__ __forceinline__ f2 load2(const H *q) {
    if constexpr (std::is_same<H, float>::value) {
      return *reinterpret_cast<const f2 *>(q);
    } else if constexpr (std::is_same<H, __half>::value) {
      const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(q));
      return f2_pack(v.x, v.y);
    } else {
      const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(q));
      return f2_pack(v.x, v.y);
    }
  }
  static __device__ __forceinline__ void store2(H *q, f2 v) {
    if constexpr (std::is_same<H, float>::value) {
      *reinterpret_cast<f2 *>(q) = v;
    } else if constexpr (std::is_same<H, __half>::value) {
      const float2 x = f2_unpack(v);
      *reinterpret_cast<__half2 *>(q) = __floats2half2_rn(x.x, x.y);
    } else {
      const float2 x = f2_unpack(v);
      *reinterpret_cast<__nv_bfloat162 *>(q) = __floats2bfloat162_rn(x.x, x.y);
    }
  }
  static __device__ __forceinline__ void load4(const H *q, float (&x)[4]) {
    if constexpr (std::is_same<H, float>::value) {
      const float4 v = *reinterpret_cast<const float4 *>(q);
      x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
    } else {
      const uint2 v = *reinterpret_cast<const uint2 *>(q);
      H h[4];
      memcpy(h, &v, 8);
#pragma unroll
      for (int k = 0; k < 4; k++) x[k] = widen<float>(h[k]);
    }
  }
  static __device__ __forceinline__ void store4(H *q, float a, float b, float c, float d) {
    if constexpr (std::is_same<H, float>::value) {
      *reinterpret_cast<float4 *>(q) = make_float4(a, b, c, d);
    } else {
      const H h[4] = {narrow<H>(a), narrow<H>(b), narrow<H>(c), narrow<H>(d)};
      uint2 v;
      memcpy(&v, h, 8);
      *reinterpret_cast<uint2 *>(q) = v;
    }
  }
};

// A chunk pair's constants in shared memory (pipe_args.h).  inv(i), mul(i): inv' and mul of the
// chunk's positions i and i + 1, i even (0 past the line's end).
struct PairCoefBase {
  const f2 *K;   // interior inv' and mul; c_hi, c_lo
  const f2 *wt;  // the chunk's carry weights (kWt*)
  const f2 *pw;  // [W] products of mul over each warp's chunks
};
template <bool SPLIT>
struct PairCoef : PairCoefBase {
  const ulonglong2 *Ti, *Tm;
  __device__ __forceinline__ ulonglong2 inv(int i) const { return Ti[i / 2]; }
  __device__ __forceinline__ ulonglong2 mul(int i) const { return Tm[i / 2]; }
};
// Each substrate's coefficients on their own (odd S, where the pairs would not fit).  Four 8-byte
// loads and the pairing moves in place of two 16-byte loads, in ragged chunks only: 64 x 1256 x 64 x 3
// 94 us a step (the longest y line with pairs, 1240: 93), where other kernels took 283; 1072 x 64 x
// 64 x 5 119 (285).
template <>
struct PairCoef<true> : PairCoefBase {
  const float *Ti0, *Ti1, *Tm0, *Tm1;  // of the pair's two substrates
  __device__ __forceinline__ void at(const f2 *tab, int S, int npad, int sa, int sb, int lo) {
    const float *const t = reinterpret_cast<const float *>(tab);
    Ti0 = t + sa * npad + lo;
    Ti1 = t + sb * npad + lo;
    Tm0 = Ti0 + S * npad;
    Tm1 = Ti1 + S * npad;
  }
  static __device__ __forceinline__ ulonglong2 two(const float *a, const float *b) {
    const float2 x = *reinterpret_cast<const float2 *>(a), y = *reinterpret_cast<const float2 *>(b);
    return make_ulonglong2(f2_pack(x.x, y.x), f2_pack(x.y, y.y));
  }
  __device__ __forceinline__ ulonglong2 inv(int i) const { return two(Ti0 + i, Ti1 + i); }
  __device__ __forceinline__ ulonglong2 mul(int i) const { return two(Tm0 + i, Tm1 + i); }
};
// What a thread does with the Dirichlet application after the solve.
struct PairDir {
  bool on0, on1;    // the column's substrate is flagged
  bool face0, face1;  // the whole line lies on a face
  bool any;         // some lane of the warp has a flagged column
  float val0, val1;
};

// Chunk q of a warp (lanes q*PW ..) ends with B_q from a zero carry; the inclusive
// scan over the warp's chunks gives the end value of chunks 0..q, and the last
// one is the warp's.  The suffix scan serves the back substitution.
template <int CPW>
__device__ __forceinline__ f2 scan_fwd(f2 B, int q, const f2 *wt) {
  constexpr int PW = 32 / CPW;
#pragma unroll
  for (int d = 1, k = kWtF0; d < CPW; d <<= 1, k++) {
    const f2 B2 = __shfl_up_sync(0xffffffffu, B, d * PW);
    if (q >= d) B = f2_fma(wt[k], B2, B);
  }
  return B;
}
template <int CPW>
__device__ __forceinline__ f2 scan_bwd(f2 B, int q, const f2 *wt) {
  constexpr int PW = 32 / CPW;
#pragma unroll
  for (int d = 1; d < CPW; d <<= 1) {
    const f2 B2 = __shfl_down_sync(0xffffffffu, B, d * PW);
    if (q + d < CPW) B = f2_fma(wt[d == 1 ? kWtF0 : kWtB1], B2, B);
  }
  return B;
}

// One chunk of a column pair: e = L_N d, forward recurrence from a zero carry
// (its end only), the true carry, the forward recurrence again (kept), the same
// backward, c d + y, Dirichlet, write-back.  Running each recurrence a second
// time from the true carry costs one packed FMA per position -- the products
// pf, pb that would correct the first result cost the same FMA and a
// shared-memory load each.
// KIND kInner: MAXM positions of constant coefficients strictly inside the line;
// kFull: MAXM positions, coefficients from the tables; kRagged: any chunk.
// Returns false when a consumer's wait for the tile timed out.
enum { kInner, kFull, kRagged };
template <int MAXM, int KIND, int CPW, int VEC, typename Cols, typename Coef>
__device__ __forceinline__ bool pipe_chunk(const Cols col, const int len, const int lo,
                                           const int n, const int wc, const int W, const int q,
                                           const int p, const Coef &cf, f2 *s_end,
                                           f2 *s_beg, const int ncons, const PairDir &dir,
                                           const bool st0, const bool st1, const bool ok) {
  constexpr int PW = 32 / CPW;
  constexpr bool FAST = KIND == kInner;
  const unsigned FULL = 0xffffffffu;
  f2 v[MAXM];
  const f2 zero = 0;
  f2 g = zero;
  auto at = [&](int i) {  // position i, clamped to the line
    if (KIND == kFull && i >= 0 && i < MAXM) return col.one(i);
    return col.one(max(-lo, min(i, n - 1 - lo)));
  };
  if constexpr (FAST) {
    const f2 c0 = cf.K[0], c1 = cf.K[1];
    const f2 before = col.one(-1), after = col.one(MAXM);
#pragma unroll
    for (int i = 0; i < MAXM; i += VEC) {
      f2 b[VEC];
      col.block(i, b);
#pragma unroll
      for (int k = 0; k < VEC; k++) v[i + k] = b[k];
    }
    f2 am = f2_sub(before, v[0]);  // d_{i-1} - d_i
#pragma unroll
    for (int i = 0; i < MAXM; i++) {
      const f2 a = f2_sub(v[i], i + 1 < MAXM ? v[i + 1] : after);
      v[i] = f2_mul(f2_sub(a, am), c0);  // (d_i - d_{i-1}) + (d_i - d_{i+1})
      am = a;
      g = f2_fma(c1, g, v[i]);
    }
  } else {
    // Positions are clamped to the line: the ghost values d_{-1} = d_0 and d_n = d_{n-1} of the
    // zero-flux ends come of themselves, and what follows the line's end has zero differences
    // and zero coefficients, so that it carries nothing into the line from either side.
#pragma unroll
    for (int i = 0; i < MAXM; i++) v[i] = at(i);
    f2 am = f2_sub(at(-1), v[0]);
    const f2 after = at(MAXM);
#pragma unroll
    for (int i = 0; i < MAXM; i += 2) {
      const ulonglong2 ti = cf.inv(i), tm = cf.mul(i);
#pragma unroll
      for (int k = i; k < i + 2; k++) {
        const f2 a = f2_sub(v[k], k + 1 < MAXM ? v[k + 1] : after);
        v[k] = f2_mul(f2_sub(a, am), k == i ? ti.x : ti.y);
        am = a;
        g = f2_fma(k == i ? tm.x : tm.y, g, v[k]);
      }
    }
  }
  g = scan_fwd<CPW>(g, q, cf.wt);
  if (q == CPW - 1) s_end[wc * PW + p] = g;
  f2 prev = __shfl_up_sync(FULL, g, PW);
  // The first carry barrier also ANDs the outcome of every consumer's wait
  // for the tile: on a timeout all consumers leave together, before any
  // write-back (what they computed from the unfinished stage stays local).
  if (!consumers_all(ok, ncons)) return false;
  {
    f2 c = zero;  // what the warps before this one carry in
#pragma unroll 4
    for (int u = 0; u < wc; u++) c = f2_fma(cf.pw[u], c, s_end[u * PW + p]);
    g = q == 0 ? c : f2_fma(cf.wt[kWtFx], c, prev);
  }
  f2 x = zero;
  if constexpr (FAST) {
    const f2 c1 = cf.K[1];
#pragma unroll
    for (int i = 0; i < MAXM; i++) {
      g = f2_fma(c1, g, v[i]);
      v[i] = g;
    }
#pragma unroll
    for (int i = MAXM - 1; i >= 0; i--) x = f2_fma(c1, x, v[i]);
  } else {
#pragma unroll
    for (int i = 0; i < MAXM; i += 2) {
      const ulonglong2 tm = cf.mul(i);
      v[i] = f2_fma(tm.x, g, v[i]);
      g = v[i + 1] = f2_fma(tm.y, v[i], v[i + 1]);
    }
#pragma unroll
    for (int i = MAXM - 2; i >= 0; i -= 2) {
      const ulonglong2 tm = cf.mul(i);
      x = f2_fma(tm.x, f2_fma(tm.y, x, v[i + 1]), v[i]);
    }
  }
  x = scan_bwd<CPW>(x, q, cf.wt);
  if (q == 0) s_beg[wc * PW + p] = x;
  prev = __shfl_down_sync(FULL, x, PW);
  consumers_sync(ncons);
  {
    f2 c = zero;
#pragma unroll 4
    for (int u = W - 1; u > wc; u--) c = f2_fma(cf.pw[u], c, s_beg[u * PW + p]);
    x = q == CPW - 1 ? c : f2_fma(cf.wt[kWtBx], c, prev);
  }
  // No barrier before the write-back: the only reads of other chunks' positions
  // (the halos of e = L_N d) happen before the first barrier above, and the
  // carry arrays are rewritten only after barriers every warp has passed.
  const f2 chi = cf.K[2], clo = cf.K[3];
  auto with_dir = [&](f2 r, bool end) {
    float2 a = f2_unpack(r);
    if (dir.on0 && (dir.face0 || end)) a.x = dir.val0;
    if (dir.on1 && (dir.face1 || end)) a.y = dir.val1;
    return f2_pack(a.x, a.y);
  };
  if constexpr (FAST) {
    const f2 c1 = cf.K[1];
    auto finish = [&](auto dirc) {
#pragma unroll
      for (int i = MAXM - VEC; i >= 0; i -= VEC) {
        f2 d[VEC];
        col.block(i, d);
#pragma unroll
        for (int k = VEC - 1; k >= 0; k--) {
          x = f2_fma(c1, x, v[i + k]);
          d[k] = f2_fma(chi, d[k], f2_fma(clo, d[k], x));  // c_hi d + (c_lo d + y)
          if constexpr (decltype(dirc)::value) d[k] = with_dir(d[k], false);
        }
        col.put_block(i, d, st0, st1);
      }
    };
    if (dir.any) finish(std::true_type{}); else finish(std::false_type{});
  } else {
    auto finish = [&](auto dirc) {
#pragma unroll
      for (int i = MAXM - 2; i >= 0; i -= 2) {
        const ulonglong2 tm = cf.mul(i);
#pragma unroll
        for (int k = i + 1; k >= i; k--) {
          x = f2_fma(k == i ? tm.x : tm.y, x, v[k]);
          const f2 d = at(k);
          f2 r = f2_fma(chi, d, f2_fma(clo, d, x));
          if constexpr (decltype(dirc)::value)
            r = with_dir(r, lo + k == 0 || lo + k == n - 1);
          col.put(k, r, st0 && (KIND == kFull || k < len), st1 && (KIND == kFull || k < len));
        }
      }
    };
    if (dir.any) finish(std::true_type{}); else finish(std::false_type{});
  }
  return true;
}

// MODE 0: x tiles (per-row bulk copies, Src and B before the solve);
// MODE 1: y/z tiles (tensor boxes).  PSX > 0 (x tiles only): the substrate
// count S, known at compile time, so the staged positions (S apart) need no
// per-access address arithmetic; 0: S read at run time.  CW: columns per tile
// (32, or 24 or 16 for long lines).  SPLIT: coefficients staged per substrate.  H: the field's storage type (E, or bf16 / fp16
// with E = float): stages and TMA copies hold H, registers and constants E.
template <int MAXM, int MODE, int PSX = 0, int CW = 32, typename H = float, bool SPLIT = false>
__global__ void __maxnreg__(pipe_regs(MAXM))
    sweep_pipe_kernel(const __grid_constant__ CUtensorMap map, const PipeArgs a) {
  static_assert(CW == 32 || CW == 24 || CW == 16, "tiles of 32, 24 or 16 columns");
  typedef float E;
  constexpr int CPW = pipe_chunks_per_warp(CW);
  constexpr int PW = 32 / CPW;    // lanes of a chunk, one per column pair (CW = 24: four idle)
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int T = a.tab.T, n = a.n, S = a.S, NS = a.stages;
  const int64_t stage_elems = a.stage_elems;
  const int W = (T + CPW - 1) / CPW;  // consumer warps
  const int ncls = pipe_classes(S), npad = pipe_npad(W * CPW * MAXM);
  H *stage0 = reinterpret_cast<H *>(smem_raw);
  // constants (pipe_tab_pairs), 16-byte aligned after the stages: offset arithmetic on the shared
  // array itself (a pointer rounded through an integer would hide from the compiler that what is
  // derived from it lives in shared memory, turning its loads into generic ones)
  f2 *tab = reinterpret_cast<f2 *>(smem_raw + ((size_t)NS * stage_elems * sizeof(H) + 15) / 16 * 16);
  const int ntab = pipe_tab_pairs(MAXM, S, W, CPW, SPLIT);
  f2 *s_end = tab + ntab;   // [W][PW] warp ends (forward)
  f2 *s_beg = s_end + W * PW;  // [W][PW] warp starts (backward)
  uint64_t *full = reinterpret_cast<uint64_t *>(s_beg + W * PW);
  uint64_t *done = full + NS;
  uint64_t *ready = done + NS;  // x tiles with a preparation: the stage is prepared

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // (the planner keeps tile, row and column counts below 2^31)
  const int first = blockIdx.x;
  const int count = ((int)a.ntiles - first + (int)gridDim.x - 1) / (int)gridDim.x;
  const int ncons = W * 32;
  H *field = static_cast<H *>(a.field);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&done[s], W);
      mbar_init(&ready[s], 1);
    }
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  {
    const f2 *gT = static_cast<const f2 *>(a.tab.tabT);
    for (int q = threadIdx.x; q < ntab; q += blockDim.x) tab[q] = __ldg(gT + q);
  }
  __syncthreads();
  // Launched with programmatic serialisation: everything above ran while the kernel before it
  // finished; its results are visible from here on.  (The next kernel of the stream may be
  // scheduled from now on; it waits here in its turn.)
  grid_dependency_sync();

  // x tiles: Src and B before the solve, applied by warp 1 (the preparer) when
  // the launch has one (a.prep_warp: the host sets it exactly when there is a
  // source update or a Dirichlet application before the solve)
  const bool prep = MODE == 0 && a.prep_warp != 0;
  const bool srcs = prep && (a.flags & kSrc) && a.has_src;
  const bool dirb = prep && (a.flags & kDirBefore);
  const int cons0 = prep ? 2 : 1;  // first consumer warp
  // A tile with more source entries than the preparer holds prefetched (32 * kPF: dense agents)
  // gets its Src and B from all the consumers instead, before its solve.  Preparer and
  // consumers decide from the tile's entry count in the row offsets (read-only global data),
  // so they always agree, whatever the outcome of any wait.
  constexpr int kPF = 8;
  auto tile_range = [&](long long kk, long long &e0, long long &e1) {
    e0 = e1 = 0;
    if (!srcs || kk >= count) return;
    const long long r0 = (first + kk * gridDim.x) * a.rows_per_tile;
    e0 = __ldg(a.src_row_off + r0);
    e1 = __ldg(a.src_row_off + min(r0 + (long long)a.rows_per_tile, (long long)a.nrows));
  };
  auto is_dense = [&](long long e0, long long e1) { return e1 - e0 > 32 * kPF; };
  // B before the solve on a tile's staged rows: warp w of nw takes rows w, w + nw, ...; the
  // lanes walk a face row (a lane's substrate is fixed when S divides 32: flag and value once)
  auto dir_rows = [&](H *sg, long long r0, int rows, int w, int nw) {
    const bool lane_s = 32 % S == 0;
    const bool on_l = lane_s && a.dir_on[lane % S];
    const H val_l = on_l ? narrow<H>(dir_value<E>(a.flags, a.dir_val, lane % S)) : H(0);
    for (int rr = w; rr < rows; rr += nw) {
      const uint32_t row = (uint32_t)r0 + (uint32_t)rr;
      const int z = (int)(row / (uint32_t)a.ny), y = (int)row - z * a.ny;
      H *trow = sg + (size_t)rr * a.pitch;
      if (y == 0 || y == a.ny - 1 || z == 0 || z == a.nz - 1) {
        if (lane_s) {
          if (on_l)
            for (int q = lane; q < a.rowlen; q += 32) trow[q] = val_l;
        } else {
          for (int q = lane; q < a.rowlen; q += 32) {
            const int ss = q % S;
            if (a.dir_on[ss]) trow[q] = narrow<H>(dir_value<E>(a.flags, a.dir_val, ss));
          }
        }
      } else {
        for (int q = lane; q < 2 * S; q += 32) {
          const int ss = q % S;
          if (a.dir_on[ss])
            trow[q < S ? ss : (a.nx - 1) * S + ss] = narrow<H>(dir_value<E>(a.flags, a.dir_val, ss));
        }
      }
    }
  };

  if (warp == 0) {  // ------------------------------------------------ producer
    // x tiles: up to 32 rows per tile, one bulk copy each, issued by the lanes
    // in parallel (one thread issuing them in turn bounds the short-row tiles);
    // y/z tiles: one or two tensor boxes, lane 0 alone.  Each lane waits for
    // the stage itself (its own acquire of the consumers' writes) and for its
    // own stores; the lanes agree on the outcome of every bounded wait.
    constexpr unsigned pmask = MODE == 0 ? 0xffffffffu : 1u;
    if (MODE != 0 && lane != 0) return;
    auto rows_of = [&](long long tile) {
      const long long r0 = tile * a.rows_per_tile;
      return (int)min((long long)a.rows_per_tile, a.nrows - r0);
    };
    auto issue_load = [&](long long k, int s) {
      const long long tile = first + k * gridDim.x;
      H *dst = stage0 + s * stage_elems;
      if constexpr (MODE == 0) {
        const int rows = rows_of(tile);
        const uint32_t rb = (uint32_t)(a.gpitch * sizeof(H));
        // the expected bytes before any copy is issued: the phase cannot
        // complete while the producer's own arrival is pending
        if (lane == 0) mbar_arrive_expect_tx(&full[s], rb * rows);
        __syncwarp();
        for (int r = lane; r < rows; r += 32)
          bulk_g2s(dst + (size_t)r * a.pitch, field + (tile * a.rows_per_tile + r) * a.gpitch, rb,
                   &full[s]);
      } else {
        const int plane = (int)((uint32_t)tile / (uint32_t)a.tiles_per_plane);
        const int c0 = (int)((uint32_t)tile % (uint32_t)a.tiles_per_plane) * CW;
        mbar_arrive_expect_tx(&full[s], (uint32_t)(stage_elems * sizeof(H)));
        for (int b = 0; b < a.nbox; b++)
          tma_load_3d(dst + (size_t)b * a.box_rows * CW, &map, c0, b * a.box_rows, plane, &full[s]);
      }
    };
    auto issue_store = [&](long long k, int s) {
      const long long tile = first + k * gridDim.x;
      const H *src = stage0 + s * stage_elems;
      if constexpr (MODE == 0) {
        const int rows = rows_of(tile);
        const uint32_t rb = (uint32_t)(a.gpitch * sizeof(H));
        for (int r = lane; r < rows; r += 32)
          bulk_s2g(field + (tile * a.rows_per_tile + r) * a.gpitch, src + (size_t)r * a.pitch, rb);
      } else {
        const int plane = (int)((uint32_t)tile / (uint32_t)a.tiles_per_plane);
        const int c0 = (int)((uint32_t)tile % (uint32_t)a.tiles_per_plane) * CW;
        for (int b = 0; b < a.nbox; b++)
          tma_store_3d(&map, c0, b * a.box_rows, plane, src + (size_t)b * a.box_rows * CW);
      }
      bulk_commit();
    };
    const long long pre = count < NS ? count : NS;
    for (long long k = 0; k < pre; k++) issue_load(k, (int)k);
    long long k = 0;
    bool ok = true;
    for (; k < count; k++) {
      const int s = (int)(k % NS);
      ok = mbar_wait_bounded(&done[s], (uint32_t)((k / NS) & 1), a.status);
      if (!__all_sync(pmask, ok)) {
        ok = false;
        break;
      }
      issue_store(k, s);
      if (k + NS < count) {
        bulk_wait_read_all();  // the stage is free once every lane's store has read it
        __syncwarp(pmask);
        issue_load(k + NS, s);
      }
    }
    if (!ok && lane == 0) {  // drain the loads still in flight (bounded) before exiting
      for (long long j = k; j < count && j < k + NS; j++)
        mbar_wait_bounded(&full[j % NS], (uint32_t)((j / NS) & 1), a.status);
    }
    bulk_wait_all();
    return;
  }

  if (prep && warp == 1) {  // ---------------------------------------- preparer
    constexpr unsigned pmask = 0xffffffffu;
    // Src then B on tile kk's stage once it has landed (x tiles), then `ready`.
    // The source entries are unique elements (aggregated on the host or the
    // device), so the lanes update them independently.  They flow ahead of the
    // tiles: the entry range of a tile is loaded two preparations before its
    // own, its first 32*PF entries (PF per lane) one preparation before, so a
    // preparation waits on global memory only for a tile with more entries.
    // The Dirichlet rows follow the sources (a source can sit on a face).
    constexpr int PF = kPF;
    int2 prc[PF];
    E pal[PF], psc[PF];
    long long pe0 = 0, pe1 = 0, qe0 = 0, qe1 = 0;  // entry ranges: the next tile, the one after
    auto fetch_entries = [&]() {
#pragma unroll
      for (int j = 0; j < PF; j++) {
        const long long e = pe0 + lane + 32 * j;
        const bool v = e < pe1 && !is_dense(pe0, pe1);
        prc[j] = v ? __ldg(a.src_rowcol + e) : make_int2(-1, 0);
        pal[j] = v ? ldg<E>(a.src_alpha, e) : E(0);
        psc[j] = v ? ldg<E>(a.src_scale, e) : E(0);
      }
    };
    if (srcs) {
      tile_range(0, pe0, pe1);
      fetch_entries();
      tile_range(1, qe0, qe1);
    }
    auto prepare = [&](long long kk) -> bool {
      const int s = (int)(kk % NS);
      bool okw = mbar_wait_bounded(&full[s], (uint32_t)((kk / NS) & 1), a.status);
      if (!__all_sync(pmask, okw)) return false;
      H *const sg = stage0 + s * stage_elems;
      const long long r0 = (first + kk * gridDim.x) * a.rows_per_tile;
      const int rows = (int)min((long long)a.rows_per_tile, a.nrows - r0);
      const bool dense = srcs && is_dense(pe0, pe1);  // then the consumers prepare the tile
      if (srcs) {
        if (!dense) {
#pragma unroll
          for (int j = 0; j < PF; j++)
            if (prc[j].x >= 0) {
              H *q = sg + (prc[j].x - r0) * a.pitch + prc[j].y;
              *q = narrow<H>((widen<E>(*q) + pal[j]) * psc[j]);
            }
          __syncwarp();
        }
        pe0 = qe0;  // the next tile's entries, the range of the one after it
        pe1 = qe1;
        fetch_entries();
        tile_range(kk + 2, qe0, qe1);
      }
      if (dirb && !dense) {
        dir_rows(sg, r0, rows, 0, 1);
        __syncwarp();
      }
      if (lane == 0) mbar_arrive(&ready[s]);  // release: the warp's writes, ordered by __syncwarp
      return true;
    };
    for (long long k = 0; k < count; k++)
      if (!prepare(k)) break;  // (a timeout: the consumers' bounded wait on `ready` ends too)
    return;
  }

  // ---------------------------------------------------------------- consumers
  const int wc = warp - cons0;          // consumer warp
  const int p = lane % PW, q = lane / PW;  // column pair, chunk of the warp
  const int t = wc * CPW + q;              // chunk (t >= T: none)
  // x tiles of one substrate pair row p with row p + PW (consecutive lanes then read
  // consecutive rows, whose 16-byte accesses hit distinct banks); all others pair neighbours
  constexpr bool kRowPairs = MODE == 0 && PSX == 1;
  const int col0 = kRowPairs ? p : 2 * p, col1 = kRowPairs ? p + PW : 2 * p + 1;
  const int lo = t * MAXM;
  const int len = max(0, min(MAXM, n - lo));  // (0: a lane without a chunk)
  // columns of the stage: an x tile of rows_per_tile * S < CW columns leaves lanes without one,
  // which work on column 0 and store nothing
  const int ncol = MODE == 0 ? a.rows_per_tile * S : CW;
  const bool st0 = col0 < ncol, st1 = col1 < ncol;
  auto offset = [&](int c) {
    if (c >= ncol) c = 0;
    return MODE == 0 ? (c / S) * a.pitch + c % S : c;
  };
  constexpr int PS = MODE == 0 ? PSX : CW;
  constexpr bool kPair = PS > 0 && PS % 2 == 0;
  constexpr int VEC = MODE != 0 ? 1 : PSX == 1 ? 4 : PSX == 2 ? 2 : 1;
  ColPair<H, PS, kPair, VEC> col;
  col.ps_rt = MODE == 0 ? S : CW;
  const int off0 = offset(col0) + lo * col.ps(), off1 = offset(col1) + lo * col.ps();
  // The kind of the warp's chunks.  Full chunks at a line's ends run unclamped only in 16-bit
  // fields, which the solve bounds, not HBM (320 x 256 x 288 x 4, FP16: 94-119 us a sweep, 101-132
  // clamped); in FP32 the third copy of the solve cost 1% at 400^3 x 4 and 5% over 48 ragged grids.
  constexpr bool kHasFull = !std::is_same<H, float>::value;
  const bool inner = __all_sync(0xffffffffu, len == MAXM && lo >= max(a.k0, 1) && lo + MAXM <= n - 1);
  const bool full_chunks = kHasFull && __all_sync(0xffffffffu, len == MAXM);
  const bool dir_after = (a.flags & kDirAfter) != 0;
  const int ctid = threadIdx.x - 32 * cons0;  // consumer thread
  long long cn0 = 0, cn1 = 0;                 // entry range of the next tile (dense check)
  if (srcs) tile_range(0, cn0, cn1);
  PairCoef<SPLIT> cf;
  PairDir dir;
  auto set_substrates = [&](int sa, int sb) {
    const int cls = S == 1 ? 0 : S % 2 == 0 ? sa / 2 : sa;
    cf.K = tab + cls * 4;
    const f2 *w;
    if constexpr (SPLIT) {
      cf.at(tab + 4 * ncls, S, npad, sa, sb, lo);
      w = tab + 4 * ncls + ncls * npad;
    } else {  // (each pointer from tab itself: from a common one 400^3 x 4 took 1059 us a step, so 1050)
      cf.Ti = reinterpret_cast<const ulonglong2 *>(tab + 4 * ncls + cls * npad + lo);
      cf.Tm = reinterpret_cast<const ulonglong2 *>(tab + 4 * ncls + (ncls + cls) * npad + lo);
      w = tab + 4 * ncls + 2 * ncls * npad;
    }
    cf.wt = w + (cls * (W * CPW) + t) * kWtN;
    cf.pw = w + ncls * (W * CPW) * kWtN + cls * W;
    dir.on0 = dir_after && a.dir_on[sa];
    dir.on1 = dir_after && a.dir_on[sb];
    dir.val0 = dir.on0 ? dir_value<E>(a.flags, a.dir_val, sa) : E(0);
    dir.val1 = dir.on1 ? dir_value<E>(a.flags, a.dir_val, sb) : E(0);
    dir.face0 = dir.face1 = false;
    dir.any = __any_sync(0xffffffffu, dir.on0 || dir.on1);
  };
  // A thread's substrates are the same in every tile when S divides the tile width (and, for
  // z tiles, the row pitch): its per-substrate constants are then loaded once, not per tile.
  const bool s_fixed = MODE == 0 || (CW % S == 0 && (a.mode == 1 || a.gpitch % S == 0));
  if (s_fixed) set_substrates(col0 % S, col1 % S);
  // The per-tile index arithmetic runs in 32 bits (a 64-bit division is a long
  // software sequence, and every consumer thread repeats it per tile).
  int st = -1, round = -1;  // the tile's stage, how often the ring has wrapped
  for (int k = 0; k < count; k++) {
    if (++st == NS) st = 0;
    if (st == 0) round++;
    // (a timed-out wait is acted on at the first carry barrier of the chunk
    // solve; the steps before it only touch this stage and registers)
    // (x tiles with a preparation: the preparer's `ready`, after its own wait for the data)
    const bool ok = mbar_wait_bounded(prep ? &ready[st] : &full[st], (uint32_t)(round & 1), a.status);
    const int tile = first + k * (int)gridDim.x;
    H *const stg = stage0 + st * stage_elems;
    if (srcs) {
      const long long c0 = cn0, c1 = cn1;
      tile_range(k + 1, cn0, cn1);  // the next tile's range, used one tile later
      if (is_dense(c0, c1)) {       // every consumer agrees (global data); done whatever `ok`
        const long long r0 = (long long)tile * a.rows_per_tile;
        const int rows = (int)min((long long)a.rows_per_tile, a.nrows - r0);
        constexpr int U = 4;
        for (long long eb = c0 + ctid; eb < c1; eb += (long long)ncons * U) {
          int2 rc[U];
          E al[U], sc[U];
#pragma unroll
          for (int j = 0; j < U; j++) {
            const long long e = eb + (long long)ncons * j;
            const bool v = e < c1;
            rc[j] = v ? __ldg(a.src_rowcol + e) : make_int2(-1, 0);
            al[j] = v ? ldg<E>(a.src_alpha, e) : E(0);
            sc[j] = v ? ldg<E>(a.src_scale, e) : E(0);
          }
#pragma unroll
          for (int j = 0; j < U; j++)
            if (rc[j].x >= 0) {
              H *q = stg + (rc[j].x - r0) * a.pitch + rc[j].y;
              *q = narrow<H>((widen<E>(*q) + al[j]) * sc[j]);
            }
        }
        consumers_sync(ncons);
        if (dirb) {
          dir_rows(stg, r0, rows, wc, W);
          consumers_sync(ncons);
        }
      }
    }
    if constexpr (MODE == 0) {
      if (dir.any) {  // (only the Dirichlet application after the solve needs the face)
        const uint32_t r0 = (uint32_t)(tile * a.rows_per_tile);
        auto face = [&](int c) {
          const uint32_t row = r0 + (uint32_t)(c / S);
          const int z = (int)(row / (uint32_t)a.ny), y = (int)row - z * a.ny;
          return y == 0 || y == a.ny - 1 || z == 0 || z == a.nz - 1;
        };
        dir.face0 = face(col0);
        dir.face1 = kRowPairs || PSX == 0 ? face(col1) : dir.face0;
      }
    } else {
      // columns past the field or in a row's padding hold zeros, which stay zeros or are not
      // stored; z tiles of odd rows have pairs across two rows
      const int plane = (int)((uint32_t)tile / (uint32_t)a.tiles_per_plane);
      const uint32_t cg = ((uint32_t)tile - (uint32_t)plane * (uint32_t)a.tiles_per_plane) *
                              (uint32_t)CW + (uint32_t)col0;
      if (!s_fixed || dir.any) {
        uint32_t xs = cg, y = 0;
        if (a.mode != 1) {
          y = cg / (uint32_t)a.gpitch;
          xs = cg - y * (uint32_t)a.gpitch;
        }
        if (!s_fixed) set_substrates((int)(xs % (uint32_t)S), (int)((xs + 1) % (uint32_t)S));
        if (dir.any) {
          auto face = [&](uint32_t xs, uint32_t y) {
            const bool edge = a.mode == 1 ? plane == 0 || plane == a.nz - 1
                                          : y == 0 || (int)y == a.ny - 1;
            const int x = (int)(xs / (uint32_t)S);
            return x < a.nx && (edge || x == 0 || x == a.nx - 1);
          };
          dir.face0 = face(xs, y);
          const bool next_row = a.mode != 1 && xs + 1 == (uint32_t)a.gpitch;
          dir.face1 = next_row ? face(0, y + 1) : face(xs + 1, y);
        }
      }
    }
    col.p0 = stg + off0;
    col.p1 = stg + off1;
    bool solved;
    if (kHasFull && full_chunks && !inner)
      solved = pipe_chunk<MAXM, kHasFull ? kFull : kRagged, CPW, VEC>(
          col, len, lo, n, wc, W, q, p, cf, s_end, s_beg, ncons, dir, st0, st1, ok);
    else
      solved = inner ? pipe_chunk<MAXM, kInner, CPW, VEC>(col, len, lo, n, wc, W, q, p, cf, s_end,
                                                          s_beg, ncons, dir, st0, st1, ok)
                     : pipe_chunk<MAXM, kRagged, CPW, VEC>(col, len, lo, n, wc, W, q, p, cf, s_end,
                                                           s_beg, ncons, dir, st0, st1, ok);
    if (!solved) break;
    fence_proxy_async_smem();  // generic-proxy writes -> visible to the bulk store
    __syncwarp();
    if (lane == 0) mbar_arrive(&done[st]);
  }
}

// Chunk capacities: 16 and 24 positions of 32- and 16-column tiles; y/z tiles
// of 32 and 24 columns also 48 (lines whose shorter chunks would take more warps
// than fit).  x tiles know the substrate count at compile time where it
// is 1, 2, 4 or 8 (their chunk starts must then be multiples of the positions
// one access reads: the capacity, or 0).
template <int MAXM, int CW, typename H, typename F>
cudaError_t pipe_kernels(F &&f) {  // f(x kernel for S, S), ..., f(y/z kernel, -1)
  cudaError_t e = f((const void *)sweep_pipe_kernel<MAXM, 1, 0, CW, H>, -1);
  if constexpr (MAXM <= 24) {
    if (e == cudaSuccess) e = f((const void *)sweep_pipe_kernel<MAXM, 0, 0, CW, H>, 0);
    if (e == cudaSuccess) e = f((const void *)sweep_pipe_kernel<MAXM, 0, 1, CW, H>, 1);
    if (e == cudaSuccess) e = f((const void *)sweep_pipe_kernel<MAXM, 0, 2, CW, H>, 2);
    if (e == cudaSuccess) e = f((const void *)sweep_pipe_kernel<MAXM, 0, 4, CW, H>, 4);
    if (e == cudaSuccess) e = f((const void *)sweep_pipe_kernel<MAXM, 0, 8, CW, H>, 8);
  }
  return e;
}
// The tiles of `split` coefficients (odd S).
template <int CW, typename H, typename F>
cudaError_t pipe_split_kernels(F &&f) {
  const cudaError_t e = f((const void *)sweep_pipe_kernel<kSplitMaxm, 1, 0, CW, H, true>, -1);
  return e != cudaSuccess ? e
                          : f((const void *)sweep_pipe_kernel<kSplitMaxm, 0, 0, CW, H, true>, 0);
}
// The second tile width of a capacity.
constexpr int pipe_narrow(int maxm) { return maxm <= 24 ? 16 : 24; }

template <int MAXM, typename H>
cudaError_t allow_pipe_smem(size_t bytes) {
  auto set = [&](const void *k, int) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  cudaError_t e = pipe_kernels<MAXM, 32, H>(set);
  if (e == cudaSuccess) e = pipe_kernels<MAXM, pipe_narrow(MAXM), H>(set);
  if constexpr (MAXM == kSplitMaxm) {
    if (e == cudaSuccess) e = pipe_split_kernels<32, H>(set);
    if (e == cudaSuccess) e = pipe_split_kernels<16, H>(set);
  }
  return e;
}

template <int MAXM, int CW, typename H>
cudaError_t launch_pipe_cw(const CUtensorMap &map, const PipeArgs &a, int grid, size_t smem,
                           cudaStream_t st) {
  constexpr int CPW = pipe_chunks_per_warp(CW);
  const int threads = ((a.tab.T + CPW - 1) / CPW + 1 + a.prep_warp) * 32;
  if (threads > 32 * pipe_sm_warps(MAXM)) return cudaErrorInvalidConfiguration;
  const int psx = (a.S == 1 || a.S == 2 || a.S == 4 || a.S == 8) ? a.S : 0;
  void *args[] = {const_cast<CUtensorMap *>(&map), const_cast<PipeArgs *>(&a)};
  const void *k = nullptr;
  const int want = a.mode != 0 ? -1 : psx;
  auto pick = [&](const void *f, int s) {
    if (s == want) k = f;
    return cudaSuccess;
  };
  if (a.split) {
    if constexpr (MAXM == kSplitMaxm) pipe_split_kernels<CW, H>(pick);
  } else {
    pipe_kernels<MAXM, CW, H>(pick);
  }
  if (!k) return cudaErrorInvalidConfiguration;
  // a.overlap: the launch latency and the staging of the constants overlap the end of the kernel
  // before.
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = a.overlap ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, k, args);
}

template <int MAXM, typename H>
cudaError_t launch_pipe_one(const CUtensorMap &map, const PipeArgs &a, int grid, size_t smem,
                            cudaStream_t st) {
  if (a.cw == 32) return launch_pipe_cw<MAXM, 32, H>(map, a, grid, smem, st);
  if (a.cw == pipe_narrow(MAXM))
    return launch_pipe_cw<MAXM, pipe_narrow(MAXM), H>(map, a, grid, smem, st);
  return cudaErrorInvalidConfiguration;
}

}  // namespace bfv
