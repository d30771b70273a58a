// Adjoint (reverse-mode) kernels of the LOD step, derived from the forward
// stages:  rho+ = B Z^-1 B Y^-1 B X^-1 B Src(rho).
//
// Each 1D matrix A = (1 + lambda dt/3) I + r L_N is symmetric, so A^-T = A^-1
// and the adjoint sweeps are the forward sweep kernels run on the adjoint
// field in reverse order (Z, Y, X); B's adjoint zeroes the Dirichlet faces
// (kMaskZero).  For a sweep u = A^-1 d with adjoint mu = A^-1 ubar,
//     dL/dlambda_s += -(dt/3)      * sum_{elements of s} mu * u
//     dL/dD_s      += -(dt/dx^2)   * sum_{lines of s} sum_i (mu_{i+1}-mu_i)(u_{i+1}-u_i)
// (L_N = G^T G with G the first difference).  These sums are reduced to
// FP64's precision (ff_add for FP32 fields) in a fixed order -- per-block
// partials, then one block over the partials -- so repeated runs give
// bit-identical gradients.
//
// Src: u1 = (u0 + alpha) / (1 + beta) per element, alpha = sum_k dt w_k S_k
// rho*_k, beta = sum_k dt w_k (S_k + U_k).  Hence du1/du0 = 1/(1+beta) and,
// for agent k in that voxel, du1/dS_k = dt w_k (rho*_k - u1) / (1 + beta) and
// du1/dU_k = -dt w_k u1 / (1 + beta).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace bfv {

// A float as a double by integer instructions (the conversion runs on the FP64
// pipe, two lanes a clock and SM); infinities and NaN take the conversion.
__device__ __forceinline__ double widen_f64(float v) {
  const unsigned b = __float_as_uint(v), mag = b & 0x7fffffffu;
  if (mag - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((b & 0x80000000u) | ((mag >> 3) + 0x38000000u)),
                            (int)(mag << 29));
  return (double)v;
}

constexpr int kFF = 8;  // elements added in floats at a time

// Sums of eight products in floats, to no fewer bits than FP64 gives:
//   s1 += sum a c,   s2 += sum (b - a)(d - c)
// Every product and every difference enters as a pair of floats that is exactly it (Knuth's
// two-sum, the FMA's exact product error), and the pairs are added to three floats (FSum): the sum
// of the first two is exact, the third collects rounding errors, about 2^-70 of the sum of the
// terms' sizes.  Per group, FP64 then rounds twice where eight FP64 FMAs round eight times.
//
// The operands are scaled by powers of two to a largest size in [1, 2), so nothing overflows.
// What may be lost at the other end, scaled operands below 2^-149 and products and product
// errors below it, is less than 2^-142 in either sum, 2^-62 of a sum of at least 2^-80; and it is
// nothing when the operands' sizes span so little that every product is a multiple of 2^-149.
// Groups that are neither, or not finite, are added in FP64.
struct FSum {
  float h = 0.f, m = 0.f, l = 0.f;
  static __device__ __forceinline__ float two_sum(float &s, float x) {  // the error
    const float t = __fadd_rn(s, x), v = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(x, v));
    s = t;
    return e;
  }
  __device__ __forceinline__ void add(float x) { add_small(two_sum(h, x)); }
  __device__ __forceinline__ void add_small(float x) { l = __fadd_rn(l, two_sum(m, x)); }
  __device__ __forceinline__ double value() const {
    return widen_f64(h) + (widen_f64(m) + widen_f64(l));
  }
};
__device__ __forceinline__ float ff_two_diff(float x, float y, float &err) {
  const float s = __fsub_rn(x, y), t = __fsub_rn(s, x);
  err = __fsub_rn(__fsub_rn(x, __fsub_rn(s, t)), __fadd_rn(y, t));
  return s;
}
// The power of two that brings `top` to [1, 2) (subnormals: as far as one goes), as its exponent.
__device__ __forceinline__ int ff_exponent(float top) {
  return min((int)(__float_as_uint(top) >> 23), 253) - 127;
}
// again(k, x, y, z, w): reads element k's a, b, c, d once more (the rare path; keeping them would take
// 32 registers) and says whether it has a difference (the last of a line has none: b = a, d = c
// there, but inf - inf would be NaN).
template <typename Again>
__device__ __forceinline__ void ff_add(const float (&a)[kFF], const float (&b)[kFF],
                                       const float (&c)[kFF], const float (&d)[kFF], Again &&again,
                                       double &s1, double &s2) {
  float ta = 0.f, tc = 0.f;
#pragma unroll
  for (int k = 0; k < kFF; k++) {
    ta = fmaxf(ta, fmaxf(fabsf(a[k]), fabsf(b[k])));
    tc = fmaxf(tc, fmaxf(fabsf(c[k]), fabsf(d[k])));
  }
  const int ea = ff_exponent(ta), ec = ff_exponent(tc);
  const float fa = __uint_as_float((unsigned)(127 - ea) << 23);
  const float fc = __uint_as_float((unsigned)(127 - ec) << 23);
  FSum f1, f2;
#pragma unroll
  for (int k = 0; k < kFF; k++) {
    const float x = __fmul_rn(a[k], fa), y = __fmul_rn(c[k], fc);
    float p = __fmul_rn(x, y);
    f1.add(p);
    f1.add_small(__fmaf_rn(x, y, -p));
    float de, df;
    const float dx = ff_two_diff(__fmul_rn(b[k], fa), x, de);
    const float dy = ff_two_diff(__fmul_rn(d[k], fc), y, df);
    p = __fmul_rn(dx, dy);  // (dx + de)(dy + df), four exact products but for the smallest
    const float p1 = __fmul_rn(dx, df), p2 = __fmul_rn(de, dy);
    f2.add(p);
    f2.add_small(__fmaf_rn(dx, dy, -p));
    f2.add_small(p1);
    f2.add_small(p2);
    f2.l = __fadd_rn(f2.l, __fmaf_rn(de, df, __fadd_rn(__fmaf_rn(dx, df, -p1),
                                                       __fmaf_rn(de, dy, -p2))));
  }
  const float least = fminf(fabsf(f1.h), fabsf(f2.h)), most = fabsf(f1.h) + fabsf(f2.h);
  if (!(least >= 0x1p-80f && most <= 3.4e38f)) {
    float x, y, z, w;
    unsigned la = 0xffffffffu, lc = 0xffffffffu;  // smallest sizes - 1: zeros are the largest
    auto size = [](float v) { return (__float_as_uint(v) & 0x7fffffffu) - 1u; };
#pragma unroll 1
    for (int k = 0; k < kFF; k++) {
      again(k, x, y, z, w);
      la = min(la, min(size(x), size(y)));
      lc = min(lc, min(size(z), size(w)));
    }
    // binades from the smallest nonzero operands to the largest
    const int span = (int)(__float_as_uint(ta) >> 23) - max((int)((la + 1u) >> 23), 1) +
                     (int)(__float_as_uint(tc) >> 23) - max((int)((lc + 1u) >> 23), 1);
    if (!(most <= 3.4e38f) || span > 103) {
#pragma unroll 1
      for (int k = 0; k < kFF; k++) {
        const bool diff = again(k, x, y, z, w);
        s1 = fma((double)x, (double)z, s1);
        if (diff) s2 = fma((double)y - (double)x, (double)w - (double)z, s2);
      }
      return;
    }
  }
  const double scale = __hiloint2double((1023 + ea + ec) << 20, 0);
  s1 = fma(f1.value(), scale, s1);
  s2 = fma(f2.value(), scale, s2);
}

// Positions of a line one thread walks at a time.
constexpr int kReduceSeg = 32;

// Per-block partial sums of (sum mu*u, sum dmu*du along the axis) for every
// substrate.  A thread's substrate never changes: tid < used, a multiple of S,
// and it takes items tid, tid + used, ...
//   y, z: an item is kReduceSeg consecutive positions of one line (neighbouring
//         threads take neighbouring lines), each element read and widened once;
//   x:    an item is one element; its neighbour S further on is the next lanes'.
// FP64 fields are bound by their four FP64 operations per element (4.2M
// elements: 29 us at the measured FP64 rate; one element per item with a 64-bit
// division each took 45).  FP32 fields sum eight elements at a time in three
// floats first (ff_add): 4.2M elements in 33 us along y and z and 39 along x (FP64 fields 46;
// pairs of floats, 48 bits, took 24 and 26), bound by the float instructions, about 80 an
// element.  Every element widened to FP64 took 50, with the division and four conversions 72.
// partial layout: [block][2][S].
template <typename E>
__global__ void __launch_bounds__(kReduceThreads, reduce_blocks_per_sm(sizeof(E)))
    adj_reduce_kernel(const E *__restrict__ mu, const E *__restrict__ u, long long nel, int S,
                      long long stride, int n_axis, long long used, double *__restrict__ partial) {
  __shared__ double sh[2][kReduceThreads + 32];
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double s1 = 0.0, s2 = 0.0;
  // What stands for both ends of a difference that is none: zero (FP64), or the element itself
  // (FP32, which works on the elements' pairs; ff_add sees to infinities).
  auto none = [](E v) { return sizeof(E) == 4 ? v : E(0); };
  if (tid < used && stride == S) {  // x
    const long long rowlen = (long long)n_axis * S;
    const long long step = used % rowlen;
    long long at = tid % rowlen;  // the element's place in its row
    for (long long e = tid; e < nel;) {
      E m0[kFF], m1[kFF], u0[kFF], u1[kFF], md[kFF], ud[kFF];
      const long long at0 = at, e0 = e;
#pragma unroll
      for (int k = 0; k < kFF; k++, e += used) {
        const bool ok = e < nel, next = ok && at + S < rowlen;
        m0[k] = ok ? mu[e] : E(0);
        u0[k] = ok ? u[e] : E(0);
        m1[k] = next ? mu[e + S] : none(m0[k]);
        u1[k] = next ? u[e + S] : none(u0[k]);
        md[k] = next ? m0[k] : none(m0[k]);
        ud[k] = next ? u0[k] : none(u0[k]);
        at += step;
        if (at >= rowlen) at -= rowlen;
      }
      if constexpr (sizeof(E) == 4) {
        auto again = [&](int k, E &x, E &y, E &z, E &w) {
          const long long ek = e0 + k * used;
          const bool ok = ek < nel, diff = ok && (at0 + k * step) % rowlen + S < rowlen;
          x = ok ? mu[ek] : E(0);
          z = ok ? u[ek] : E(0);
          y = diff ? mu[ek + S] : x;
          w = diff ? u[ek + S] : z;
          return diff;
        };
        ff_add(m0, m1, u0, u1, again, s1, s2);
      } else {
#pragma unroll
        for (int k = 0; k < kFF; k++) {
          s1 = fma(m0[k], u0[k], s1);
          s2 = fma(m1[k] - md[k], u1[k] - ud[k], s2);
        }
      }
    }
  } else if (tid < used) {
    const long long ncol = nel / n_axis;
    const int nseg = (n_axis + kReduceSeg - 1) / kReduceSeg;
    for (long long w = tid; w < ncol * nseg; w += used) {
      const long long seg = w / ncol, c = w - seg * ncol, plane = c / stride;
      const int i0 = (int)seg * kReduceSeg, i1 = min(n_axis, i0 + kReduceSeg);
      long long e = (plane * n_axis + i0) * stride + (c - plane * stride);
      E mp = mu[e], up = u[e];
      for (int i = i0; i < i1; i += kFF) {  // positions i .. i+7 and the one after each
        E m0[kFF], m1[kFF], u0[kFF], u1[kFF], md[kFF], ud[kFF];
#pragma unroll
        for (int k = 0; k < kFF; k++) {
          const bool ok = i + k < i1, next = ok && i + k + 1 < n_axis;
          m1[k] = next ? mu[e + (k + 1) * stride] : E(0);
          u1[k] = next ? u[e + (k + 1) * stride] : E(0);
        }
        e += kFF * stride;
#pragma unroll
        for (int k = 0; k < kFF; k++) {
          const bool ok = i + k < i1, next = ok && i + k + 1 < n_axis;
          m0[k] = ok ? mp : E(0);
          u0[k] = ok ? up : E(0);
          mp = m1[k];
          up = u1[k];
          md[k] = next ? m0[k] : none(m0[k]);
          ud[k] = next ? u0[k] : none(u0[k]);
          if (!next) {  // the line's last position (or none)
            m1[k] = none(m0[k]);
            u1[k] = none(u0[k]);
          }
        }
        if constexpr (sizeof(E) == 4) {
          auto again = [&](int k, E &x, E &y, E &z, E &w) {
            const long long ek = e + (k - kFF) * stride;
            const bool ok = i + k < i1, diff = ok && i + k + 1 < n_axis;
            x = ok ? mu[ek] : E(0);
            z = ok ? u[ek] : E(0);
            y = diff ? mu[ek + stride] : x;
            w = diff ? u[ek + stride] : z;
            return diff;
          };
          ff_add(m0, m1, u0, u1, again, s1, s2);
        } else {
#pragma unroll
          for (int k = 0; k < kFF; k++) {
            s1 = fma(m0[k], u0[k], s1);
            s2 = fma(m1[k] - md[k], u1[k] - ud[k], s2);
          }
        }
      }
    }
  }
  // Threads S apart hold the same substrate: a tree over those groups (fixed order).
  int groups = ((int)blockDim.x + S - 1) / S;
  sh[0][threadIdx.x] = s1;
  sh[1][threadIdx.x] = s2;
  if (threadIdx.x < 32) sh[0][blockDim.x + threadIdx.x] = sh[1][blockDim.x + threadIdx.x] = 0.0;
  __syncthreads();
  while (groups > 1) {
    const int half = (groups + 1) / 2;
    if ((int)threadIdx.x < (groups - half) * S) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + half * S];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + half * S];
    }
    __syncthreads();
    groups = half;
  }
  if ((int)threadIdx.x < S) {
    const int sub = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) % S);
    partial[((long long)blockIdx.x * 2 + 0) * S + sub] = sh[0][threadIdx.x];
    partial[((long long)blockIdx.x * 2 + 1) * S + sub] = sh[1][threadIdx.x];
  }
}

// One block: sum the partials and accumulate the gradients.  A warp takes one
// (sum, substrate) at a time, its lanes every 32nd block, then a shuffle tree:
// a fixed order.  One thread per substrate walking all the blocks took 65-87 us,
// longer than the sums themselves.
// (Templated on the field type only so that each precision's translation unit
// owns its instance.)
constexpr int kReduceFinalThreads = 512;
template <typename E>
__global__ void __launch_bounds__(kReduceFinalThreads)
    adj_reduce_final_kernel(const double *__restrict__ partial, int nblocks, int S,
                            double scale_lambda, double scale_D, double *dlambda, double *dD) {
  const int lane = threadIdx.x & 31;
  for (int j = threadIdx.x >> 5; j < 2 * S; j += blockDim.x >> 5) {
    double a = 0.0;
#pragma unroll 8
    for (int k = lane; k < nblocks; k += 32) a += partial[(long long)k * 2 * S + j];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
    if (lane == 0) {
      if (j < S) dlambda[j] += scale_lambda * a;
      else dD[j - S] += scale_D * a;
    }
  }
}

// Secretion and uptake gradients per (agent, substrate): one thread each, no
// reduction.  elem[k*S+s] = voxel_k*S + s; entry[k*S+s] = index of that
// element in the aggregated source list (its 1/(1+beta)), or -1 when the
// element has none.  dsec or dupt may be NULL.
template <typename E>
__global__ void src_adjoint_agents_kernel(const E *__restrict__ gbar, const E *__restrict__ u1,
                                          const int64_t *__restrict__ elem,
                                          const int64_t *__restrict__ entry,
                                          const E *__restrict__ src_scale,
                                          const double *__restrict__ weight,
                                          const double *__restrict__ target, long long n, double dt,
                                          int S, double *__restrict__ dsec,
                                          double *__restrict__ dupt) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const long long e = elem[i], ent = entry[i];
  const double scale = ent >= 0 ? (double)src_scale[ent] : 1.0;
  const double w = weight ? weight[i / S] : 1.0;
  const double gw = (double)gbar[e] * dt * w * scale, u = (double)u1[e];
  if (dsec) dsec[i] += gw * (target[i] - u);
  if (dupt) dupt[i] -= gw * u;
}

// gbar <- gbar / (1 + beta) on the elements that have a source entry.
template <typename E>
__global__ void src_adjoint_scale_kernel(E *__restrict__ gbar, const int64_t *__restrict__ src_elem,
                                         const E *__restrict__ src_scale, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) gbar[src_elem[i]] *= src_scale[i];
}

}  // namespace bfv
