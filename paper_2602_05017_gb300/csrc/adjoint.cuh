// Adjoint (reverse-mode) kernels of the LOD step, derived from the forward
// stages:  rho+ = B Z^-1 B Y^-1 B X^-1 B Src(rho).
//
// Each 1D matrix A = (1 + lambda dt/3) I + r L_N is symmetric, so A^-T = A^-1
// and the adjoint sweeps are the forward sweep kernels run on the adjoint
// field in reverse order (Z, Y, X); B's adjoint zeroes the Dirichlet faces
// (kMaskZero).  For a sweep u = A^-1 d with adjoint mu = A^-1 ubar,
//     dL/dlambda_s += -(dt/3)      * sum_{elements of s} mu * u
//     dL/dD_s      += -(dt/dx^2)   * sum_{lines of s} sum_i (mu_{i+1}-mu_i)(u_{i+1}-u_i)
// (L_N = G^T G with G the first difference).  These sums are reduced in FP64
// in a fixed order -- per-block partials, then one block over the partials --
// so repeated runs give bit-identical gradients.
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

// A float as a double.  The conversion instruction runs on the FP64 pipe (two
// lanes a clock and SM), which the sums below already fill, so the value is
// widened by integer instructions: subnormals -- an adjoint field far from its
// sources is full of them and of zeros -- after a multiplication by 2^64.  Only
// infinities and NaN take the conversion.
__device__ __forceinline__ double widen_f64(double v) { return v; }
__device__ __forceinline__ double widen_f64(float v) {
  const bool sub = fabsf(v) < 1.17549435e-38f;  // below 2^-126
  const unsigned b = __float_as_uint(sub ? v * 18446744073709551616.0f : v);
  const unsigned mag = b & 0x7fffffffu;
  if (mag >= 0x7f800000u) return (double)v;
  const unsigned hi = mag == 0u ? 0u : (mag >> 3) + (sub ? 0x34000000u : 0x38000000u);
  return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(mag << 29));
}

// Positions of a line one thread walks at a time.
constexpr int kReduceSeg = 32;

// Per-block partial sums of (sum mu*u, sum dmu*du along the axis) for every
// substrate.  A thread's substrate never changes: tid < used, a multiple of S,
// and it takes items tid, tid + used, ...
//   y, z: an item is kReduceSeg consecutive positions of one line (neighbouring
//         threads take neighbouring lines), each element read and widened once;
//   x:    an item is one element; its neighbour S further on is the next lanes'.
// Bound by its four FP64 operations per element (4.2M elements: 29 us at the
// measured FP64 rate).  One element per item with a 64-bit division each and two
// conversions more took 45 us (FP64 fields) and 72 us (FP32).
// partial layout: [block][2][S].
template <typename E>
__global__ void __launch_bounds__(kReduceThreads)
    adj_reduce_kernel(const E *__restrict__ mu, const E *__restrict__ u, long long nel, int S,
                      long long stride, int n_axis, long long used, double *__restrict__ partial) {
  __shared__ double sh[2][kReduceThreads + 32];
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double s1 = 0.0, s2 = 0.0;
  if (tid < used && stride == S) {  // x
    const long long rowlen = (long long)n_axis * S;
    const long long step = used % rowlen;
    long long at = tid % rowlen;  // the element's place in its row
#pragma unroll 4
    for (long long e = tid; e < nel; e += used) {
      const double m0 = widen_f64(mu[e]), u0 = widen_f64(u[e]);
      s1 = fma(m0, u0, s1);
      if (at + S < rowlen)
        s2 = fma(widen_f64(mu[e + S]) - m0, widen_f64(u[e + S]) - u0, s2);
      at += step;
      if (at >= rowlen) at -= rowlen;
    }
  } else if (tid < used) {
    const long long ncol = nel / n_axis;
    const int nseg = (n_axis + kReduceSeg - 1) / kReduceSeg;
    for (long long w = tid; w < ncol * nseg; w += used) {
      const long long seg = w / ncol, c = w - seg * ncol, plane = c / stride;
      const int i0 = (int)seg * kReduceSeg, i1 = min(n_axis, i0 + kReduceSeg);
      long long e = (plane * n_axis + i0) * stride + (c - plane * stride);
      double m0 = widen_f64(mu[e]), u0 = widen_f64(u[e]);
      int i = i0 + 1;
      for (; i + 8 <= i1; i += 8) {
        E mb[8], ub[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
          mb[k] = mu[e + (k + 1) * stride];
          ub[k] = u[e + (k + 1) * stride];
        }
        e += 8 * stride;
#pragma unroll
        for (int k = 0; k < 8; k++) {
          const double m1 = widen_f64(mb[k]), u1 = widen_f64(ub[k]);
          s1 = fma(m0, u0, s1);
          s2 = fma(m1 - m0, u1 - u0, s2);
          m0 = m1;
          u0 = u1;
        }
      }
      for (; i <= i1; i++) {  // the rest, and the difference to the next segment's first position
        s1 = fma(m0, u0, s1);
        if (i == n_axis) break;
        e += stride;
        const double m1 = widen_f64(mu[e]), u1 = widen_f64(u[e]);
        s2 = fma(m1 - m0, u1 - u0, s2);
        m0 = m1;
        u0 = u1;
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
