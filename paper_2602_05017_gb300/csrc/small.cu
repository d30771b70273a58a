// Small grids (FP64): every step of a biofvm_step call in ONE cooperative,
// persistent launch.
//
// On a grid as small as 50^3 a step is latency-bound: each sweep kernel spends
// its time on the first loads of every line and on the serial Thomas chain,
// and three kernels per step add their launch and drain gaps.  Here one launch
// runs all the steps.  A step has three phases, the x-, y- and z-sweep (Src and
// the Dirichlet application before the x-solve fused into the first, the
// applications after each solve into each), with a grid barrier after each; in
// a phase the warps of the grid take items of adjacent lines (lines.cuh).
//
// The field is in L2 throughout.  A phase is one round of L2 loads, about 6 m
// dependent FP64 operations (m positions a chunk) and one round of stores, then
// the barrier; all SMs take part in every phase.  50^3, one substrate: 19.3 us a step
// (25.8 with planes of the field staged in shared memory for x and y together:
// 50 planes keep 50 SMs busy), 64^3 x 2: 29.7 (69.2).
//
// The barrier is grid_sync.cuh's.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "grid_sync.cuh"
#include "internal.h"
#include "lines.cuh"

namespace bfv {

namespace {

constexpr int small_threads(int maxm) { return 32 * small_warps(maxm); }

template <int MAXM, int AXIS>
__device__ __forceinline__ void small_phase(const SmallArgs &a) {
  const int lane = threadIdx.x & 31;
  const LineTab &tb = a.tab[AXIS];
  const int lpw = 32 / tb.T;
  const int lines = AXIS == 0 ? a.ny * a.nz * a.S : AXIS == 1 ? a.nz * a.nx * a.S : a.nx * a.ny * a.S;
  const int items = (lines + lpw - 1) / lpw;
  // consecutive items to a CTA (they share sectors in L1), as many to each within one
  const int it0 = (int)((long long)items * blockIdx.x / gridDim.x);
  const int it1 = (int)((long long)items * (blockIdx.x + 1) / gridDim.x);
  for (int it = it0 + (int)(threadIdx.x >> 5); it < it1; it += (int)(blockDim.x >> 5)) {
    const ItemLane L = item_lane(AXIS, it, lane, tb, a.nx, a.ny, a.nz, a.S, lines);
    ItemDir<double> none{false, false, 0.0}, dir = none;
    if (a.any_dir && L.len > 0 && a.dir_on[L.s])
      dir = ItemDir<double>{true, L.face, __ldg(a.dir_val + L.s)};
    const long long first = L.base + L.lo * L.ps;
    auto prep = [&](double(&v)[MAXM]) {
      if (AXIS == 0 && a.has_src) {
        const int r0 = it * lpw / a.S, r1 = min(a.ny * a.nz, (it * lpw + lpw - 1) / a.S + 1);
        const long long e0 = __ldg(a.src_row_off + r0), e1 = __ldg(a.src_row_off + r1);
        const long long row_first = (long long)r0 * a.nx * a.S;
        if (e1 - e0 <= kFewSources) {
          item_sources<double, MAXM>(v, e0, e1, row_first, (int)(first - row_first), L.len, a.S,
                                     lane, a.src_elem, a.src_alpha, a.src_scale);
        } else {
          item_sources_in_field<double>(a.rho, e0, e1, row_first, a.nx * a.S, r0, it * lpw, lpw,
                                        a.S, lane, a.src_elem, a.src_alpha, a.src_scale);
#pragma unroll
          for (int i = 0; i < MAXM; i++) v[i] = i < L.len ? a.rho[first + i * L.ps] : 0.0;
        }
      }
    };
    solve_item<double, MAXM>(a.rho + first, L.ps, L.len, L.lo, L.s, lane, tb, a.S,
                             AXIS == 0 ? dir : none, dir, prep);
  }
}

template <int MAXM, bool CLUSTER>
__global__ void __launch_bounds__(small_threads(MAXM), 1) small_steps_kernel(const SmallArgs a) {
  unsigned want = 0;
  for (int step = 0; step < a.n_steps; step++) {
    small_phase<MAXM, 0>(a);
    if (!grid_barrier<CLUSTER>(a.bar, want += gridDim.x, a.status)) return;
    small_phase<MAXM, 1>(a);
    if (!grid_barrier<CLUSTER>(a.bar, want += gridDim.x, a.status)) return;
    small_phase<MAXM, 2>(a);
    if (step + 1 < a.n_steps &&
        !grid_barrier<CLUSTER>(a.bar, want += gridDim.x, a.status)) return;
  }
}

}  // namespace

cudaError_t launch_small_f64(const SmallArgs &a, int maxm, int grid, int threads, bool cluster,
                             cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  if (cluster) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)grid;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  } else {
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
  }
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  switch (maxm) {
    case 8:
      return cluster ? cudaLaunchKernelEx(&cfg, small_steps_kernel<8, true>, a)
                     : cudaLaunchKernelEx(&cfg, small_steps_kernel<8, false>, a);
    case 16:
      return cluster ? cudaLaunchKernelEx(&cfg, small_steps_kernel<16, true>, a)
                     : cudaLaunchKernelEx(&cfg, small_steps_kernel<16, false>, a);
  }
  return cudaErrorInvalidValue;
}

}  // namespace bfv
