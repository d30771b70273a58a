// A CUDA runtime and kernel launchers for the host half of the library (csrc/api.cpp) on machines
// without a GPU: device memory is host memory, copies run at once, launches are recorded and
// compute nothing.  Launchers that no test reaches are left undefined (bound lazily).
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "internal.h"
#include "pipe_args.h"
#include "pipe_plan.h"

namespace {
std::map<void *, size_t> g_mem;
long g_fail_after = -1;  // allocations until one fails (-1: none does)
int g_instantiated = 0;
struct PipeRecord {
  int mode, cw, maxm, grid, overlap;
};
std::vector<PipeRecord> g_pipe;
bfv::SrcAdjLaunch g_src_adjoint;

CUresult encode_map(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                    CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// -- what the tests ask ------------------------------------------------------------------------
void stand_in_fail_allocation(long after) { g_fail_after = after; }
int stand_in_graphs_made() { return g_instantiated; }
void stand_in_forget_launches() { g_pipe.clear(); }
int stand_in_pipe_launches(PipeRecord *out, int max) {
  for (int i = 0; i < max && i < (int)g_pipe.size(); i++) out[i] = g_pipe[i];
  return (int)g_pipe.size();
}
// The pipelined sweep's tile for an axis (gp: elements between rows): 1 and its columns, positions
// and split, or 0.
int stand_in_pipe_shape(int axis, int nx, int ny, int nz, int ns, int esz, int gp, int chunk,
                        int cw, int out[3]) {
  bfv::PipeKnobs k;
  k.chunk = chunk;
  k.cw = cw;
  bfv::PipeShape p;
  if (!bfv::pipe_shape(axis, nx, ny, nz, ns, esz, gp, k, p) || p.smem > bfv::kMaxDynamicSmem)
    return 0;
  out[0] = p.cw;
  out[1] = p.m;
  out[2] = p.split;
  return 1;
}
// The source adjoint's last launch: entries it walks, entries its map holds, the largest of them
// and the length of the list they index.
void stand_in_source_adjoint(int64_t out[4]) {
  const bfv::SrcAdjLaunch &a = g_src_adjoint;
  out[0] = a.n;
  auto it = g_mem.find(const_cast<int64_t *>(a.entry));
  out[1] = it == g_mem.end() ? 0 : (int64_t)(it->second / 8);
  out[2] = -1;
  for (int64_t i = 0; i < out[1] && i < a.n; i++) out[2] = a.entry[i] > out[2] ? a.entry[i] : out[2];
  out[3] = a.n_entries;
}

// -- runtime -----------------------------------------------------------------------------------
cudaError_t cudaMalloc(void **p, size_t n) {
  if (g_fail_after >= 0 && g_fail_after-- == 0) return *p = nullptr, cudaErrorMemoryAllocation;
  *p = malloc(n);
  g_mem[*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  g_mem.erase(p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  if (n) memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
  *p = cudaDeviceProp{};
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "an error of the stand-in"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
  g_instantiated++;
  *e = reinterpret_cast<cudaGraphExec_t>(&g_instantiated);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *r) {
  *f = reinterpret_cast<void *>(&encode_map);
  *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}

// -- launchers ---------------------------------------------------------------------------------
namespace bfv {
static cudaError_t record(const PipeArgs &a, int maxm, int grid) {
  g_pipe.push_back({a.mode, a.cw, maxm, grid, a.overlap});
  return cudaSuccess;
}
cudaError_t launch_pipe_f32(const CUtensorMap &, const PipeArgs &a, int maxm, int grid, size_t,
                            cudaStream_t) { return record(a, maxm, grid); }
cudaError_t launch_pipe_bf16(const CUtensorMap &, const PipeArgs &a, int maxm, int grid, size_t,
                             cudaStream_t) { return record(a, maxm, grid); }
cudaError_t launch_pipe_fp16(const CUtensorMap &, const PipeArgs &a, int maxm, int grid, size_t,
                             cudaStream_t) { return record(a, maxm, grid); }
cudaError_t allow_pipe_smem_f32(int, size_t) { return cudaSuccess; }
cudaError_t allow_pipe_smem_bf16(int, size_t) { return cudaSuccess; }
cudaError_t allow_pipe_smem_fp16(int, size_t) { return cudaSuccess; }
cudaError_t allow_x_smem_f32(int, size_t) { return cudaSuccess; }
cudaError_t allow_x_smem_f64(int, size_t) { return cudaSuccess; }
cudaError_t allow_stream_smem_f64() { return cudaSuccess; }
cudaError_t launch_x_f32(const XLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_x_f64(const XLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_col_f32(const ColLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_col_f64(const ColLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_stream_f32(const StreamArgs &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_stream_f64(const StreamArgs &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_adj_reduce_f32(const ReduceLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_adj_reduce_f64(const ReduceLaunch &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_src_adjoint_f32(const SrcAdjLaunch &a, cudaStream_t) {
  return g_src_adjoint = a, cudaSuccess;
}
cudaError_t launch_src_adjoint_f64(const SrcAdjLaunch &a, cudaStream_t) {
  return g_src_adjoint = a, cudaSuccess;
}
cudaError_t launch_pitch_rows(const void *, void *, int64_t, int, int, int, size_t, int,
                              cudaStream_t) { return cudaSuccess; }
}  // namespace bfv
