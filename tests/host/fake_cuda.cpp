// A CUDA runtime in host memory and stand-ins for the kernels' launchers, so
// that the library's host code (capi.cu, surrogate.cu, serve.cu) runs on a CPU.
// Device memory is malloc'd and recorded; a launcher checks that every buffer
// it is given lies in live device memory and is large enough, and counts the
// ones that do not (fake_bad) instead of touching them.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>

#include "launch.h"
#include "mlp.h"
#include "runtime.h"

namespace {

std::mutex mu;
struct Block {
  size_t bytes;
  int device;
};
std::map<char*, Block> live;
long long allocs = 0, fail_at = -1, bad = 0, in_use = 0;
long long capacity = 1LL << 40;
const void* scored_at = nullptr;

// Inside one block of live memory, of the given device (-1: of any).
bool inside(const void* p, size_t bytes, int device = -1) {
  std::lock_guard<std::mutex> lock(mu);
  char* c = (char*)p;
  auto it = live.upper_bound(c);
  if (it == live.begin()) return false;
  --it;
  return (device < 0 || it->second.device == device) && c + bytes <= it->first + it->second.bytes;
}
// A kernel of device 0 would access [p, p + bytes).
void touch(const void* p, size_t bytes) {
  if (!p || !inside(p, bytes, 0)) ++bad;
}

}  // namespace

extern "C" {
void fake_fail_alloc(long long nth) { fail_at = nth < 0 ? -1 : allocs + nth; }   // the nth allocation from now (0: the next)
long long fake_allocs() { return allocs; }
long long fake_bad() { return bad; }
const void* fake_scored_at() { return scored_at; }   // the trace that the last score kernel was given
long long fake_in_use() { return in_use; }
void fake_move(void* p, int device) { live[(char*)p].device = device; }   // as memory of another device
void fake_capacity(long long c) { capacity = c; }

cudaError_t cudaMalloc(void** p, size_t n) {
  std::lock_guard<std::mutex> lock(mu);
  if (allocs++ == fail_at || in_use + (long long)n > capacity) return cudaErrorMemoryAllocation;
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  live[(char*)*p] = Block{n, 0};
  in_use += (long long)n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::lock_guard<std::mutex> lock(mu);
  auto it = live.find((char*)p);
  if (it == live.end()) return cudaErrorInvalidValue;
  in_use -= (long long)it->second.bytes;
  live.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  if (allocs++ == fail_at) return cudaErrorMemoryAllocation;
  *p = malloc(n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *f = (size_t)(capacity - in_use);
  *t = (size_t)capacity;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  const bool to = k == cudaMemcpyHostToDevice || k == cudaMemcpyDeviceToDevice;
  const bool from = k == cudaMemcpyDeviceToHost || k == cudaMemcpyDeviceToDevice;
  if ((to && !inside(d, n)) || (from && !inside(s, n))) {
    ++bad;
    return cudaErrorInvalidValue;
  }
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void* p, int v, size_t n) {
  if (!p || !inside(p, n)) {
    ++bad;
    return cudaErrorInvalidValue;
  }
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeUnregistered;
  a->device = -2;
  if (inside(p, 1)) {
    a->type = cudaMemoryTypeDevice;
    a->device = inside(p, 1, 0) ? 0 : 1;
  }
  return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : 0;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = nullptr, cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) { return *s = cudaStreamCaptureStatusNone, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}

namespace opmm {

// ------------------------------------------------------------------ fits
cudaError_t launch_gather(const float* const* src, const DevSac* sacs, float* dst, int n, cudaStream_t) {
  touch(src, sizeof(float*) * (size_t)n);
  touch(sacs, sizeof(DevSac) * (size_t)n);
  touch(dst, 4);
  return cudaSuccess;
}
cudaError_t launch_nominal(const DevSac* sacs, int n, int, const float*, float* pc, cudaStream_t) {
  touch(sacs, sizeof(DevSac) * (size_t)n);
  touch(pc, 72 * (size_t)n);
  return cudaSuccess;
}
cudaError_t launch_simulate(const float* opc, int n, const DevSac*, const int*, const long long* off, float* out,
                            cudaStream_t, int) {
  touch(opc, 72 * (size_t)n);
  touch(off, 8 * (size_t)n);
  touch(out, 4);
  return cudaSuccess;
}
cudaError_t launch_score(const float* opc, int m, const DevSac& sac, const float* trace, float* f, int, cudaStream_t) {
  touch(opc, 72 * (size_t)m);
  touch(trace, 4 * (size_t)sac.L);
  if ((uintptr_t)trace & 3) ++bad;
  scored_at = trace;
  touch(f, 4 * (size_t)m);
  return cudaSuccess;
}
cudaError_t launch_finalize(const DevSac*, const float*, const float*, const int*, int, const float*, float, float, int n,
                            opmm_fit_result* out, cudaStream_t, const int*, int) {
  touch(out, sizeof *out * (size_t)n);
  if (inside(out, sizeof *out * (size_t)n)) memset((void*)out, 0, sizeof *out * (size_t)n);
  return cudaSuccess;
}
cudaError_t launch_refine(int, const DevSac*, const float*, const float*, const float*, int, int, float, float, float, float,
                          int, float*, opmm_fit_result*, unsigned*, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_admit(const DevSac*, const float*, const float*, const int*, int, DevSac*, float*, float*, int*, int,
                         cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_advance(const int*, int, int*, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_search_v(int, const SearchParams& P, int, int, cudaStream_t) {
  touch(P.unit_best, 4 * (size_t)kUnitRecFloats * (size_t)P.n_units);
  return cudaSuccess;
}

// The search kernel's launch shapes: simplices per group, coordinates, groups.
static const int kShapes[][4] = {{16, 18, 2, 0}, {16, 18, 2, 0}, {8, 18, 2, 0},  {32, 18, 2, 0}, {27, 9, 2, 0},
                                 {16, 18, 4, 0}, {27, 9, 4, 0},  {24, 18, 3, 0}, {16, 18, 2, 1}, {32, 18, 2, 1},
                                 {16, 18, 4, 1}, {24, 18, 3, 1}, {27, 9, 4, 1}};
int search_variant_count() { return 13; }
int search_variant_g(int v) { return kShapes[v][0] * kShapes[v][2]; }
int search_variant_groups(int v) { return kShapes[v][2]; }
int search_variant_dim(int v) { return kShapes[v][1]; }
int search_variant_minb(int) { return 1; }
int search_variant_lean(int v) { return v == 1; }
int search_variant_pack(int v) { return kShapes[v][3]; }
int search_variant_threads(int) { return 384; }
int search_variant_default(int dim, int k) { return k > 0 ? -1 : dim == 9 ? 12 : 9; }
int search_variant_for(int unit, int dim) {
  for (int v = search_variant_count() - 1; v >= 0; --v)
    if (search_variant_g(v) == unit && search_variant_dim(v) == dim) return v;
  return -1;
}
cudaError_t search_occupancy_v(int, int, int* b) { return *b = 1, cudaSuccess; }

// ------------------------------------------------------------------ network
namespace mlp {
cudaError_t gemm_prepare() { return cudaSuccess; }
cudaError_t gemm(const GemmLaunch& L, cudaStream_t) {
  for (int i = 0; i < L.np; ++i) {
    const GemmProblem& p = L.p[i];
    touch(p.A, 2 * (size_t)L.M * L.K);
    touch(p.B, 2 * (size_t)L.N * L.K);
    if (p.out_bf16) touch(p.out_bf16, 2 * (size_t)L.M * L.N);
    if (p.out_f32) touch(p.out_f32, 4 * (size_t)L.ksplit * L.M * L.N);
  }
  return cudaSuccess;
}
cudaError_t head_centres(const __nv_bfloat16* H, const __nv_bfloat16*, const float*, int n, float* pc, cudaStream_t) {
  touch(H, 2 * (size_t)n * kHidden);
  touch(pc, 4 * (size_t)n * kOut);
  return cudaSuccess;
}
cudaError_t head_train(const __nv_bfloat16* H, const __nv_bfloat16*, const float*, const float* T, const float* Z, int M,
                       float* Y, float* dY, float* row_loss, __nv_bfloat16* dZ, float*, float*, float*, int*, cudaStream_t) {
  touch(H, 2 * (size_t)M * kHidden);
  touch(T, 4 * (size_t)M * kOut);
  touch(Z, 4 * (size_t)M * kHidden);
  touch(Y, 4 * (size_t)M * kOut);
  touch(dY, 4 * (size_t)M * kOut);
  touch(row_loss, 4 * (size_t)M);
  touch(dZ, 2 * (size_t)M * kHidden);
  return cudaSuccess;
}
cudaError_t grad_finish(const FinishArgs&, cudaStream_t) { return cudaSuccess; }
cudaError_t adam_corrections(float, float, int, float* a, float* b) { return *a = *b = 1.0f, cudaSuccess; }
cudaError_t adamw(float*, const float*, float*, float*, int, float, float, float, float, float, int, const AdamLayout&,
                  __nv_bfloat16*, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t pack_params(const float*, int, const AdamLayout&, __nv_bfloat16*, cudaStream_t) { return cudaSuccess; }
cudaError_t featurize(const DevSac* sacs, const float* traces, int n, __nv_bfloat16* X, cudaStream_t) {
  touch(sacs, sizeof(DevSac) * (size_t)n);
  touch(traces, 4);
  touch(X, 2 * (size_t)n * kIn);
  return cudaSuccess;
}
cudaError_t featurize_noisy(uint64_t, const long long*, const DevSac* sacs, const float* traces, int n, float,
                            __nv_bfloat16* X, int, cudaStream_t) {
  touch(sacs, sizeof(DevSac) * (size_t)n);
  touch(traces, 4 * (size_t)n * kTrainLcap);
  touch(X, 2 * (size_t)n * kIn);
  return cudaSuccess;
}
cudaError_t bump(long long* p, long long, cudaStream_t) { return touch(p, 8), cudaSuccess; }
cudaError_t gen_desc(uint64_t, const long long*, int n, const float*, const float*, int, DevSac* sacs, float* hidden,
                     float* target, int, cudaStream_t) {
  touch(sacs, sizeof(DevSac) * (size_t)n);
  touch(hidden, 4 * (size_t)n * kOut);
  touch(target, 4 * (size_t)n * kOut);
  return cudaSuccess;
}
}  // namespace mlp

}  // namespace opmm
