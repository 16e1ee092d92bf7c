// The CUDA runtime calls and kernel launches of the host library, replaced by
// host stand-ins: device memory is host memory, launches only record their
// settings, several devices and stream captures are imitated. Linked with the
// library's host sources it shows, without a GPU, what they do with buffers,
// captures and launch settings.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>
#include <vector>

#include "octgrav_internal.h"

namespace {

struct Block {
  size_t bytes;
  int device;
};
struct Launch {
  int nparts, stage, ppl;
};
using Refs = std::vector<const void*>;  // buffers that a captured launch writes

int device;
size_t used[4], limit[4];
unsigned long long context[4];
std::map<void*, Block> live;
std::vector<Launch> launches;
int capturing, broken, frees, bad_frees, device_syncs, dangling;
Refs captured;
std::map<std::pair<int, int>, float> times;  // (parts, staging) -> ms
Launch last;

void replay(const Refs& refs) {
  for (const void* p : refs) dangling += live.find(const_cast<void*>(p)) == live.end();
}

void record(const og::KParams& p, int ppl) {
  last = {p.nparts > 1 ? p.nparts : 1, p.stage, ppl};
  launches.push_back(last);
  if (capturing && p.nparts > 1) captured.push_back(p.part_out);
}

int context_id_of(void*, unsigned long long* id) {
  *id = context[device];
  return 0;
}

}  // namespace

extern "C" {

// ---- what the tests set and read
void fake_reset() {  // new devices: what an earlier test left behind is gone with its context
  static unsigned long long contexts = 100;
  device = capturing = broken = frees = bad_frees = device_syncs = dangling = 0;
  for (int d = 0; d < 4; ++d) {
    used[d] = 0;
    limit[d] = ~size_t{0};
    context[d] = contexts++;
  }
  live.clear();
  launches.clear();
  captured.clear();
  times.clear();
}
void fake_set_device(int d) { device = d; }
void fake_set_limit(int d, size_t bytes) { limit[d] = bytes; }
void fake_set_context(int d, unsigned long long id) { context[d] = id; }
size_t fake_used(int d) { return used[d]; }
int fake_frees() { return frees; }
int fake_bad_frees() { return bad_frees; }
int fake_dangling() { return dangling; }
int fake_launches() { return static_cast<int>(launches.size()); }
void fake_launch(int k, int* nparts_stage_ppl) {
  nparts_stage_ppl[0] = launches[k].nparts;
  nparts_stage_ppl[1] = launches[k].stage;
  nparts_stage_ppl[2] = launches[k].ppl;
}
void fake_set_time(int nparts, int stage, float ms) { times[{nparts, stage}] = ms; }
// a capture of the caller's own, begun on another thread; replay returns 0 while what it holds is alive
void fake_begin_capture() {
  ++capturing;
  captured.clear();
}
int fake_end_capture() {
  --capturing;
  return broken;
}
int fake_replay() {
  replay(captured);
  return dangling;
}

// ---- CUDA runtime
cudaError_t cudaGetDevice(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 0;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
  if (bytes > limit[device] || used[device] > limit[device] - bytes) return cudaErrorMemoryAllocation;
  *p = aligned_alloc(256, (bytes + 255) & ~size_t{255});
  if (!*p) return cudaErrorMemoryAllocation;
  live[*p] = {bytes, device};
  used[device] += bytes;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  const auto it = live.find(p);
  if (it == live.end()) {
    ++bad_frees;
    return cudaErrorInvalidValue;
  }
  used[it->second.device] -= it->second.bytes;
  live.erase(it);
  free(p);
  ++frees;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  ++device_syncs;
  if (!capturing) return cudaSuccess;
  broken = 1;  // in every mode, from every thread
  return cudaErrorStreamCaptureUnsupported;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(malloc(1));
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  free(s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(malloc(1));
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free(e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  const auto it = times.find({last.nparts, last.stage});
  *ms = it == times.end() ? 1.f : it->second;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  ++capturing;
  captured.clear();
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  --capturing;
  *g = reinterpret_cast<cudaGraph_t>(new Refs(captured));
  return broken ? cudaErrorStreamCaptureInvalidated : cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(new Refs(*reinterpret_cast<Refs*>(g)));
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete reinterpret_cast<Refs*>(g);
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  delete reinterpret_cast<Refs*>(e);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  replay(*reinterpret_cast<Refs*>(e));
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(&context_id_of);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // extern "C"

// ---- launches
namespace og {

cudaError_t launch_walk_eval(const KParams& p, int ppl, int, bool, cudaStream_t, LaunchInfo*) {
  record(p, ppl);
  return cudaSuccess;
}
cudaError_t launch_walk_eval_noalloc(KParams p, int ppl, int, cudaStream_t, int* bits) {
  record(p, ppl);
  *bits = 0;
  return cudaSuccess;
}
cudaError_t prepare_walk_eval(int, int, int, int, LaunchInfo*) { return cudaSuccess; }
cudaError_t split_sum(const float4*, int, int, float4*, cudaStream_t) { return cudaSuccess; }
cudaError_t encode_mp_map(CUtensorMap*, const void*, int) { return cudaSuccess; }
cudaError_t gpu_unpermute(const float4*, const int*, int64_t, double*, double*, cudaStream_t) { return cudaSuccess; }

// not imitated
cudaError_t gpu_build(const GpuBuild&, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t gpu_build_tables(const GpuBuild&, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t gpu_build_kernels(const GpuBuild&, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t gpu_build_items(const GpuBuild&, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t gpu_refit(const GpuBuild&, cudaStream_t) { return cudaErrorNotSupported; }
size_t gpu_build_scratch_bytes(int64_t, int, int64_t) { return 256; }
cudaError_t pull_host(void*, const void*, size_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t sim_kick_drift(double*, double*, const double*, int64_t, double, double, bool, cudaStream_t) {
  return cudaErrorNotSupported;
}
cudaError_t sim_energy_partials(const double*, const double*, const double*, int64_t, double*, cudaStream_t) {
  return cudaErrorNotSupported;
}
int64_t direct_chunks(int64_t, int64_t) { return 1; }
cudaError_t direct_sum(const double*, const double*, int64_t, const int64_t*, int64_t, double, double, double*, double*,
                       double*, cudaStream_t) {
  return cudaErrorNotSupported;
}
cudaError_t mlp_sample_features(const MlpSampleArgs&, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t mlp_sample_labels(const MlpSampleArgs&, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t mlp_standardise(float*, const float*, int64_t, float*, float*, float*, cudaStream_t) {
  return cudaErrorNotSupported;
}
int mlp_blocks(int) { return 1; }
cudaError_t mlp_gradient(const float*, const float*, const float*, int, float*, float*, float*, cudaStream_t) {
  return cudaErrorNotSupported;
}
cudaError_t mlp_train_steps(float*, float*, float*, const float*, const float*, int, int, int, int, uint64_t, float,
                            const float2*, float*, float*, int*, cudaStream_t) {
  return cudaErrorNotSupported;
}

}  // namespace og
