// host_runtime.cpp -- the CUDA runtime calls of capi.cpp on host memory, and launchers that run no
// kernel but check what the real one would address: every table a launch hands over must lie in
// a live allocation that reaches to its last entry, and every id must name a block of the pool.
// With it the C ABI's memory handling (allocation failures included) is tested without a GPU.
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <map>

#include "../../paper_1204_5849_gb300/csrc/map_internal.hpp"

using namespace mapgb;

namespace {

std::map<char*, size_t> live;      // device allocations
long long allocs = 0, fail_from = 0, live_bytes = 0, launches = 0, bad = 0, syncs = 0, d2h = 0;
long long graph_launches = 0;
bool capturing = false;
int pool_blocks = 0;               // pool ids below this are blocks of the pool (host_set_blocks)

cudaError_t take(void** p, size_t n) {
  *p = nullptr;
  if (fail_from && ++allocs >= fail_from) return cudaErrorMemoryAllocation;
  *p = calloc(n ? n : 1, 1);
  live[(char*)*p] = n;
  live_bytes += (long long)n;
  return cudaSuccess;
}

// [p, p + n) lies in one live allocation
bool in(const void* p, size_t n) {
  auto it = live.upper_bound((char*)p);
  if (!p || it == live.begin()) return false;
  --it;
  return (char*)p + n <= it->first + it->second;
}

template <typename X>
bool table(const X* p, size_t n) { return in(p, n * sizeof(X)); }

size_t interior(const KernelConfig& k) { return (size_t)kNV * k.nb * k.nb * (k.ndim == 3 ? k.nb : 1); }

// ids of a launch, and the largest of them (-1: a fault)
int last_id(const int* ids, int n) {
  if (n <= 0 || !table(ids, (size_t)n)) return -1;
  int m = 0;
  for (int q = 0; q < n; ++q) {
    if (ids[q] < 0 || ids[q] >= pool_blocks) return -1;
    if (ids[q] > m) m = ids[q];
  }
  return m;
}

cudaError_t launched(bool good, long long* cnt) {
  if (!capturing) ++launches;
  if (cnt) ++*cnt;
  if (!good) ++bad;
  return cudaSuccess;
}

cudaError_t step(const KernelConfig& k, const StepLaunch& L, int elem, long long* cnt) {
  const int m = last_id(L.blocks, L.nblocks);
  bool good = m >= 0 && table(L.geo, m + 1) && table(L.pushes, (size_t)(m + 1) * 27) && table(L.dyn, 1);
  if (good && L.refl) {
    good = table(L.refl, m + 1);
    const size_t slot = (size_t)2 * k.ndim * kNV * k.nb * k.nb * elem;
    for (int q = 0; good && q < L.nblocks; ++q) {
      const int s = L.refl[L.blocks[q]].slot;
      if (s >= 0) good = in(L.freg, (s + 1) * slot);
    }
  }
  return launched(good, cnt);
}

cudaError_t reflux(const KernelConfig& k, const RefluxLaunch& L, int elem, long long* cnt) {
  bool good = table(L.tasks, (size_t)L.ntasks);
  const size_t slot = (size_t)2 * k.ndim * kNV * k.nb * k.nb * elem;
  for (int q = 0; good && q < L.ntasks; ++q) {
    const RefluxTask& t = L.tasks[q];
    good = t.coarse >= 0 && t.coarse < pool_blocks && in(L.freg, (t.cslot + 1) * slot) && table(L.geo, t.coarse + 1);
    for (int f = 0; f < 6; ++f)
      for (int c = 0; c < 4; ++c)
        if (t.fslot[f][c] >= 0) good = good && in(L.freg, (t.fslot[f][c] + 1) * slot);
  }
  return launched(good, cnt);
}

cudaError_t blocks_geo(const int* ids, int n, const BlockGeo* geo, long long* cnt) {
  const int m = last_id(ids, n);
  return launched(m >= 0 && table(geo, m + 1), cnt);
}

}  // namespace

extern "C" {

// every allocation from the k-th on fails (0: none)
void host_fail_from(long long k) {
  fail_from = k;
  allocs = 0;
}
// a capture of the pool's stream by the caller, on or off
void host_set_capturing(int on) { capturing = on != 0; }
void host_set_blocks(int n) { pool_blocks = n; }
// live device bytes, launches, launches that would have addressed memory outside their tables,
// stream synchronisations, device-to-host copies, graph launches
void host_counts(long long* out) {
  const long long v[6] = {live_bytes, launches, bad, syncs, d2h, graph_launches};
  memcpy(out, v, sizeof v);
}

cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = calloc(n ? n : 1, 1);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  auto it = live.find((char*)p);
  if (it == live.end()) {
    ++bad;                                     // freed twice, or never allocated
    return cudaErrorInvalidValue;
  }
  live_bytes -= (long long)it->second;
  live.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  const void* dev = k == cudaMemcpyHostToDevice ? d : s;
  if (!in(dev, n) || !d || !s) return cudaErrorInvalidValue;
  if (k == cudaMemcpyDeviceToHost) ++d2h;
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (!in(p, n)) return cudaErrorInvalidValue;
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  ++syncs;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  free((void*)s);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  capturing = true;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  *g = (cudaGraph_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* ex, cudaGraph_t, unsigned long long) {
  *ex = (cudaGraphExec_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  ++graph_launches;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  free((void*)g);
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t ex) {
  free((void*)ex);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free((void*)e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 4 : 232448;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  return cudaErrorInvalidValue;
}

int map_cfl_dt_noalloc(const void*, int, int, int, int, const double*, const map_params*, void*, double*) {
  return MAP_EUNSUPPORTED;
}

}  // extern "C"

namespace mapgb {

#define LAUNCHERS(SFX, ELEM)                                                                                       \
  cudaError_t launch_step_##SFX(const KernelConfig& k, const StepLaunch& L, cudaStream_t, long long* c) {           \
    return step(k, L, ELEM, c);                                                                                    \
  }                                                                                                                \
  cudaError_t launch_fill_##SFX(const KernelConfig&, const FillLaunch& L, cudaStream_t, long long* c) {             \
    if (L.nblocks <= 0) return cudaSuccess;                                                                        \
    const int m = last_id(L.blocks, L.nblocks);                                                                    \
    return launched(m >= 0 && table(L.regions, (size_t)(m + 1) * 27), c);                                          \
  }                                                                                                                \
  cudaError_t launch_restrict_##SFX(const KernelConfig&, const RestrictLaunch& L, cudaStream_t, long long* c) {     \
    if (L.nparents <= 0) return cudaSuccess;                                                                       \
    const int m = last_id(L.parents, L.nparents);                                                                  \
    return launched(m >= 0 && table(L.children, (size_t)(m + 1) * 8), c);                                          \
  }                                                                                                                \
  cudaError_t launch_cfl_##SFX(const KernelConfig&, const CflLaunch& L, cudaStream_t, long long* c) {               \
    return blocks_geo(L.blocks, L.nblocks, L.geo, c);                                                              \
  }                                                                                                                \
  cudaError_t launch_flags_##SFX(const KernelConfig&, const FlagLaunch& L, cudaStream_t, long long* c) {            \
    const int m = last_id(L.blocks, L.nblocks);                                                                    \
    return launched(m >= 0 && table(L.geo, m + 1) && table(L.flags, (size_t)L.nblocks) &&                          \
                        table(L.est, (size_t)L.nblocks), c);                                                       \
  }                                                                                                                \
  cudaError_t launch_sums_##SFX(const KernelConfig&, const SumLaunch& L, cudaStream_t, long long* c) {              \
    return blocks_geo(L.blocks, L.nblocks, L.geo, c);                                                              \
  }                                                                                                                \
  cudaError_t launch_pack_##SFX(const KernelConfig& k, const PackLaunch& L, cudaStream_t, long long* c) {           \
    return launched(last_id(L.blocks, L.nblocks) >= 0 &&                                                           \
                        in(L.host_layout, L.nblocks * interior(k) * (L.staging_f32 ? 4 : 8)), c);                  \
  }                                                                                                                \
  cudaError_t launch_regrid_##SFX(const KernelConfig&, const RegridLaunch& L, cudaStream_t, long long* c) {         \
    return launched(table(L.tasks, (size_t)L.ntasks), c);                                                          \
  }                                                                                                                \
  cudaError_t launch_reflux_##SFX(const KernelConfig& k, const RefluxLaunch& L, cudaStream_t, long long* c) {       \
    return reflux(k, L, ELEM, c);                                                                                  \
  }                                                                                                                \
  cudaError_t launch_conduction_##SFX(const KernelConfig&, const CondLaunch& L, cudaStream_t, long long* c) {       \
    return blocks_geo(L.blocks, L.nblocks, L.geo, c);                                                              \
  }                                                                                                                \
  int cond_loop_capacity_##SFX(const KernelConfig&, int) { return 0; }                                             \
  cudaError_t launch_cond_loop_##SFX(const KernelConfig&, const CondLoopLaunch&, cudaStream_t, long long*) {        \
    return cudaErrorInvalidValue;                                                                                  \
  }                                                                                                                \
  size_t step_smem_##SFX(const KernelConfig&, int, int) { return 1; }

LAUNCHERS(f64, 8)
LAUNCHERS(f32, 4)

#define STEP_VARIANT(NAME, ELEM)                                                                                   \
  cudaError_t launch_step_##NAME(const KernelConfig& k, const StepLaunch& L, cudaStream_t, long long* c) {          \
    return step(k, L, ELEM, c);                                                                                    \
  }
STEP_VARIANT(hllc_f64, 8)
STEP_VARIANT(hllc_f32, 4)
STEP_VARIANT(rfx_f64, 8)
STEP_VARIANT(rfx_f32, 4)
STEP_VARIANT(hllc_rfx_f64, 8)
STEP_VARIANT(hllc_rfx_f32, 4)
STEP_VARIANT(hlld_f64, 8)
STEP_VARIANT(hlld_f32, 4)
STEP_VARIANT(hlld_rfx_f64, 8)
STEP_VARIANT(hlld_rfx_f32, 4)

cudaError_t launch_finalize(const FinalizeLaunch& L, cudaStream_t, long long* c) {
  const bool good = table(L.dyn, (size_t)L.nprob);
  for (int q = 0; good && q < L.nprob; ++q) L.dyn[q].dt = L.dyn[q].dtc = 1e-3;
  return launched(good, c);
}
cudaError_t launch_zero_alpha(ProbDyn* dyn, int n, cudaStream_t, long long* c) { return launched(table(dyn, (size_t)n), c); }
cudaError_t launch_speeds_out(const ProbDyn*, int, double*, cudaStream_t, long long* c) { return launched(true, c); }

}  // namespace mapgb
