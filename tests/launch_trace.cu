// The host side of the solver with every kernel launch and CUDA runtime call replaced by a
// recording stand-in (device memory is host memory, launches change nothing but the decision
// that ends an increment's iterations).  Prints one line per recorded call; the checks are in
// test_launch_trace.py.  Usage: launch_trace SCENARIO [precision nx ny nz]
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>

namespace {
void rec(const char* f, ...) {
  va_list a;
  va_start(a, f);
  std::vprintf(f, a);
  std::printf("\n");
  va_end(a);
}
}  // namespace

// ---------------------------------------------------------------- runtime stand-ins --
#define cudaDeviceGetAttribute trace_cudaDeviceGetAttribute
#define cudaEventCreate trace_cudaEventCreate
#define cudaEventCreateWithFlags trace_cudaEventCreateWithFlags
#define cudaEventDestroy trace_cudaEventDestroy
#define cudaEventElapsedTime trace_cudaEventElapsedTime
#define cudaEventQuery trace_cudaEventQuery
#define cudaEventRecord trace_cudaEventRecord
#define cudaEventSynchronize trace_cudaEventSynchronize
#define cudaFree trace_cudaFree
#define cudaFreeAsync trace_cudaFreeAsync
#define cudaFreeHost trace_cudaFreeHost
#define cudaFuncSetAttribute trace_cudaFuncSetAttribute
#define cudaGetDevice trace_cudaGetDevice
#define cudaGetDeviceCount trace_cudaGetDeviceCount
#define cudaGetErrorString trace_cudaGetErrorString
#define cudaGetLastError trace_cudaGetLastError
#define cudaGraphAddNode trace_cudaGraphAddNode
#define cudaGraphConditionalHandleCreate trace_cudaGraphConditionalHandleCreate
#define cudaGraphCreate trace_cudaGraphCreate
#define cudaGraphDestroy trace_cudaGraphDestroy
#define cudaGraphExecDestroy trace_cudaGraphExecDestroy
#define cudaGraphInstantiate trace_cudaGraphInstantiate
#define cudaGraphLaunch trace_cudaGraphLaunch
#define cudaMalloc trace_cudaMalloc
#define cudaMallocFromPoolAsync trace_cudaMallocFromPoolAsync
#define cudaMallocHost trace_cudaMallocHost
#define cudaMemPoolCreate trace_cudaMemPoolCreate
#define cudaMemPoolSetAttribute trace_cudaMemPoolSetAttribute
#define cudaMemcpy trace_cudaMemcpy
#define cudaMemcpyAsync trace_cudaMemcpyAsync
#define cudaMemsetAsync trace_cudaMemsetAsync
#define cudaSetDevice trace_cudaSetDevice
#define cudaStreamBeginCaptureToGraph trace_cudaStreamBeginCaptureToGraph
#define cudaStreamCreateWithFlags trace_cudaStreamCreateWithFlags
#define cudaStreamDestroy trace_cudaStreamDestroy
#define cudaStreamEndCapture trace_cudaStreamEndCapture
#define cudaStreamGetCaptureInfo trace_cudaStreamGetCaptureInfo
#define cudaStreamIsCapturing trace_cudaStreamIsCapturing
#define cudaStreamSynchronize trace_cudaStreamSynchronize
#define cudaStreamUpdateCaptureDependencies trace_cudaStreamUpdateCaptureDependencies
#define cudaStreamWaitEvent trace_cudaStreamWaitEvent
#define OKAY { return cudaSuccess; }
static cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
static cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
static cudaError_t cudaSetDevice(int) OKAY
static cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 232448; return cudaSuccess; }
static cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(n ? n : 1, 1); return cudaSuccess; }
static cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
static cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
static cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
static cudaError_t cudaMemPoolCreate(cudaMemPool_t*, const cudaMemPoolProps*) { return cudaErrorNotSupported; }
static cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) OKAY
static cudaError_t cudaMallocFromPoolAsync(void**, size_t, cudaMemPool_t, cudaStream_t) { return cudaErrorNotSupported; }
static cudaError_t cudaFreeAsync(void*, cudaStream_t) OKAY
static cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
static cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
static cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
static cudaError_t cudaStreamSynchronize(cudaStream_t) { rec("sync"); return cudaSuccess; }
static cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)std::malloc(1); return cudaSuccess; }
static cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
static cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) OKAY
static cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) { *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
static cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) OKAY
static cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaSuccess; }
static cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus* c, unsigned long long*, cudaGraph_t*,
                                     const cudaGraphNode_t** d, const cudaGraphEdgeData**, size_t* n) {
  *c = cudaStreamCaptureStatusActive;
  *d = nullptr;
  *n = 0;
  return cudaSuccess;
}
static cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                                                unsigned) OKAY
static cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = nullptr; return cudaSuccess; }
static cudaError_t cudaGraphDestroy(cudaGraph_t) OKAY
static cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
  *h = 1;
  return cudaSuccess;
}
static cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
  static cudaGraph_t body[1] = {nullptr};
  p->conditional.phGraph_out = body;
  return cudaSuccess;
}
static cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)std::malloc(1);
  return cudaSuccess;
}
static cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { std::free(e); return cudaSuccess; }
static cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) OKAY
static cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)std::malloc(1); return cudaSuccess; }
static cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
static cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
static cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) OKAY
static cudaError_t cudaEventQuery(cudaEvent_t) OKAY
static cudaError_t cudaEventSynchronize(cudaEvent_t) OKAY
static cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
static cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) OKAY
static cudaError_t cudaGetLastError() OKAY
static const char* cudaGetErrorString(cudaError_t) { return "recorded"; }

#include "../paper_2402_09996_gb300/csrc/api.cu"

namespace {
// Where a flag of a status record lies, by name.
const char* flag_name(const IterStatus* st, const int* p) {
  if (!p) return "none";
  if (p == &st->done) return "done";
  const char* base = (const char*)st;
  return (const char*)p >= base && (const char*)p < base + sizeof(IterStatus) ? "status" : "other";
}
template <typename T>
void rec_line(const LineArgs<T>& a, int sign, const char* how, unsigned gx, unsigned gy) {
  rec("line %s sign=%d kind=%d goes_by=%s HC=%d grid=%u,%u nz=%lld", how, sign, a.side.kind,
      a.side.st ? flag_name(a.side.st, a.done) : (a.done ? "other" : "none"), a.HC, gx, gy,
      a.A ? a.A / (a.stride) : 0LL);
  if (a.side.kind == kSideResid) a.side.st->done = 1;
}
}  // namespace

namespace rve {
int x_threads() { return kXThreads; }
int line_threads() { return kLineThreads; }
int z_threads() { return kZThreads; }
template <typename T, int NP>
cudaError_t launch_xpass_np(const XArgs<T>& a, bool commit, int grid, size_t smem, cudaStream_t) {
  rec("x np=%d commit=%d L=%d grid=%d smem=%zu quad=%d", NP, (int)commit, a.L, grid, smem, a.quad);
  return cudaSuccess;
}
template <typename T, int NP>
cudaError_t launch_material_point_np(const MatDev<T>&, long long, const T*, const T*, const T*, T*, T*, T, int,
                                     const T*, cudaStream_t) OKAY
template <typename T, int NP>
cudaError_t launch_material_point_vjp_np(const MatDev<T>&, long long, const T*, const T*, const T*, const T*, T, int,
                                         const T*, T*, T*, T*, T*, T*, const T*, cudaStream_t) OKAY
template <typename T, int NP>
cudaError_t launch_adj_tangent_np(const MatDev<T>&, long long, const T*, const T*, const T*, const T*, T, int,
                                  const double*, T*, T*, T*, T*, T*, T*, const T*, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_rate_table(T*, bool, const RateGrid&, const RateGrid&, double, double, double, double, double,
                              cudaStream_t) {
  rec("rate_table");
  return cudaSuccess;
}
template <typename T>
cudaError_t launch_line(const LineArgs<T>& a, int sign, dim3 g, size_t, cudaStream_t) {
  rec_line(a, sign, "alone", g.x, g.y);
  return cudaSuccess;
}
template <typename T, int NP>
cudaError_t launch_xpass_group_np(const XGroup<T>&, bool, int, size_t, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_line_group(const LineGroup<T>& g, int sign, int, size_t, cudaStream_t) {
  for (int m = 0; m < g.n; ++m)
    rec_line(g.m[m], sign, "group", (unsigned)g.gx[m], (unsigned)((g.start[m + 1] - g.start[m]) / g.gx[m]));
  return cudaSuccess;
}
template <typename T>
cudaError_t launch_zgreen_group(const ZGroup<T>&, int, size_t, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_group_guard(const GuardGroup&, cudaGraphConditionalHandle, cudaStream_t) OKAY
template <typename T>
size_t line_group_smem(int, int) { return 0; }
template <typename T>
size_t zgreen_group_smem(int, int) { return 0; }
template <typename T>
cudaError_t launch_zgreen(const ZArgs<T>&, dim3, size_t, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_shift(C2<T>*, C2<T>*, long long, int, const double*, bool, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_xfft(const XFftArgs<T>&, int, dim3, size_t, cudaStream_t) OKAY
template <typename T, typename O>
cudaError_t launch_field(const T*, O*, long long, double, cudaStream_t) OKAY
template <typename T, typename O>
cudaError_t launch_von_mises(const T*, O*, long long, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_loop_guard(IterStatus*, int, cudaGraphConditionalHandle, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_adj_sums(const T*, const T*, const T*, const T*, const uint32_t*, const int*, int, long long,
                            double*, double*, cudaStream_t) OKAY
template <typename T>
cudaError_t launch_adj(int, long long, cudaStream_t, const void*, const void*, const void*, void*, void*,
                       const double*) OKAY
}  // namespace rve

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  rve_options o;
  rve_options_default(&o);
  o.precision = argc > 2 ? std::atoi(argv[2]) : RVE_FP32;
  const int nx = argc > 5 ? std::atoi(argv[3]) : 16, ny = argc > 5 ? std::atoi(argv[4]) : 16,
            nz = argc > 5 ? std::atoi(argv[5]) : 16;
  o.graphs = what != "step_host";
  o.autotune = what == "tune";
  o.batch_group = 1;
  o.max_iter = 20;
  std::vector<uint32_t> gid((size_t)nx * ny * nz, 0u);
  const double euler[3] = {0.0, 0.0, 0.0};
  rve_t h[2] = {nullptr, nullptr};
  for (rve_t& q : h)
    if (rve_create(&q, nx, ny, nz, gid.data(), 0, 1, euler, &o) != RVE_OK) return std::printf("%s\n", rve_last_error(q)), 1;
  rec("-- begin");
  rve_status s = RVE_OK;
  if (what == "step_host" || what == "step_graph" || what == "tune") {
    s = rve_step(h[0], 1, nullptr);
  } else if (what == "group") {
    s = rve_step_batch(h, 2, 1, nullptr, nullptr);
  } else if (what == "material") {
    rve_material m;
    rve_material_default(&m);
    s = rve_set_material(h[0], &m);
  } else {
    return 2;
  }
  rec("-- end %d", (int)s);
  for (rve_t q : h) rve_destroy(q);
  return s == RVE_OK ? 0 : 1;
}
