// Periodic Voronoi labelling with the centroid-plane twin split (input generation).
//
// Sec. 2.1: grain n is the set of points not farther from generator s_n than from any
// other generator, here on the periodic unit cell.  Labels are decided exactly:
// voxel centre ((i+1/2)/nx, ...), per-axis difference folded to [-1/2, 1/2]
// (d > 1/2 -> d - 1, then d < -1/2 -> d + 1), squared distance (dx*dx + dy*dy) + dz*dz
// with every operation rounded separately (no fused multiply-add), strict "<" while
// scanning generators in index order so ties go to the lowest index.
//
// Synthetic twins: a twinned parent p is cut by the plane through its centroid with
// normal n_p.  The centroid is (centre of the voxel holding s_p) + (integer sum of
// minimum-image voxel offsets) / count; a voxel goes to the twin (id n_parent + p)
// when (dx*n0 + dy*n1) + dz*n2 > 0 for its minimum-image offset from the centroid in
// voxel units (dx >= n/2 -> dx - n, dx < -n/2 -> dx + n).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/rve.h"
#include "scratch.h"

namespace {

__device__ __forceinline__ double fold_unit(double d) {
  if (d > 0.5) d = __dadd_rn(d, -1.0);
  if (d < -0.5) d = __dadd_rn(d, 1.0);
  return d;
}

__device__ __forceinline__ int wrap_int(int d, int n) {
  // minimum image in [-n/2, n/2)
  int r = (d + n / 2) % n;
  if (r < 0) r += n;
  return r - n / 2;
}

// Labelling kernel.  Deciding a voxel needs the exactly rounded FP64 distances only where two
// generators are almost equally near, so most of the work is done in float on few generators:
//  - a CTA labels a tile of 16 x 8 x 4 voxels.  With D_s the (periodic) distance of generator
//    s from the tile's centre and r the tile's half diagonal, a voxel's nearest generator has
//    D_s <= min D + 2 r (triangle inequality), so the others are dropped for the whole tile
//    (about 10 of 200 generators at 128^3 stay);
//  - each voxel takes the float squared distances of the tile's list.  Their error is below
//    1e-6 (coordinates in [0, 1], |difference| <= 1/2 per axis), so a generator that leads by
//    more than kNear = 4e-6 is the exact one; otherwise the generators within kNear of the
//    least are compared by the exact FP64 expression, in index order.
// The labels equal those of the full FP64 scan (GB300 runs 2 FP64 operations per clock and
// SM: the scan of 200 generators at 128^3 took 17 ms).  128^3, 200 generators, half
// of them twinned: rve_label_voronoi 17.7 -> 0.38 ms with its copies.
// Offset sums of the twinned parents' voxels (sums != NULL) are added per warp and label before
// the atomics.
constexpr int kTx = 16, kTy = 8, kTz = 4, kTileThreads = kTx * kTy;
constexpr int kTileList = 256;  // generators kept per tile; tiles with more scan all of them
constexpr float kNear = 4e-6f;

__device__ __forceinline__ float fold_unit_f(float d) {
  if (d > 0.5f) d -= 1.0f;
  if (d < -0.5f) d += 1.0f;
  return d;
}
__device__ __forceinline__ float dist2_f(float x, float y, float z, const float4& s) {
  const float dx = fold_unit_f(x - s.x), dy = fold_unit_f(y - s.y), dz = fold_unit_f(z - s.z);
  return dx * dx + dy * dy + dz * dz;
}

__global__ void __launch_bounds__(kTileThreads)
    k_voronoi(int nx, int ny, int nz, int n_seed, const double* __restrict__ seeds, const float4* __restrict__ seeds_f,
              uint32_t* __restrict__ label, const uint8_t* __restrict__ twinned, const int* __restrict__ seed_vox,
              unsigned long long* __restrict__ sums) {
  __shared__ float4 list[kTileList];  // (x, y, z, index bits)
  __shared__ float wmin[kTileThreads / 32];
  __shared__ int wcnt[kTileThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tx = (nx + kTx - 1) / kTx, ty = (ny + kTy - 1) / kTy;
  const long long tile = blockIdx.x;
  const int i0 = (int)(tile % tx) * kTx, j0 = (int)((tile / tx) % ty) * kTy, k0 = (int)(tile / ((long long)tx * ty)) * kTz;
  const int ni = min(kTx, nx - i0), nj = min(kTy, ny - j0), nk = min(kTz, nz - k0);
  const float ax = 1.0f / (float)nx, ay = 1.0f / (float)ny, az = 1.0f / (float)nz;
  const float cx = ((float)i0 + 0.5f * (float)ni) * ax, cy = ((float)j0 + 0.5f * (float)nj) * ay,
              cz = ((float)k0 + 0.5f * (float)nk) * az;
  const float hx = 0.5f * (float)(ni - 1) * ax, hy = 0.5f * (float)(nj - 1) * ay, hz = 0.5f * (float)(nk - 1) * az;
  const float r = sqrtf(hx * hx + hy * hy + hz * hz);
  float dmin = INFINITY;
  for (int s = tid; s < n_seed; s += kTileThreads) dmin = fminf(dmin, dist2_f(cx, cy, cz, seeds_f[s]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
  if (lane == 0) wmin[wid] = dmin;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kTileThreads / 32; ++w) dmin = fminf(dmin, wmin[w]);
  const float reach = sqrtf(dmin) + 2.0f * r + 1e-5f;
  const float reach2 = reach * reach;
  int n_list = 0;
  for (int b = 0; b < n_seed && n_list <= kTileList; b += kTileThreads) {
    const int s = b + tid;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    bool keep = false;
    if (s < n_seed) {
      q = seeds_f[s];
      keep = dist2_f(cx, cy, cz, q) <= reach2;
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) wcnt[wid] = __popc(m);
    __syncthreads();
    int at = n_list + __popc(m & ((1u << lane) - 1u));
#pragma unroll
    for (int w = 0; w < kTileThreads / 32; ++w) {
      if (w < wid) at += wcnt[w];
      n_list += wcnt[w];
    }
    if (keep && at < kTileList) list[at] = make_float4(q.x, q.y, q.z, __int_as_float(s));
    __syncthreads();
  }
  const bool all = n_list > kTileList;  // too many for the list: scan every generator
  const int n = all ? n_seed : n_list;
  const int ti = tid % kTx, tj = tid / kTx;
  const int i = i0 + ti, j = j0 + tj;
  const float x = ((float)i + 0.5f) * ax, y = ((float)j + 0.5f) * ay;
  for (int tk = 0; tk < nk; ++tk) {
    const int k = k0 + tk;
    const bool mine = ti < ni && tj < nj;
    uint32_t lab = 0;
    if (mine) {
      const float z = ((float)k + 0.5f) * az;
      float b1 = INFINITY, b2 = INFINITY;
      for (int t = 0; t < n; ++t) {
        const float4 q = all ? seeds_f[t] : list[t];
        const float d2 = dist2_f(x, y, z, q);
        if (d2 < b1) {
          b2 = b1;
          b1 = d2;
          lab = all ? (uint32_t)t : (uint32_t)__float_as_int(q.w);
        } else {
          b2 = fminf(b2, d2);
        }
      }
      if (!(b2 - b1 > kNear)) {
        const double ex = __ddiv_rn(__dadd_rn((double)i, 0.5), (double)nx);
        const double ey = __ddiv_rn(__dadd_rn((double)j, 0.5), (double)ny);
        const double ez = __ddiv_rn(__dadd_rn((double)k, 0.5), (double)nz);
        double best = INFINITY;
        for (int t = 0; t < n; ++t) {
          const float4 q = all ? seeds_f[t] : list[t];
          if (!(dist2_f(x, y, z, q) <= b1 + kNear)) continue;
          const int s = all ? t : __float_as_int(q.w);
          const double dx = fold_unit(__dadd_rn(ex, -seeds[3 * s + 0]));
          const double dy = fold_unit(__dadd_rn(ey, -seeds[3 * s + 1]));
          const double dz = fold_unit(__dadd_rn(ez, -seeds[3 * s + 2]));
          const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
          if (d2 < best) {
            best = d2;
            lab = (uint32_t)s;
          }
        }
      }
      label[(long long)i + (long long)nx * (j + (long long)ny * k)] = lab;
    }
    if (sums) {
      const bool add = mine && twinned[lab];
      const unsigned m = __match_any_sync(0xffffffffu, add ? (int)lab : -1);
      if (add) {
        const int ox = wrap_int(i - seed_vox[3 * lab + 0], nx);
        const int oy = wrap_int(j - seed_vox[3 * lab + 1], ny);
        const int oz = wrap_int(k - seed_vox[3 * lab + 2], nz);
        if (max(nx, max(ny, nz)) <= (1 << 25)) {  // 32 offsets of n / 2 fit an int
          const int sx = __reduce_add_sync(m, ox), sy = __reduce_add_sync(m, oy), sz = __reduce_add_sync(m, oz);
          if (lane == __ffs(m) - 1) {
            atomicAdd(&sums[4 * lab + 0], (unsigned long long)(long long)sx);
            atomicAdd(&sums[4 * lab + 1], (unsigned long long)(long long)sy);
            atomicAdd(&sums[4 * lab + 2], (unsigned long long)(long long)sz);
            atomicAdd(&sums[4 * lab + 3], (unsigned long long)__popc(m));
          }
        } else {
          atomicAdd(&sums[4 * lab + 0], (unsigned long long)(long long)ox);
          atomicAdd(&sums[4 * lab + 1], (unsigned long long)(long long)oy);
          atomicAdd(&sums[4 * lab + 2], (unsigned long long)(long long)oz);
          atomicAdd(&sums[4 * lab + 3], 1ull);
        }
      }
    }
  }
}

__device__ __forceinline__ double fold_grid(double d, int n) {
  const double h = 0.5 * (double)n;
  if (d >= h) return __dadd_rn(d, -(double)n);
  if (d < -h) return __dadd_rn(d, (double)n);
  return d;
}

__global__ void k_twin_split(int nx, int ny, int nz, int n_parent, uint32_t* __restrict__ label,
                             const uint8_t* __restrict__ twinned, const double* __restrict__ cent,
                             const double* __restrict__ normal) {
  const long long nvox = (long long)nx * ny * nz;
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nvox) return;
  const uint32_t p = label[v];
  if (!twinned[p]) return;
  const int i = (int)(v % nx);
  const int j = (int)((v / nx) % ny);
  const int k = (int)(v / ((long long)nx * ny));
  const double dx = fold_grid(__dadd_rn(__dadd_rn((double)i, 0.5), -cent[3 * p + 0]), nx);
  const double dy = fold_grid(__dadd_rn(__dadd_rn((double)j, 0.5), -cent[3 * p + 1]), ny);
  const double dz = fold_grid(__dadd_rn(__dadd_rn((double)k, 0.5), -cent[3 * p + 2]), nz);
  const double side = __dadd_rn(__dadd_rn(__dmul_rn(dx, normal[3 * p + 0]), __dmul_rn(dy, normal[3 * p + 1])),
                                __dmul_rn(dz, normal[3 * p + 2]));
  if (side > 0.0) label[v] = (uint32_t)(n_parent + (int)p);
}

// Per generator: float coordinates, seed voxel (min(trunc(s * n), n - 1) per axis), zero sums.
__global__ void k_seed_prepare(int n_parent, int nx, int ny, int nz, const double* __restrict__ seeds,
                               float4* __restrict__ seeds_f, int* __restrict__ seed_vox,
                               unsigned long long* __restrict__ sums) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_parent) return;
  seeds_f[p] = make_float4((float)seeds[3 * p], (float)seeds[3 * p + 1], (float)seeds[3 * p + 2], 0.f);
  const int n[3] = {nx, ny, nz};
  for (int a = 0; a < 3; ++a) {
    const int v = (int)__dmul_rn(seeds[3 * p + a], (double)n[a]);
    seed_vox[3 * p + a] = v < n[a] - 1 ? v : n[a] - 1;
  }
  for (int a = 0; a < 4; ++a) sums[4 * p + a] = 0ull;
}

// Centroid of each twinned parent: (seed voxel centre) + (integer offset sum) / count, every
// operation rounded separately.
__global__ void k_centroids(int n_parent, const int* __restrict__ seed_vox,
                            const unsigned long long* __restrict__ sums, double* __restrict__ cent) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n_parent) return;
  const long long cnt = (long long)sums[4 * p + 3];
  for (int a = 0; a < 3; ++a) {
    const double base = __dadd_rn((double)seed_vox[3 * p + a], 0.5);
    cent[3 * p + a] = cnt > 0 ? __dadd_rn(base, __ddiv_rn((double)(long long)sums[4 * p + a], (double)cnt)) : base;
  }
}

// Device scratch of one labelling: the host inputs in the order they are copied (seeds,
// normals, twin flags), then what the kernels derive.
struct Scratch {
  double *seeds, *normal;
  uint8_t* twinned;
  float4* seeds_f;
  double* cent;
  unsigned long long* sums;
  int* seed_vox;
};

}  // namespace

namespace rve {
void set_global_error(const std::string& msg);
}

#define LBL_CUDA(call)                                                      \
  do {                                                                      \
    cudaError_t _e = (call);                                                \
    if (_e != cudaSuccess) {                                                \
      rve::set_global_error(std::string(who) + ": " + #call + ": " + cudaGetErrorString(_e));               \
      return RVE_ERR_CUDA;                                                  \
    }                                                                       \
  } while (0)

namespace {

// The checks that the entry points share; *any_twin: some parent is twinned.
rve_status check_inputs(const char* who, int nx, int ny, int nz, int n_parent, const double* seeds,
                        const uint8_t* twinned, const double* twin_normal, const uint32_t* out, bool* any_twin) {
  if (nx < 1 || ny < 1 || nz < 1 || n_parent < 1 || !seeds || !out) {
    rve::set_global_error(std::string(who) + ": bad sizes or NULL pointer");
    return RVE_ERR_INVALID_ARG;
  }
  for (long long s = 0; s < 3LL * n_parent; ++s)
    if (!(seeds[s] >= 0.0 && seeds[s] < 1.0)) {
      rve::set_global_error(std::string(who) + ": seeds must lie in [0, 1)");
      return RVE_ERR_INVALID_ARG;
    }
  *any_twin = false;
  if (twinned)
    for (int p = 0; p < n_parent; ++p) *any_twin |= twinned[p] != 0;
  if (*any_twin && !twin_normal) {
    rve::set_global_error(std::string(who) + ": twin_normal is NULL");
    return RVE_ERR_INVALID_ARG;
  }
  return RVE_OK;
}

// The labelling's kernels on a stream; the inputs are already in the scratch.
rve_status label_on_device(const char* who, int nx, int ny, int nz, int n_parent, bool any_twin, const Scratch& sc,
                           uint32_t* label, cudaStream_t st) {
  const unsigned pg = (unsigned)((n_parent + 127) / 128);
  k_seed_prepare<<<pg, 128, 0, st>>>(n_parent, nx, ny, nz, sc.seeds, sc.seeds_f, sc.seed_vox, sc.sums);
  LBL_CUDA(cudaGetLastError());
  const long long tiles =
      (long long)((nx + kTx - 1) / kTx) * ((ny + kTy - 1) / kTy) * (long long)((nz + kTz - 1) / kTz);
  k_voronoi<<<(unsigned)tiles, kTileThreads, 0, st>>>(nx, ny, nz, n_parent, sc.seeds, sc.seeds_f, label, sc.twinned,
                                                      sc.seed_vox, any_twin ? sc.sums : nullptr);
  LBL_CUDA(cudaGetLastError());
  if (any_twin) {
    k_centroids<<<pg, 128, 0, st>>>(n_parent, sc.seed_vox, sc.sums, sc.cent);
    LBL_CUDA(cudaGetLastError());
    const long long nvox = (long long)nx * ny * nz;
    k_twin_split<<<(unsigned)((nvox + 255) / 256), 256, 0, st>>>(nx, ny, nz, n_parent, label, sc.twinned, sc.cent,
                                                                 sc.normal);
    LBL_CUDA(cudaGetLastError());
  }
  return RVE_OK;
}

}  // namespace

extern "C" rve_status rve_label_voronoi(int nx, int ny, int nz, int n_parent, const double* seeds,
                                        const uint8_t* twinned, const double* twin_normal, uint32_t* out,
                                        int out_on_device, void* stream) {
  const char* who = "rve_label_voronoi";
  bool any_twin = false;
  const rve_status bad = check_inputs(who, nx, ny, nz, n_parent, seeds, twinned, twin_normal, out, &any_twin);
  if (bad) return bad;
  const size_t nvox = (size_t)nx * ny * nz, n = (size_t)n_parent;
  cudaStream_t st = stream ? (cudaStream_t)stream : cudaStreamPerThread;
  // one allocation: 16-byte rows first, then 8-byte, 4-byte and byte arrays; the inputs are
  // packed on the host and copied at once
  const size_t in_bytes = any_twin ? 49 * n : 24 * n, in_room = (49 * n + 15) / 16 * 16;
  std::vector<char> host(in_bytes);  // outlives the scratch
  rve::CallScratch buf;
  LBL_CUDA(buf.alloc(in_room + (16 + 24 + 32 + 12) * n + (out_on_device ? 0 : nvox * sizeof(uint32_t)), st));
  char* d = (char*)buf.p;
  Scratch sc;
  sc.seeds = (double*)d;
  sc.normal = sc.seeds + 3 * n;
  sc.twinned = (uint8_t*)(sc.normal + 3 * n);
  d += in_room;
  sc.seeds_f = (float4*)d;
  sc.cent = (double*)(d + 16 * n);
  sc.sums = (unsigned long long*)(d + 40 * n);
  sc.seed_vox = (int*)(d + 72 * n);
  uint32_t* lab = out_on_device ? out : (uint32_t*)(d + 84 * n);
  std::memcpy(host.data(), seeds, 24 * n);
  if (any_twin) {
    std::memcpy(host.data() + 24 * n, twin_normal, 24 * n);
    std::memcpy(host.data() + 48 * n, twinned, n);
  }
  LBL_CUDA(cudaMemcpyAsync(sc.seeds, host.data(), in_bytes, cudaMemcpyHostToDevice, st));
  const rve_status s = label_on_device(who, nx, ny, nz, n_parent, any_twin, sc, lab, st);
  if (s) return s;
  if (!out_on_device) LBL_CUDA(cudaMemcpyAsync(out, lab, sizeof(uint32_t) * nvox, cudaMemcpyDeviceToHost, st));
  LBL_CUDA(cudaStreamSynchronize(st));
  return RVE_OK;
}

// ---------------------------------------------------------------------------------
// Labelling without device allocation.
//
// For callers that may not allocate device memory (a caller-owned memory pool, loops
// that cannot afford the device-wide synchronisation of cudaMalloc/cudaFree, embedding
// where allocation is forbidden), the scratch of the labelling lives in one static
// device array of fixed size; only the caller's output buffer is written besides it.
namespace {

constexpr int kNoAllocMax = RVE_NOALLOC_MAX_PARENTS;

struct NoAllocScratch {
  float4 seeds_f[kNoAllocMax];
  double seeds[3 * kNoAllocMax];
  double cent[3 * kNoAllocMax];
  double normal[3 * kNoAllocMax];
  unsigned long long sums[4 * kNoAllocMax];
  int seed_vox[3 * kNoAllocMax];
  uint8_t twinned[kNoAllocMax];
};

// Held by every GPU that loads this library until the process exits.  In host code the
// name is only a stand-in: kernels receive the device address looked up below.
static __device__ __align__(256) NoAllocScratch g_noalloc;

// Device address of g_noalloc per device ordinal, looked up once per device.
std::mutex g_noalloc_mu;
NoAllocScratch* g_noalloc_ptr[64] = {nullptr};

}  // namespace

extern "C" rve_status rve_label_voronoi_noalloc(int nx, int ny, int nz, int n_parent, const double* seeds,
                                                const uint8_t* twinned, const double* twin_normal,
                                                uint32_t* out, void* stream) {
  const char* who = "rve_label_voronoi_noalloc";
  if (n_parent > kNoAllocMax) {
    rve::set_global_error("rve_label_voronoi_noalloc: n_parent " + std::to_string(n_parent) +
                          " exceeds the no-allocation maximum of " + std::to_string(kNoAllocMax));
    return RVE_ERR_INVALID_ARG;
  }
  bool any_twin = false;
  const rve_status bad = check_inputs(who, nx, ny, nz, n_parent, seeds, twinned, twin_normal, out, &any_twin);
  if (bad) return bad;
  int dev = 0;
  LBL_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    rve::set_global_error("rve_label_voronoi_noalloc: device ordinal out of range");
    return RVE_ERR_INVALID_ARG;
  }
  NoAllocScratch* na = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void* p = nullptr;
      LBL_CUDA(cudaGetSymbolAddress(&p, g_noalloc));
      g_noalloc_ptr[dev] = static_cast<NoAllocScratch*>(p);
    }
    na = g_noalloc_ptr[dev];
  }
  cudaStream_t st = stream ? (cudaStream_t)stream : cudaStreamPerThread;
  const Scratch sc = {na->seeds, na->normal, na->twinned, na->seeds_f, na->cent, na->sums, na->seed_vox};
  LBL_CUDA(cudaMemcpyAsync(na->seeds, seeds, 3 * sizeof(double) * n_parent, cudaMemcpyHostToDevice, st));
  if (any_twin) {
    LBL_CUDA(cudaMemcpyAsync(na->twinned, twinned, n_parent, cudaMemcpyHostToDevice, st));
    LBL_CUDA(cudaMemcpyAsync(na->normal, twin_normal, 3 * sizeof(double) * n_parent, cudaMemcpyHostToDevice, st));
  }
  const rve_status s = label_on_device(who, nx, ny, nz, n_parent, any_twin, sc, out, st);
  if (s) return s;
  LBL_CUDA(cudaStreamSynchronize(st));
  return RVE_OK;
}
