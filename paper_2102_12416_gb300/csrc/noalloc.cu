// Allocation-free residual of a caller-owned padded state array.
//
// Some callers cannot allocate device memory at the point where they need a
// residual: services that reserve all device memory up front and forbid
// later allocations (a fixed footprint, or a framework whose caching
// allocator must account for every byte), and loops that cannot afford the
// device-wide synchronisation a cudaMalloc or cudaFree may bring.  For them
// this file keeps the reduction scratch in a fixed file-scope device array
// instead of a workspace: every GPU that loads the library holds it (256 KB)
// until exit.
//
// The array is shared by every call on a device and keeps the last call's
// contents; each call overwrites every partial it later reads, so nothing has
// to be cleared first.  Calls whose kernels overlap on the GPU (different
// streams without ordering) race on the array and give wrong results.
#include <mutex>

#include "runtime.h"

using namespace jgb;

namespace {

constexpr int kMaxPlanes = JACOBI_NOALLOC_MAX_PLANES;
constexpr int kNaThreads = 256;
constexpr int kNaRows = 8;  // rows a warp walks with its y neighbours in registers

// Two partials per CTA (a plane, or a share of its rows): sum of r^2, sum of b^2.
static __device__ __align__(256) double g_noalloc_scratch[2 * kMaxPlanes];

// r = s - 6u of one point.  FP64: four of the five sums on the integer pipe when
// all lanes' neighbours are inside the adders' domain (the same rounded sums, by
// dadd_near, or dadd_nn where some lane's are out of its reach; the last sum, 6u,
// the difference and the square stay on the FP64 pipe).  FP32: resid_split where the
// operands' magnitudes show it to be exact.
__device__ __forceinline__ double noalloc_r(double xm, double xp, double ym, double yp, double zm, double zp, double c, bool use) {
  const uint32_t hi = max(max(max((uint32_t)__double2hiint(xm), (uint32_t)__double2hiint(xp)),
                              max((uint32_t)__double2hiint(ym), (uint32_t)__double2hiint(yp))),
                          max((uint32_t)__double2hiint(zm), (uint32_t)__double2hiint(zp)));
  double sxy, sz;
  if (__all_sync(0xffffffffu, !use || hi < kEmuHiLimit)) {
    int far = 0;
    sxy = dadd_near(dadd_near(xm, xp, far), dadd_near(ym, yp, far), far);
    sz = dadd_near(zm, zp, far);
    if (__any_sync(0xffffffffu, use && far < 0 && sum_far(xm, xp, ym, yp, zm, zp, true) < 0)) {
      sxy = dadd_nn(dadd_nn(xm, xp), dadd_nn(ym, yp));
      sz = dadd_nn(zm, zp);
    }
  } else {
    sxy = __dadd_rn(__dadd_rn(xm, xp), __dadd_rn(ym, yp));
    sz = __dadd_rn(zm, zp);
  }
  return __dsub_rn(__dadd_rn(sxy, sz), __dmul_rn(6.0, c));
}
__device__ __forceinline__ double noalloc_r(float xm, float xp, float ym, float yp, float zm, float zp, float c, bool) {
  const float v[7] = {xm, xp, ym, yp, zm, zp, c};
  Magnitudes m;
  m.add(v);
  float d, e;
  if (resid_split(xm, xp, ym, yp, zm, zp, c, d, e) && m.split_exact()) return __dadd_rn(widen_f32(d), widen_f32(e));
  return resid_f64(xm, xp, ym, yp, zm, zp, c);
}

// CTA (plane, share of its rows): its warps take strips of 32 columns x kNaRows
// rows.  Bound by the FP64 pipe (FP64: 4 operations per point beside 4
// integer-pipe sums, FP32: 2); the boundary sum is taken only at the points
// that touch the boundary and the planes are split while they alone do not fill
// the chip.  256^3 FP64: 528 us with both sums in FP64 at every point and one CTA
// per plane, 247 us so.
template <typename T>
__global__ void __launch_bounds__(kNaThreads) k_noalloc_planes(const T* __restrict__ u, int64_t nx, int64_t ny, int64_t nz,
                                                             int split, double* scratch) {
  const int64_t k = 1 + blockIdx.x / split;  // padded plane index
  const int sub = blockIdx.x % split;
  const int64_t px = nx + 2, pp = px * (ny + 2);
  const int64_t j0 = 1 + ny * sub / split, j1 = 1 + ny * (sub + 1) / split;
  const int lane = threadIdx.x & 31;
  const int64_t cols = (nx + 31) / 32, tasks = cols * ((j1 - j0 + kNaRows - 1) / kNaRows);
  double ar = 0.0, ab = 0.0;
  for (int64_t t = threadIdx.x >> 5; t < tasks; t += kNaThreads / 32) {
    const int64_t i = 1 + (t % cols) * 32 + lane, ja = j0 + t / cols * kNaRows, jb = min(ja + kNaRows, j1);
    const bool use = i <= nx;
    const T* p = u + k * pp + ja * px + (use ? i : nx);  // lanes past the row reread its last point
    T ym = p[-px], c = p[0];
    for (int64_t j = ja; j < jb; ++j, p += px) {
      const T yp = p[px], xm = p[-1], xp = p[1], zm = p[-pp], zp = p[pp];
      const double r = noalloc_r(xm, xp, ym, yp, zm, zp, c, use);
      if (use) ar = fma(r, r, ar);
      if (use && (i == 1 || i == nx || j == 1 || j == ny || k == 1 || k == nz)) {
        const double sb = __dadd_rn(__dadd_rn(__dadd_rn(i == 1 ? (double)xm : 0.0, i == nx ? (double)xp : 0.0),
                                              __dadd_rn(j == 1 ? (double)ym : 0.0, j == ny ? (double)yp : 0.0)),
                                    __dadd_rn(k == 1 ? (double)zm : 0.0, k == nz ? (double)zp : 0.0));
        ab = fma(sb, sb, ab);
      }
      ym = c;
      c = yp;
    }
  }
  __shared__ double red[kNaThreads / 32];
  const double sr = block_sum<kNaThreads>(ar, red);
  const double sbb = block_sum<kNaThreads>(ab, red);
  if (threadIdx.x == 0) {
    scratch[2 * blockIdx.x] = sr;
    scratch[2 * blockIdx.x + 1] = sbb;
  }
}

// One CTA: fixed-order sum of the partials, then |r|, |b|, rel.
__global__ void __launch_bounds__(kNaThreads) k_noalloc_finish(const double* scratch, int n, double* out) {
  double r = 0.0, b = 0.0;
  for (int q = threadIdx.x; q < n; q += kNaThreads) {
    r += scratch[2 * q];
    b += scratch[2 * q + 1];
  }
  __shared__ double red[kNaThreads / 32];
  r = block_sum<kNaThreads>(r, red);
  b = block_sum<kNaThreads>(b, red);
  if (threadIdx.x == 0) {
    const double rn = sqrt(r), bn = sqrt(b);
    out[0] = rn;
    out[1] = bn;
    out[2] = bn > 0.0 ? rn / bn : rn;
  }
}

// Device address of the scratch array, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_mu;
double* g_ptr[kMaxDevices] = {};

int scratch_for_current_device(double** out) {
  int dev = 0;
  JGB_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return set_error(JACOBI_EINVAL, "device index %d out of range", dev);
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return set_error(JACOBI_ECUDA, "cudaGetSymbolAddress(scratch) failed on device %d: %s", dev,
                       cudaGetErrorString(e));
    g_ptr[dev] = (double*)p;
  }
  *out = g_ptr[dev];
  return JACOBI_OK;
}

}  // namespace

extern "C" int jacobi_residual_noalloc(const void* u_padded, jacobi_dim3 grid, jacobi_dtype dtype, double* out,
                                       void* stream) {
  if (!u_padded || !out) return set_error(JACOBI_EINVAL, "null pointer");
  if (dtype != JACOBI_F64 && dtype != JACOBI_F32) return set_error(JACOBI_EINVAL, "bad dtype");
  if (grid.nx < 1 || grid.ny < 1 || grid.nz < 1) return set_error(JACOBI_EINVAL, "grid sizes must be positive");
  if (grid.nz > kMaxPlanes)
    return set_error(JACOBI_EINVAL, "jacobi_residual_noalloc: nz = %lld exceeds the fixed scratch limit of %d planes",
                     (long long)grid.nz, kMaxPlanes);
  double* scratch = nullptr;
  int rc = scratch_for_current_device(&scratch);
  if (rc) return rc;
  const cudaStream_t s = (cudaStream_t)stream;
  // Shares per plane: about eight CTAs for each of 152 SMs, no less than kNaRows
  // rows each, within the scratch array.
  const int64_t split = std::max<int64_t>(1, std::min<int64_t>({(1216 + grid.nz - 1) / grid.nz, (grid.ny + kNaRows - 1) / kNaRows,
                                                               kMaxPlanes / grid.nz}));
  const unsigned ctas = (unsigned)(grid.nz * split);
  if (dtype == JACOBI_F64)
    k_noalloc_planes<double><<<ctas, kNaThreads, 0, s>>>((const double*)u_padded, grid.nx, grid.ny, grid.nz, (int)split, scratch);
  else
    k_noalloc_planes<float><<<ctas, kNaThreads, 0, s>>>((const float*)u_padded, grid.nx, grid.ny, grid.nz, (int)split, scratch);
  JGB_CUDA(cudaGetLastError());
  k_noalloc_finish<<<1, kNaThreads, 0, s>>>(scratch, (int)ctas, out);
  JGB_CUDA(cudaGetLastError());
  return JACOBI_OK;
}
