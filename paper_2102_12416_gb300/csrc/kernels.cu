// Jacobi3D support kernels for sm_103a: initial state, state scatter/gather,
// the |b| partials, the deterministic per-grid reduction and the explicit
// pack/copy form of the halo exchange.  The stencil step kernels (Sec. 4.3
// Jacobi iteration, fused face pack, FP64 residual, persistent driver) are in
// step.cu.

#include "kernels.cuh"

namespace jgb {

namespace {

// ---------------------------------------------------------------------------
// Initial values
// ---------------------------------------------------------------------------
__device__ double init_value(const InitDev& I, int64_t gi, int64_t gj, int64_t gk) {
  const bool bnd = gi == 0 || gj == 0 || gk == 0 || gi == I.NX + 1 || gj == I.NY + 1 ||
                   gk == I.NZ + 1;
  const uint64_t idx = ((uint64_t)gk * (uint64_t)(I.NY + 2) + (uint64_t)gj) * (uint64_t)(I.NX + 2) +
                       (uint64_t)gi;
  if (!bnd) {
    if (I.interior == 0) return 0.0;
    if (I.interior == 1) return u01(I.interior_seed, idx);
  }
  if (I.bc == 2) return u01(I.bc_seed, idx);
  const double x = (double)gi / (double)(I.NX + 1);
  const double y = (double)gj / (double)(I.NY + 1);
  const double z = (double)gk / (double)(I.NZ + 1);
  double g = radd(radd(x, rmul(2.0, y)), rmul(3.0, z));
  if (I.bc == 1) g = radd(g, rmul(I.noise_amp, u01(I.bc_seed, idx)));
  return g;
}

template <typename T> __device__ __forceinline__ T to_state(double v);
template <> __device__ __forceinline__ double to_state<double>(double v) { return v; }
template <> __device__ __forceinline__ float to_state<float>(double v) { return __double2float_rn(v); }

// Entries of the (padded) receive slot of face f.
__device__ __forceinline__ int64_t face_elems(const BlockDev& B, int f) {
  if (f == XM || f == XP) return (int64_t)B.nz * B.ry;
  if (f == YM || f == YP) return (int64_t)B.nz * B.rx;
  return (int64_t)B.ry * B.rx;
}

// Offset of interior point (i, j, k) in the block's padded storage.
__device__ __forceinline__ int64_t cell(const BlockDev& B, int64_t i, int64_t j, int64_t k) {
  return k * B.plane_pitch + j * B.rx + i;
}

// ---------------------------------------------------------------------------
// Whole-state kernels: initial state, scatter from a padded array, gather.
//
// Each of them is a pass over memory, so what counts is loads in flight.  A
// block is walked as *extended rows* (j, k), j in [-1, ny], k in [-1, nz]: a
// row of the interior, or one of a y or z receive slot (j or k outside), all
// nx elements long with pitch rx, so interior and slots take the same code; the
// two x ghosts of an interior row are read beside it.  A block's rows are
// split over nsub CTAs (state_split), a warp takes 32 / LPR rows at a time (LPR
// lanes per row, 32 unless the block is narrower), and each lane keeps eight
// elements in flight.  With one CTA per block (before) a small grid left most
// of the chip idle, and a batch paid that once per grid.  jacobi_set_state (with
// its |b| and domain check) and jacobi_copy_out on the device, before -> now:
// 64^3 FP64 in 32^3 blocks 130 -> 20 and 51 -> 13 us; 512^3 FP64 in 64^3 blocks
// 2.69 -> 0.50 and 0.66 -> 0.33 ms; 768^3 FP32 7.8 -> 1.25 and 1.28 -> 0.77 ms; 256
// FP32 grids of 16..192 set and read back 66 -> 8.5 ms.
// ---------------------------------------------------------------------------
struct RowWalk {
  int lo, ey, r, r1, step, j, k, sj, sk, x, lpr;
};

// Rows of this CTA's share; lo = 1 walks the extended rows, 0 the interior only.
__device__ __forceinline__ RowWalk row_walk(const BlockDev& B, int lo, int sub, int nsub) {
  RowWalk W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  W.lo = lo;
  W.ey = B.ny + 2 * lo;
  const int rows = W.ey * (B.nz + 2 * lo);
  int sh = 5;
  while (sh > 0 && (1 << (sh - 1)) >= B.nx) --sh;  // lanes per row: the power of two >= nx, at most 32
  W.lpr = 1 << sh;
  W.x = lane & (W.lpr - 1);
  const int rpw = 32 >> sh;
  W.step = nwarps * rpw;
  W.r = (int)((int64_t)rows * sub / nsub) + warp * rpw + (lane >> sh);
  W.r1 = (int)((int64_t)rows * (sub + 1) / nsub);
  W.j = W.r % W.ey;
  W.k = W.r / W.ey;
  W.sj = W.step % W.ey;
  W.sk = W.step / W.ey;
  return W;
}
__device__ __forceinline__ void row_next(RowWalk& W) {
  W.r += W.step;
  W.j += W.sj;
  W.k += W.sk;
  if (W.j >= W.ey) {
    W.j -= W.ey;
    W.k += 1;
  }
}

// Storage of extended row (j, k) at parity p; null where both are outside.
template <typename T>
__device__ __forceinline__ T* ext_row(const BlockDev& B, int p, int j, int k) {
  const bool jo = j < 0 || j >= B.ny, ko = k < 0 || k >= B.nz;
  if (jo && ko) return nullptr;
  if (ko) return (T*)B.recv[k < 0 ? ZM : ZP][p] + (int64_t)j * B.rx;
  if (jo) return (T*)B.recv[j < 0 ? YM : YP][p] + (int64_t)k * B.rx;
  return (T*)B.u[p] + (int64_t)k * B.plane_pitch + (int64_t)j * B.rx;
}

// Outside the domain of the integer-pipe adders: sign set, or an exponent field
// that is too large.  FP32 states never use them.
__device__ __forceinline__ bool emu_outside(double v) { return (uint32_t)__double2hiint(v) >= kEmuHiLimit; }
__device__ __forceinline__ bool emu_outside(float) { return false; }

// A grid whose state holds a value outside that domain is flagged: the step
// kernels then keep its sums on the FP64 pipe.  By the discrete maximum
// principle Jacobi iterates stay within the range of the boundary and initial
// data, so a state that passes keeps passing.  The kernels that install a state
// gather the flag in emu_acc; the |b| reduction that follows them publishes it as
// emu_bad and clears it for the next state.
template <typename T>
__device__ __forceinline__ void emu_flag(bool bad, GridNorm* norms, int grid) {
  if (sizeof(T) == 8 && __syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&norms[grid].emu_acc, 1u);
}

__device__ __forceinline__ void block_to_shared(BlockDev& d, const BlockDev* s) {
  for (int q = threadIdx.x; q < (int)(sizeof(BlockDev) / 4); q += blockDim.x) ((uint32_t*)&d)[q] = ((const uint32_t*)s)[q];
  __syncthreads();
}

// |b|^2 partial of one work item: the residual expression with every interior
// value 0, so only points beside a Dirichlet face contribute and only those are
// visited, each once: the item's z-face planes, the y-face rows of its other
// planes, the x-face columns of the other rows.  `ghost(f, i, j, k)` is the
// boundary value across face f of point (i, j, k).  (Visiting every point, as
// before: 1.5 ms at 512^3 FP64, 5.2 ms at 768^3 FP32.)  The ranges are written
// with 0/1 flags on purpose: as max() of the 16-bit item fields, ptxas 13.0
// gave empty ranges at -O1 and above (and right ones at -O0).
template <typename G>
__device__ __forceinline__ void bnorm_add(double& acc, const BlockDev& B, const G& ghost, int i, int j, int k) {
  double v[6] = {0, 0, 0, 0, 0, 0};
  if (i == 0 && B.nbr[XM] < 0) v[0] = ghost(XM, i, j, k);
  if (i == B.nx - 1 && B.nbr[XP] < 0) v[1] = ghost(XP, i, j, k);
  if (j == 0 && B.nbr[YM] < 0) v[2] = ghost(YM, i, j, k);
  if (j == B.ny - 1 && B.nbr[YP] < 0) v[3] = ghost(YP, i, j, k);
  if (k == 0 && B.nbr[ZM] < 0) v[4] = ghost(ZM, i, j, k);
  if (k == B.nz - 1 && B.nbr[ZP] < 0) v[5] = ghost(ZP, i, j, k);
  const double sb = __dadd_rn(__dadd_rn(__dadd_rn(v[0], v[1]), __dadd_rn(v[2], v[3])), __dadd_rn(v[4], v[5]));
  acc = fma(sb, sb, acc);
}
template <typename G>
__device__ __forceinline__ double bnorm_item(const BlockDev& B, const WorkItem& w, const G& ghost) {
  const int nx = B.nx, ny = B.ny, nz = B.nz, tid = threadIdx.x;
  const int za = w.z0, zb = w.z1;
  const int xa = w.x0 >= 0 ? w.x0 : 0, ya = w.x0 >= 0 ? w.y0 : w.ya;
  const int xb = w.x0 >= 0 ? min(w.x0 + TX, nx) : nx, yb = min(w.x0 >= 0 ? w.y0 + TY : (int)w.yb, ny);
  double acc = 0.0;
  // Planes (rows, columns) of the item on its low and high Dirichlet faces: 0
  // or 1 each (a one-point extent with both faces counts as low).  Planes
  // [ka, kb), rows [ja, jb) and columns [ia, ib) are away from them.
  const int zlo = (za == 0 && B.nbr[ZM] < 0) ? 1 : 0, zhi = (zb == nz && B.nbr[ZP] < 0 && zb - za > zlo) ? 1 : 0;
  const int ylo = (ya == 0 && B.nbr[YM] < 0) ? 1 : 0, yhi = (yb == ny && B.nbr[YP] < 0 && yb - ya > ylo) ? 1 : 0;
  const int xlo = (xa == 0 && B.nbr[XM] < 0) ? 1 : 0, xhi = (xb == nx && B.nbr[XP] < 0 && xb - xa > xlo) ? 1 : 0;
  const int ka = za + zlo, kb = zb - zhi, ja = ya + ylo, jb = yb - yhi, ib = xb - xhi;
  const int nw = xb - xa, nh = yb - ya, nd = kb - ka, nr = jb - ja;
  // One loop over the points of all three groups: the first e of each group's
  // plane (row, column) are those before the inner range, the others after it.
  const int ez = nw * nh * (zlo + zhi), ey = ez + nw * nd * (ylo + yhi), ex = ey + nr * nd * (xlo + xhi);
  for (int e = tid; e < ex; e += kThreads) {
    int i, j, k;
    if (e < ez) {
      const int n = nw * nh, t = e / n, q = e - t * n;
      k = t < zlo ? za + t : kb + t - zlo;
      j = ya + q / nw;
      i = xa + q % nw;
    } else if (e < ey) {
      const int n = nw * nd, t = (e - ez) / n, q = (e - ez) - t * n;
      j = t < ylo ? ya + t : jb + t - ylo;
      k = ka + q / nw;
      i = xa + q % nw;
    } else {
      const int n = nr * nd, t = (e - ey) / n, q = (e - ey) - t * n;
      i = t < xlo ? xa + t : ib + t - xlo;
      k = ka + q / nr;
      j = ja + q % nr;
    }
    bnorm_add(acc, B, ghost, i, j, k);
  }
  return acc;
}

// Boundary values from the receive slots of parity p, or from a padded array
// (base: the block's first interior point).
template <typename T>
struct SlotGhost {
  const BlockDev* B;
  int p;
  __device__ __forceinline__ double operator()(int f, int i, int j, int k) const {
    const int64_t e = f < YM ? (int64_t)k * B->ry + j : f < ZM ? (int64_t)k * B->rx + i : (int64_t)j * B->rx + i;
    return (double)((const T*)B->recv[f][p])[e];
  }
};
template <typename T>
struct ArrayGhost {
  const T* base;
  int64_t px, pp;  // row and plane pitch
  __device__ __forceinline__ double operator()(int f, int i, int j, int k) const {
    const int64_t d = f < YM ? 1 : f < ZM ? px : pp;
    return (double)base[(int64_t)k * pp + (int64_t)j * px + i + ((f & 1) ? d : -d)];
  }
};

// Initial state (interior and slots at parity 0) with its domain check.  The
// workspace is zero before this kernel, so a zero interior is not written.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_init(const BlockDev* __restrict__ blocks, const BlockGeom* __restrict__ geom,
                                                   const InitDev* __restrict__ inits, GridNorm* norms) {
  __shared__ BlockDev B;
  block_to_shared(B, blocks + blockIdx.x);
  const BlockGeom G = geom[blockIdx.x];
  const InitDev I = inits[G.grid];
  bool bad = false;
  auto value = [&](int i, int j, int k) {
    const T v = to_state<T>(init_value(I, G.ox + 1 + i, G.oy + 1 + j, G.oz + 1 + k));
    bad |= emu_outside(v);
    return v;
  };
  for (RowWalk W = row_walk(B, 1, blockIdx.y, gridDim.y); W.r < W.r1; row_next(W)) {
    const int j = W.j - 1, k = W.k - 1;
    T* d = ext_row<T>(B, 0, j, k);
    if (!d) continue;
    const bool inside = j >= 0 && j < B.ny && k >= 0 && k < B.nz;
    if (!inside || I.interior != 0)
      for (int i = W.x; i < B.nx; i += W.lpr) d[i] = value(i, j, k);
  }
  // x slots: lanes along y, so that a warp's FP64 divisions serve 32 values
  const int64_t n = (int64_t)B.ny * B.nz;
  const int64_t e1 = 2 * n * (blockIdx.y + 1) / gridDim.y;
  for (int64_t e = 2 * n * blockIdx.y / gridDim.y + threadIdx.x; e < e1; e += kThreads) {
    const int q = (int)(e < n ? e : e - n), k = q / B.ny, j = q - k * B.ny;
    ((T*)B.recv[e < n ? XM : XP][0])[(int64_t)k * B.ry + j] = value(e < n ? -1 : B.nx, j, k);
  }
  emu_flag<T>(bad, norms, G.grid);
}

// CTAs [0, n_items) take one work item each and write its |b|^2 partial, straight
// from a padded array of one grid (first, so that they do not trail); the
// nb * nsub CTAs after them install the array into the grid's blocks (parity p
// state and slots) and check its domain.
template <typename T>
__global__ void __launch_bounds__(kThreads, 4) k_scatter(const BlockDev* __restrict__ blocks, const BlockGeom* __restrict__ geom,
                                                         int32_t b0, int32_t n_items, int32_t nsub, const T* __restrict__ src, int64_t NX,
                                                         int64_t NY, int parity, const WorkItem* __restrict__ items, double* partials,
                                                         GridNorm* norms) {
  __shared__ BlockDev B;
  const int64_t px = NX + 2, pp = px * (NY + 2);
  if ((int)blockIdx.x < n_items) {
    const WorkItem w = items[blockIdx.x];
    block_to_shared(B, blocks + w.block);
    const BlockGeom G = geom[w.block];
    const T* base = src + (int64_t)(G.oz + 1) * pp + (int64_t)(G.oy + 1) * px + (G.ox + 1);
    const double acc = bnorm_item(B, w, ArrayGhost<T>{base, px, pp});
    __shared__ double red[kThreads / 32];
    const double s = block_sum<kThreads>(acc, red);
    if (threadIdx.x == 0) partials[w.slot] = s;
    return;
  }
  const int q = blockIdx.x - n_items, b = b0 + q / nsub;
  block_to_shared(B, blocks + b);
  const BlockGeom G = geom[b];
  const T* __restrict__ base = src + (int64_t)(G.oz + 1) * pp + (int64_t)(G.oy + 1) * px + (G.ox + 1);
  const int nx = B.nx;
  bool bad = false;
  RowWalk W = row_walk(B, 1, q % nsub, nsub);
  while (W.r < W.r1) {
    constexpr int U = 4;
    const T* s[U];
    T* d[U];
    int ge[U];  // an interior row's entry in the x slots, else -1
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = W.j - 1, k = W.k - 1;
      d[u] = W.r < W.r1 ? ext_row<T>(B, parity, j, k) : nullptr;
      s[u] = base + (int64_t)k * pp + (int64_t)j * px;
      const bool inside = d[u] && j >= 0 && j < B.ny && k >= 0 && k < B.nz;
      ge[u] = inside ? k * B.ry + j : -1;
      row_next(W);
    }
    T g[U];
    const int gi = W.x == 0 ? -1 : nx;
    if (W.x < 2) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (ge[u] >= 0) g[u] = s[u][gi];
    }
    for (int i = W.x; i < nx; i += 2 * W.lpr) {
      T v[U][2];
      const bool two = i + W.lpr < nx;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (d[u]) {
          v[u][0] = s[u][i];
          if (two) v[u][1] = s[u][i + W.lpr];
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (d[u]) {
          d[u][i] = v[u][0];
          bad |= emu_outside(v[u][0]);
          if (two) {
            d[u][i + W.lpr] = v[u][1];
            bad |= emu_outside(v[u][1]);
          }
        }
    }
    if (W.x < 2) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (ge[u] >= 0) {
          ((T*)B.recv[W.x == 0 ? XM : XP][parity])[ge[u]] = g[u];
          bad |= emu_outside(g[u]);
          if (W.lpr == 1) {  // one-point rows: this lane takes both ghosts
            const T o = s[u][nx];
            ((T*)B.recv[XP][parity])[ge[u]] = o;
            bad |= emu_outside(o);
          }
        }
    }
  }
  emu_flag<T>(bad, norms, G.grid);
}

// Rows in flight of the gather: a lane holds U rows x E elements.  Rows are kept as
// (k, j) in one word and their addresses derived twice, for the load and for the
// store, which leaves the registers to the data: blocks of up to 32 columns take 8
// rows x 1, wider ones 4 x 2 (512^3 FP32 in 32^3 blocks 572 -> 367 us, 768^3 in 64^3
// blocks 992 -> 772 us against 4 x 2 with both pointers kept; the scatter, with its
// domain check and x ghosts, spills so and keeps its pointers).
__device__ __forceinline__ int row_pack(int j, int k) { return (k + 1) << 16 | (j + 1); }

template <typename T, int U, int E>
__device__ __forceinline__ void gather_rows(const BlockDev& B, RowWalk W, T* __restrict__ base, int64_t px, int64_t pp, int parity, int padded) {
  const int nx = B.nx;
  while (W.r < W.r1) {
    int jk[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = W.j - padded, k = W.k - padded;
      bool take = W.r < W.r1;
      if (padded) {  // only Dirichlet faces lie on the padded boundary
        const bool jo = j < 0 || j >= B.ny, ko = k < 0 || k >= B.nz;
        if (jo) take = take && !ko && B.nbr[j < 0 ? YM : YP] < 0;
        if (ko) take = take && !jo && B.nbr[k < 0 ? ZM : ZP] < 0;
        if (take && !jo && !ko)
          for (int g = W.x; g < 2; g += W.lpr)
            if (B.nbr[g ? XP : XM] < 0)
              base[(int64_t)k * pp + (int64_t)j * px + (g ? nx : -1)] = ((const T*)B.recv[g ? XP : XM][parity])[(int64_t)k * B.ry + j];
      }
      jk[u] = take ? row_pack(j, k) : -1;
      row_next(W);
    }
    for (int i = W.x; i < nx; i += E * W.lpr) {
      T v[U][E];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (jk[u] < 0) continue;
        const T* s = ext_row<T>(B, parity, (jk[u] & 0xFFFF) - 1, (jk[u] >> 16) - 1);
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (i + e * W.lpr < nx) v[u][e] = s[i + e * W.lpr];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (jk[u] < 0) continue;
        T* d = base + ((int64_t)((jk[u] >> 16) - 1) * pp + (int64_t)((jk[u] & 0xFFFF) - 1) * px);
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (i + e * W.lpr < nx) d[i + e * W.lpr] = v[u][e];
      }
    }
  }
}

// Current iterate (parity p) back to an array of the whole grid: the interior,
// or (padded) with the Dirichlet faces around it.
template <typename T>
__global__ void __launch_bounds__(kThreads, 4) k_gather(const BlockDev* __restrict__ blocks, const BlockGeom* __restrict__ geom,
                                                        int32_t b0, int32_t nsub, T* __restrict__ dst, int64_t NX, int64_t NY, int parity,
                                                        int padded) {
  __shared__ BlockDev B;
  const int b = b0 + blockIdx.x / nsub;
  block_to_shared(B, blocks + b);
  const BlockGeom G = geom[b];
  const int64_t px = NX + 2 * padded, pp = px * (NY + 2 * padded);
  T* __restrict__ base = dst + (int64_t)(G.oz + padded) * pp + (int64_t)(G.oy + padded) * px + (G.ox + padded);
  const RowWalk W = row_walk(B, padded, blockIdx.x % nsub, nsub);
  if (B.nx <= 32) gather_rows<T, 8, 1>(B, W, base, px, pp, parity, padded);
  else gather_rows<T, 4, 2>(B, W, base, px, pp, parity, padded);
}

// |b|^2 partials of work items from the receive slots.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_bnorm(StepLaunch a) {
  const WorkItem w = a.items[blockIdx.x];
  const BlockDev& B = a.blocks[w.block];
  const int p = (int)((a.it - a.grids[B.grid].start_iter) & 1);
  const double acc = bnorm_item(B, w, SlotGhost<T>{&B, p});
  __shared__ double red[kThreads / 32];
  const double s = block_sum<kThreads>(acc, red);
  if (threadIdx.x == 0) a.partials[w.slot] = s;
}

// Self-test of the integer-pipe adders: out[i] = a[i] + b[i] by dadd_nn, or NaN
// where dadd_near reaches (a sum with zero included) and differs from it.
__global__ void k_selftest_dadd(const double* a, const double* b, int64_t n, double* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = i < n ? i : n - 1;  // clamped index: every lane loads in bounds
  int far = 0;
  const double r = dadd_nn(a[j], b[j]), r2 = dadd_near(a[j], b[j], far);
  if (far < 0) far = exp_far(a[j], b[j], 10);
  const bool same = far < 0 || __double_as_longlong(r) == __double_as_longlong(r2);
  if (i < n) out[i] = same ? r : __longlong_as_double(-1ll);
}

// Every binary32 bit pattern through widen_f32, against the conversion
// instruction: counts results that differ bit for bit (a NaN must stay a NaN).
__global__ void k_selftest_widen(unsigned long long* bad) {
  unsigned long long n = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < (1ull << 32); x += stride) {
    const float f = __uint_as_float((uint32_t)x);
    const double a = widen_f32(f), b = (double)f;
    const bool ok = (a != a && b != b) || __double_as_longlong(a) == __double_as_longlong(b);
    n += ok ? 0ull : 1ull;
  }
  if (n) atomicAdd(bad, n);
}

// Every binary32 bit pattern through div6 (the FP32 update's RN(s / 6) in two
// operations, with its fallback), against the division instruction sequence:
// counts results that differ bit for bit (a NaN must stay a NaN).
__global__ void k_selftest_div6(unsigned long long* bad) {
  unsigned long long n = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < (1ull << 32); x += stride) {
    const float f = __uint_as_float((uint32_t)x);
    const float a = div6(f), b = __fdiv_rn(f, 6.0f);
    const bool ok = (a != a && b != b) || __float_as_uint(a) == __float_as_uint(b);
    n += ok ? 0ull : 1ull;
  }
  if (n) atomicAdd(bad, n);
}

// Pipe-rate probe: chains of FP64 adds on the FP64 pipe (EMU = false) or
// through dadd_nn on the integer pipe (EMU = true); 8 independent chains per
// thread keep either pipe busy.  The result is stored so nothing is elided.
template <bool EMU>
__global__ void k_pipe_rate(double* out, int iters) {
  double x[8];
  for (int c = 0; c < 8; ++c) x[c] = 0.25 + 1e-3 * (double)(threadIdx.x + c);
  const double inc = 1e-9 + 1e-13 * (double)blockIdx.x;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int c = 0; c < 8; ++c) x[c] = EMU ? dadd_nn(x[c], inc) : __dadd_rn(x[c], inc);
  }
  double s = 0.0;
  for (int c = 0; c < 8; ++c) s += x[c];
  out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// One CTA per grid: thread t sums slots item_begin + t, + t + 256, ... in order,
// then a fixed tree combines the threads (one warp per grid took 16 us for
// the 4096 partials of a 512^3 grid).  which = 0: the residual; 1: |b| of a
// newly installed state, which also publishes its domain flag; 2: |b| only.
__global__ void __launch_bounds__(kThreads) k_reduce(const GridDev* grids, GridNorm* norms, const int32_t* grid_ids,
                                                     const double* partials, int which) {
  const int g = grid_ids[blockIdx.x];
  const GridDev G = grids[g];
  GridNorm& N = norms[g];
  double s = 0.0;
  for (int q = G.item_begin + threadIdx.x; q < G.item_end; q += kThreads) s += partials[q];
  __shared__ double red[kThreads / 32];
  s = block_sum<kThreads>(s, red);
  if (threadIdx.x == 0) {
    if (which == 0) {
      N.r_norm2 = s;
      N.r_norm = sqrt(s);
      const double b = sqrt(N.b_norm2);
      N.rel = b > 0.0 ? N.r_norm / b : N.r_norm;
    } else {
      N.b_norm2 = s;
      if (which == 1) {
        N.emu_bad = N.emu_acc;
        N.emu_acc = 0u;
      }
    }
  }
}

// Explicit exchange, step 1: pack each internal face of the new iterate
// (parity p ^ 1 state) into a contiguous staging buffer, or (direct) straight
// into the neighbour's receive slot for the next parity.
template <typename T>
__global__ void k_pack_faces(const BlockDev* __restrict__ blocks, const int32_t* __restrict__ ids,
                             void* const* staging, const GridDev* grids, int64_t it, int direct) {
  const int b = ids[blockIdx.x], f = blockIdx.y;
  const BlockDev& B = blocks[b];
  if (B.nbr[f] < 0) return;
  const int p = (int)((it - grids[B.grid].start_iter) & 1);
  const T* U = (const T*)B.u[p ^ 1];
  T* S = direct ? (T*)B.send[f][p ^ 1] : (T*)staging[b * 6 + f];
  const int64_t nx = B.nx, ny = B.ny, nz = B.nz, rx = B.rx, ry = B.ry;
  const int64_t n = face_elems(B, f);
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {  // padding entries copy padding
    int64_t i, j, k;
    if (f == XM || f == XP) { k = e / ry; j = e % ry; i = (f == XM) ? 0 : nx - 1; }
    else if (f == YM || f == YP) { k = e / rx; i = e % rx; j = (f == YM) ? 0 : ny - 1; }
    else { j = e / rx; i = e % rx; k = (f == ZM) ? 0 : nz - 1; }
    S[e] = U[cell(B, i, j, k)];
  }
}

// Explicit exchange, step 2: the channel transfer of each packed face into the
// neighbour's receive slot for the next parity.
template <typename T>
__global__ void k_copy_faces(const BlockDev* __restrict__ blocks, const int32_t* __restrict__ ids,
                             void* const* staging, const GridDev* grids, int64_t it) {
  const int b = ids[blockIdx.x], f = blockIdx.y;
  const BlockDev& B = blocks[b];
  if (B.nbr[f] < 0) return;
  const int p = (int)((it - grids[B.grid].start_iter) & 1);
  const T* S = (const T*)staging[b * 6 + f];
  T* D = (T*)B.send[f][p ^ 1];
  const int64_t n = face_elems(B, f);
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) D[e] = S[e];
}

// Posted receives of the GPU Messaging form: one CTA per descriptor copies
// its payload (16-byte vectors; every face buffer is a whole number of them).
__global__ void k_copy_desc(const CopyDesc* __restrict__ d, int32_t n) {
  const CopyDesc c = d[blockIdx.x];
  const uint4* src = (const uint4*)c.src;
  uint4* dst = (uint4*)c.dst;
  const int64_t nv = c.bytes / 16;
  for (int64_t q = threadIdx.x; q < nv; q += blockDim.x) dst[q] = __ldcg(src + q);
}

}  // namespace

cudaError_t launch_copy_desc(const CopyDesc* d, int32_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_copy_desc<<<n, 256, 0, s>>>(d, n);
  return cudaGetLastError();
}

cudaError_t launch_bnorm(const StepLaunch& a, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  if (a.dtype == 0) k_bnorm<double><<<a.n_items, kThreads, 0, s>>>(a);
  else k_bnorm<float><<<a.n_items, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const GridDev* grids, GridNorm* norms, const int32_t* grid_ids, int32_t n,
                          const double* partials, int which, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_reduce<<<n, kThreads, 0, s>>>(grids, norms, grid_ids, partials, which);
  return cudaGetLastError();
}

cudaError_t launch_pack_faces(const BlockDev* blocks, const int32_t* ids, int32_t n_blocks, void* const* staging,
                              const GridDev* grids, int64_t it, int32_t dtype, cudaStream_t s, bool direct) {
  if (n_blocks <= 0) return cudaSuccess;
  const dim3 grid(n_blocks, 6);
  if (dtype == 0) k_pack_faces<double><<<grid, 256, 0, s>>>(blocks, ids, staging, grids, it, direct ? 1 : 0);
  else k_pack_faces<float><<<grid, 256, 0, s>>>(blocks, ids, staging, grids, it, direct ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_copy_faces(const BlockDev* blocks, const int32_t* ids, int32_t n_blocks, void* const* staging,
                              const GridDev* grids, int64_t it, int32_t dtype, cudaStream_t s) {
  if (n_blocks <= 0) return cudaSuccess;
  const dim3 grid(n_blocks, 6);
  if (dtype == 0) k_copy_faces<double><<<grid, 256, 0, s>>>(blocks, ids, staging, grids, it);
  else k_copy_faces<float><<<grid, 256, 0, s>>>(blocks, ids, staging, grids, it);
  return cudaGetLastError();
}

cudaError_t launch_pipe_rate(bool emu, int blocks, int threads, int iters, double* out, cudaStream_t s) {
  if (emu) k_pipe_rate<true><<<blocks, threads, 0, s>>>(out, iters);
  else k_pipe_rate<false><<<blocks, threads, 0, s>>>(out, iters);
  return cudaGetLastError();
}

cudaError_t launch_selftest_dadd(const double* a, const double* b, int64_t n, double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_selftest_dadd<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, b, n, out);
  return cudaGetLastError();
}

cudaError_t launch_selftest_widen(unsigned long long* bad, cudaStream_t s) {
  k_selftest_widen<<<1216, 256, 0, s>>>(bad);
  return cudaGetLastError();
}

cudaError_t launch_selftest_div6(unsigned long long* bad, cudaStream_t s) {
  k_selftest_div6<<<1216, 256, 0, s>>>(bad);
  return cudaGetLastError();
}

// CTAs per block of the whole-state kernels for blocks of up to max_rows
// extended rows: 512 rows per CTA on large states (64 rows per warp: several
// batches of loads each, and enough CTAs for an even tail), down to 32 (one batch)
// while that leaves fewer than about four CTAs per SM.
static int state_split(int32_t n_blocks, int32_t max_rows) {
  const int64_t rows = (int64_t)n_blocks * max_rows;
  const int64_t per = std::min<int64_t>(512, std::max<int64_t>(32, rows / 608));
  return (int)std::min<int64_t>(65535, (max_rows + per - 1) / per);
}

cudaError_t launch_init(const BlockDev* blocks, const BlockGeom* geom, int32_t n_blocks, int32_t max_rows,
                        const InitDev* inits, GridNorm* norms, int32_t dtype, cudaStream_t s) {
  if (n_blocks <= 0) return cudaSuccess;
  const dim3 grid(n_blocks, state_split(n_blocks, max_rows));
  if (dtype == 0) k_init<double><<<grid, kThreads, 0, s>>>(blocks, geom, inits, norms);
  else k_init<float><<<grid, kThreads, 0, s>>>(blocks, geom, inits, norms);
  return cudaGetLastError();
}

cudaError_t launch_scatter(const BlockDev* blocks, const BlockGeom* geom, int32_t b0, int32_t nb, int32_t max_rows,
                           const void* src, int64_t NX, int64_t NY, int parity, const WorkItem* items, int32_t n_items,
                           double* partials, GridNorm* norms, int32_t dtype, cudaStream_t s) {
  if (nb <= 0) return cudaSuccess;
  const int nsub = state_split(nb, max_rows);
  const unsigned grid = (unsigned)((int64_t)nb * nsub + n_items);
  if (dtype == 0)
    k_scatter<double><<<grid, kThreads, 0, s>>>(blocks, geom, b0, n_items, nsub, (const double*)src, NX, NY, parity, items, partials, norms);
  else
    k_scatter<float><<<grid, kThreads, 0, s>>>(blocks, geom, b0, n_items, nsub, (const float*)src, NX, NY, parity, items, partials, norms);
  return cudaGetLastError();
}

cudaError_t launch_gather(const BlockDev* blocks, const BlockGeom* geom, int32_t b0, int32_t nb, int32_t max_rows, void* dst,
                          int64_t NX, int64_t NY, int parity, int padded, int32_t dtype, cudaStream_t s) {
  if (nb <= 0) return cudaSuccess;
  const int nsub = state_split(nb, max_rows);
  const unsigned grid = (unsigned)((int64_t)nb * nsub);
  const int pad = padded ? 1 : 0;
  if (dtype == 0) k_gather<double><<<grid, kThreads, 0, s>>>(blocks, geom, b0, nsub, (double*)dst, NX, NY, parity, pad);
  else k_gather<float><<<grid, kThreads, 0, s>>>(blocks, geom, b0, nsub, (float*)dst, NX, NY, parity, pad);
  return cudaGetLastError();
}

}  // namespace jgb
