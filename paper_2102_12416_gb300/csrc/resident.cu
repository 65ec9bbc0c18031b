// Resident kernel: all iterations of a small problem in one cooperative launch
// with the state in shared memory.
//
// A small grid's iteration is bound by latency: 64^3 FP64 takes 1.4 us of
// arithmetic over the whole chip, but a launch per iteration 6.6 us (launch gap,
// dependent table loads, bulk-copy fill, store drain) and the flag-driven
// persistent kernel 7.8 us (release fence, flag, bulk copies, per unit).  Here
// each CTA keeps one box of a grid, both parities, in its shared memory from the
// first iteration to the last, and only box surfaces travel, through L2, in
// packets whose every 8-byte word carries 4 bytes of payload and the sequence
// number of its iteration: an 8-byte access is single-copy atomic, so a reader
// that finds the number has the payload, and no fence, flag or release is needed.
// What an iteration costs beside its arithmetic is one store -> L2 -> load trip
// and one CTA barrier.  Per iteration, launch path -> resident: 32^3 4.9 -> 1.8 us
// (FP32) and 5.6 -> 2.2 (FP64), 64^3 5.3 -> 2.0 and 6.5 -> 4.1, 96^3 5.5 -> 3.1 and
// 11.1 -> 7.7, 128^3 FP32 6.5 -> 5.0; a call costs 10 to 40 us once (launch, tables,
// the state's way in and out).
//
// Boxes: each active grid is cut into cx * cy * cz near-equal boxes (x cuts on
// vector boundaries) regardless of its blocks, so box neighbours always face
// each other one to one; one box per SM at most (resident_plan).  Blocks and
// receive slots matter at the two ends only: the launch reads the blocks' state
// (and the Dirichlet slots) of its first iteration and writes back state and
// every receive slot of its last, which is all that later launches read.
//
// Packet buffers are double-buffered by iteration parity.  A box sends its
// surface of iteration t + 2 only after it has received its neighbour's of t + 1,
// which the neighbour sent after all its threads had read t: the buffer is free.
// Sequence numbers continue from launch to launch (ctl[0], advanced by the last
// CTA to finish), so nothing is cleared between launches.  Waits are bounded; the
// limit counts from when all CTAs have started (ctl[2], looked at only when a wait
// runs out), which other streams' kernels may delay.  (A meeting of all CTAs before
// the second iteration instead cost 3 us a call.)
#include <atomic>
#include <vector>

#include "kernels.cuh"
#include "stencil.cuh"

namespace jgb {

namespace {

// Block index along an axis and local coordinate of grid coordinate g.
__device__ __forceinline__ void axis_locate(int mode, int param, int n, int g, int& b, int& l) {
  if (mode == 1) {  // split by block extent
    b = g / param;
    l = g - b * param;
    return;
  }
  const int q = n / param, r = n % param, big = r * (q + 1);  // the first r blocks have one more
  if (g < big) {
    b = g / (q + 1);
    l = g - b * (q + 1);
  } else {
    b = r + (g - big) / q;
    l = (g - big) % q;
  }
}

// Entry of the per-axis tables for box coordinate e - 1 (e = 0 and n + 1 are the
// halo): block along the axis << 16 | local coordinate; outside the grid the
// adjacent block with kOutside set.
constexpr uint32_t kOutside = 0x80000000u;
__device__ __forceinline__ uint32_t axis_entry(int mode, int param, int N, int g) {
  int b, l;
  axis_locate(mode, param, N, min(max(g, 0), N - 1), b, l);
  return ((uint32_t)b << 16 | (uint32_t)l) | ((g < 0 || g >= N) ? kOutside : 0u);
}

// v / d for v, d < 2^16 (m = ceil(2^32 / d)).
__device__ __forceinline__ int fast_div(int v, int d, uint32_t m) { return d == 1 ? v : (int)__umulhi((uint32_t)v, m); }

__device__ __forceinline__ void st_packet(uint4* p, uint32_t a, uint32_t b, uint32_t seq) {
  const uint64_t x = (uint64_t)seq << 32 | a, y = (uint64_t)seq << 32 | b;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}
__device__ __forceinline__ bool ld_packet(const uint4* p, uint32_t& a, uint32_t& b, uint32_t seq) {
  uint64_t x, y;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
  a = (uint32_t)x;
  b = (uint32_t)y;
  return (uint32_t)(x >> 32) == seq && (uint32_t)(y >> 32) == seq;
}

template <typename T> struct Words;  // payload words of a vector / of one value
template <> struct Words<float> {
  __device__ static __forceinline__ void vec(const float (&v)[4], uint32_t (&w)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = __float_as_uint(v[q]);
  }
  __device__ static __forceinline__ void one(float v, uint32_t& a, uint32_t& b) { a = b = __float_as_uint(v); }
  __device__ static __forceinline__ float make(uint32_t a, uint32_t) { return __uint_as_float(a); }
};
template <> struct Words<double> {
  __device__ static __forceinline__ void vec(const double (&v)[2], uint32_t (&w)[4]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) one(v[q], w[2 * q], w[2 * q + 1]);
  }
  __device__ static __forceinline__ void one(double v, uint32_t& a, uint32_t& b) {
    a = (uint32_t)__double2loint(v);
    b = (uint32_t)__double2hiint(v);
  }
  __device__ static __forceinline__ double make(uint32_t a, uint32_t b) { return __hiloint2double((int)b, (int)a); }
};

// One update of a vector from its neighbours (the step kernels' arithmetic).
// FP64 inside the integer adders' domain: pair sums by dadd_near, and xy of one of
// the two points too (the pipes retire 836 and 527 G additions/s); a vector with
// operands out of its reach is computed again with dadd_nn.  64^3 4.5 -> 4.2 us per
// iteration, 108^3 11.4 -> 10.0, against dadd_nn alone.  `whole`: the second value
// belongs to the grid.
template <bool EMU>
__device__ __forceinline__ void update(const double (&c)[2], const double (&ym)[2], const double (&yp)[2], const double (&zm)[2],
                                       const double (&zp)[2], double left, double right, bool whole, double (&v)[2]) {
  if constexpr (!EMU) {
    v[0] = finish1(nsum<double, false>(left, c[1], ym[0], yp[0], zm[0], zp[0]));
    v[1] = finish1(nsum<double, false>(c[0], right, ym[1], yp[1], zm[1], zp[1]));
  } else {
    int f0 = 0, f1 = 0;
    const double x0 = dadd_near(left, c[1], f0), y0 = dadd_near(ym[0], yp[0], f0), z0 = dadd_near(zm[0], zp[0], f0);
    const double x1 = dadd_near(c[0], right, f1), y1 = dadd_near(ym[1], yp[1], f1), z1 = dadd_near(zm[1], zp[1], f1);
    v[0] = finish1(__dadd_rn(__dadd_rn(x0, y0), z0));
    v[1] = finish1(__dadd_rn(dadd_near(x1, y1, f1), z1));
    if (!whole) f1 = 0;
    if ((f0 | f1) < 0) {
      if (f0 < 0) f0 = sum_far(left, c[1], ym[0], yp[0], zm[0], zp[0], false);
      if (f1 < 0) f1 = sum_far(c[0], right, ym[1], yp[1], zm[1], zp[1], true);
      if ((f0 | f1) < 0) {
        v[0] = finish1(nsum<double, true>(left, c[1], ym[0], yp[0], zm[0], zp[0]));
        v[1] = finish1(nsum<double, true>(c[0], right, ym[1], yp[1], zm[1], zp[1]));
      }
    }
  }
}
template <bool EMU>
__device__ __forceinline__ void update(const float (&c)[4], const float (&ym)[4], const float (&yp)[4], const float (&zm)[4],
                                       const float (&zp)[4], float left, float right, bool, float (&v)[4]) {
  float s[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    s[q] = nsum<float, false>(q == 0 ? left : c[q > 0 ? q - 1 : 0], q == 3 ? right : c[q < 3 ? q + 1 : 3], ym[q], yp[q], zm[q], zp[q]);
  finish_vec(s, v);
}

constexpr uint64_t kResStartNs = 30000000000ull;

// Threads per CTA: as many as the registers of an update allow (FP32 64, FP64
// 85 per thread), since the sweep is latency-bound with fewer warps: one box of
// 4096 FP32 points took 1.9 us with 512 threads, 1.3 with 1024.
template <typename T> constexpr int kResThreads = sizeof(T) == 4 ? 1024 : 768;

// Geometry of the box in shared memory: rows of P = whole vectors + one vector
// on either side (the x halos are its nearest values), ny + 2 rows, nz + 2 planes.
struct BoxView {
  int nx, ny, nz, nvx, P, plane, nv;
  uint32_t mp, mr;  // reciprocals of a plane's and a row's length in vectors
};

// A sweep goes through the box's vectors in the order of a table: those on a face
// that is sent come first, so that their packets travel while the rest is
// computed.  An entry is the vector's place (16-byte units, 14 bits) and two flags.
constexpr uint32_t kTabShell = 0x8000u;    // on a face with a neighbour
constexpr uint32_t kTabPartial = 0x4000u;  // the grid's last column, not a whole vector
constexpr uint32_t kTabPlace = 0x3FFFu;

// Place (16-byte units) -> column, row and plane of a vector in the box.
__device__ __forceinline__ void vec_place(const BoxView& G, int at, int& tx, int& j, int& k) {
  const int pv = (G.ny + 2) * (G.nvx + 2), rv = G.nvx + 2;
  k = fast_div(at, pv, G.mp);
  const int r = at - k * pv;
  j = fast_div(r, rv, G.mr);
  tx = r - j * rv - 1;
  k -= 1;
  j -= 1;
}

// Send the faces that the vector at `at` (values u) lies on.
template <typename T>
__device__ __forceinline__ void send_faces(const BoxView& G, const ResBox& X, uint4* packets, int at, const T (&u)[V16<T>::N],
                                        uint32_t seq, int par) {
  constexpr int VEC = V16<T>::N;
  int tx, j, k;
  vec_place(G, at, tx, j, k);
  uint32_t w[4];
  Words<T>::vec(u, w);
  for (int f = YM; f <= ZP; ++f) {
    const bool z = f >= ZM;
    const int edge = z ? (f == ZM ? 0 : G.nz - 1) : (f == YM ? 0 : G.ny - 1);
    if (!(X.faces >> f & 1) || (z ? k : j) != edge) continue;
    uint4* d = packets + X.out_base[f] + (par ? X.out_units[f] : 0u) + 2 * ((z ? j : k) * G.nvx + tx);
    st_packet(d, w[0], w[1], seq);
    st_packet(d + 1, w[2], w[3], seq);
  }
  for (int f = XM; f <= XP; ++f) {
    if (!(X.faces >> f & 1) || tx != (f == XM ? 0 : G.nvx - 1)) continue;
    uint32_t a, b;
    Words<T>::one(f == XM ? u[0] : u[VEC - 1], a, b);  // (an inner x cut is on a vector boundary)
    st_packet(packets + X.out_base[f] + (par ? X.out_units[f] : 0u) + k * G.ny + j, a, b, seq);
  }
}

// All updates of one iteration: src -> dst, surfaces sent with `seq` (not in the
// last iteration).
template <typename T, bool EMU>
__device__ __forceinline__ void box_sweep(const BoxView& G, const ResBox& X, const uint16_t* tab, const T* __restrict__ src,
                                          T* __restrict__ dst, uint4* packets, bool sends, uint32_t seq, int par) {
  constexpr int VEC = V16<T>::N;
  for (int v = threadIdx.x; v < G.nv; v += kResThreads<T>) {
    const uint32_t e = tab[v];
    const int off = (int)(e & kTabPlace) * VEC;
    T c[VEC], ym[VEC], yp[VEC], zm[VEC], zp[VEC], u[VEC];
    V16<T>::load(src + off, c);
    V16<T>::load(src + off - G.P, ym);
    V16<T>::load(src + off + G.P, yp);
    V16<T>::load(src + off - G.plane, zm);
    V16<T>::load(src + off + G.plane, zp);
    const T left = src[off - 1], right = src[off + VEC];
    update<EMU>(c, ym, yp, zm, zp, left, right, !(e & kTabPartial), u);
    if (!(e & kTabPartial)) {
      V16<T>::store(dst + off, u);
    } else {  // the rest of the vector is x halo and padding
      const int real = (G.nx - 1) % VEC + 1;
#pragma unroll
      for (int q = 0; q < VEC - 1; ++q)
        if (q < real) dst[off + q] = u[q];
    }
    if (sends && (e & kTabShell)) send_faces<T>(G, X, packets, off / VEC, u, seq, par);
  }
}

template <typename T>
__global__ void __launch_bounds__(kResThreads<T>, 1) k_resident(ResLaunch a) {
  constexpr int VEC = V16<T>::N, NT = kResThreads<T>;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ ResBox X;
  __shared__ ResGrid R;
  __shared__ int s_tab;
  const int tid = threadIdx.x;
  if (tid == 0) s_tab = 0;
  for (int q = tid; q < (int)(sizeof(ResBox) / 4); q += NT) ((uint32_t*)&X)[q] = ((const uint32_t*)(a.boxes + blockIdx.x))[q];
  __syncthreads();
  for (int q = tid; q < (int)(sizeof(ResGrid) / 4); q += NT) ((uint32_t*)&R)[q] = ((const uint32_t*)(a.rgrids + X.rgrid))[q];
  const uint32_t base = *(volatile const uint32_t*)a.ctl;  // sequence number of the launch's first state
  if (tid == 0) atomicAdd(a.ctl + 2, 1u);                  // this CTA has started
  __syncthreads();
  const GridDev GD = a.grids[R.grid];
  if (GD.active) {
    BoxView G;
    G.nx = X.n[0];
    G.ny = X.n[1];
    G.nz = X.n[2];
    G.nvx = (G.nx + VEC - 1) / VEC;
    G.P = (G.nvx + 2) * VEC;
    G.plane = (G.ny + 2) * G.P;
    G.nv = G.nvx * G.ny * G.nz;
    const uint32_t pv = (G.ny + 2) * (G.nvx + 2), rv = G.nvx + 2;
    G.mp = (uint32_t)((0xFFFFFFFFull + pv) / pv);
    G.mr = (uint32_t)((0xFFFFFFFFull + rv) / rv);
    const int cells = (G.nz + 2) * G.plane;
    T* const even = (T*)smem;  // the two buffers; iteration t reads even + (t & 1) * cells
    uint16_t* tab = (uint16_t*)(even + 2 * cells);  // sweep order
    uint16_t* hdst = tab + G.nv;      // halo destinations, see below
    uint32_t* ax = (uint32_t*)(tab + (G.nv + X.n_vec + X.n_one + 1) / 2 * 2);  // per-axis block tables, x then y then z
    uint32_t* ay = ax + G.nx + 2;
    uint32_t* az = ay + G.ny + 2;
    // zeros first: padding stays finite and inside the integer adder's domain
    for (int q = tid; q < 2 * cells / VEC; q += NT) ((uint4*)smem)[q] = make_uint4(0u, 0u, 0u, 0u);
    for (int q = tid; q < G.nx + G.ny + G.nz + 6; q += NT) {
      const int d = q < G.nx + 2 ? 0 : q < G.nx + G.ny + 4 ? 1 : 2;
      const int e = d == 0 ? q : d == 1 ? q - (G.nx + 2) : q - (G.nx + G.ny + 4);
      ax[q] = axis_entry(R.mode, R.param[d], R.n[d], X.o[d] + e - 1);
    }
    // The sweep's order: shell vectors from the front, the others behind them.
    // Each warp takes 32 consecutive vectors and keeps their order.
    const int sent = (int)blockIdx.x == a.mute ? 0 : X.faces;
    for (int pass = 0; pass < 2; ++pass) {
      for (int vb = tid & ~31; vb < G.nv; vb += NT) {
        const int v = vb + (tid & 31), row = v / G.nvx, tx = v - row * G.nvx, k = row / G.ny, j = row - k * G.ny;
        bool shell = false;
        if (v < G.nv)
          shell = (tx == 0 && (sent >> XM & 1)) || (tx == G.nvx - 1 && (sent >> XP & 1)) || (j == 0 && (sent >> YM & 1)) ||
                  (j == G.ny - 1 && (sent >> YP & 1)) || (k == 0 && (sent >> ZM & 1)) || (k == G.nz - 1 && (sent >> ZP & 1));
        const bool mine = v < G.nv && shell == (pass == 0);
        const uint32_t m = __ballot_sync(0xffffffffu, mine);
        int at = 0;
        if ((tid & 31) == 0 && m) at = atomicAdd(&s_tab, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << (tid & 31)) - 1u));
        if (mine)
          tab[at] = (uint16_t)(((k + 1) * G.plane + (j + 1) * G.P) / VEC + 1 + tx | (shell ? kTabShell : 0u) |
                               ((tx + 1) * VEC > G.nx ? kTabPartial : 0u));
      }
      __syncthreads();
    }
    // Where each incoming entry goes: vectors (z then y faces) in 16-byte units,
    // single x values in values.
    for (int h = tid; h < X.n_vec + X.n_one; h += NT) {
      int e = h, at = 0;
      const int nzf = G.ny * G.nvx, nyf = G.nz * G.nvx, nxf = G.ny * G.nz;
      for (int f : {(int)ZM, (int)ZP, (int)YM, (int)YP, (int)XM, (int)XP}) {
        if (!(X.faces & 1 << f)) continue;
        const int n = f >= ZM ? nzf : f >= YM ? nyf : nxf;
        if (e >= n) {
          e -= n;
          continue;
        }
        if (f >= ZM) at = ((f == ZM ? 0 : G.nz + 1) * G.plane + (e / G.nvx + 1) * G.P) / VEC + 1 + e % G.nvx;
        else if (f >= YM) at = ((e / G.nvx + 1) * G.plane + (f == YM ? 0 : G.ny + 1) * G.P) / VEC + 1 + e % G.nvx;
        else at = (e / G.ny + 1) * G.plane + (e % G.ny + 1) * G.P + (f == XM ? VEC - 1 : VEC + G.nx);
        break;
      }
      hdst[h] = (uint16_t)at;
    }
    __syncthreads();
    // Initial state: interior and the six halo faces, from the blocks (a face
    // between two boxes: the neighbouring cells themselves) or, outside the
    // grid, from the Dirichlet slots, which both buffers keep.
    const int p = (int)((a.it0 - GD.start_iter) & 1);
    const int ex = G.nx + 2, ey = G.ny + 2, ext = ex * ey * (G.nz + 2);
    for (int e0 = tid; e0 < ext; e0 += 8 * NT) {
      T val[8];
      int at[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * NT;
        at[u] = -1;
        if (e >= ext) continue;
        const int r = e / ex, i = e - r * ex, k = r / ey, j = r - k * ey;
        const bool hx = i == 0 || i == G.nx + 1, hy = j == 0 || j == G.ny + 1, hz = k == 0 || k == G.nz + 1;
        if (hx + hy + hz > 1) continue;
        const uint32_t tx = ax[i], ty = ay[j], tz = az[k];
        const int li = tx & 0xFFFF, lj = ty & 0xFFFF, lk = tz & 0xFFFF;
        const BlockDev& B = a.blocks[R.block0 + ((int)(tz >> 16 & 0x7FFF) * R.cnt[1] + (int)(ty >> 16 & 0x7FFF)) * R.cnt[0] +
                                     (int)(tx >> 16 & 0x7FFF)];
        const T* s;
        if (tx & kOutside) s = (const T*)B.recv[i == 0 ? XM : XP][p] + (int64_t)lk * B.ry + lj;
        else if (ty & kOutside) s = (const T*)B.recv[j == 0 ? YM : YP][p] + (int64_t)lk * B.rx + li;
        else if (tz & kOutside) s = (const T*)B.recv[k == 0 ? ZM : ZP][p] + (int64_t)lj * B.rx + li;
        else s = (const T*)B.u[p] + (int64_t)lk * B.plane_pitch + (int64_t)lj * B.rx + li;
        val[u] = *s;
        at[u] = (k * G.plane + j * G.P + VEC - 1 + i) | (((tx | ty | tz) & kOutside) ? 1 << 30 : 0);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (at[u] >= 0) {
          even[at[u] & 0x3FFFFFFF] = val[u];
          if (at[u] >> 30) even[cells + (at[u] & 0x3FFFFFFF)] = val[u];
        }
    }
    const bool emu = sizeof(T) == 8 && a.emu && a.norms && a.norms[R.grid].emu_bad == 0u;
    bool ok = true;
    for (int64_t t = 0; t < a.n_iters; ++t) {
      T* src = even + ((t & 1) ? cells : 0);
      T* dst = even + ((t & 1) ? 0 : cells);
      if (t > 0) {
        // Surfaces of this iterate from the neighbours: every thread keeps up to
        // two vector entries and one x value in flight until all have arrived.
        const uint32_t seq = base + (uint32_t)t;
        const uint4* in = a.packets + X.in_base + ((t & 1) ? X.in_units : 0u);
        for (int h0 = tid; ok && (h0 < X.n_vec || h0 < X.n_one); h0 += 2 * NT) {
          // entries h0 and h0 + NT of the vectors; x values go in steps of NT, two rounds per step of 2 NT
          bool want[4] = {h0 < X.n_vec, h0 + NT < X.n_vec, h0 < X.n_one, h0 + NT < X.n_one};
          uint64_t t0 = 0, first = 0;
          for (uint32_t n = 0;; ++n) {
            uint32_t w[4][4];
            bool got[4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (want[q]) {
                const uint4* s = in + 2 * (h0 + q * NT);
                const bool g0 = ld_packet(s, w[q][0], w[q][1], seq), g1 = ld_packet(s + 1, w[q][2], w[q][3], seq);
                got[q] = g0 && g1;
              }
#pragma unroll
            for (int q = 2; q < 4; ++q)
              if (want[q]) got[q] = ld_packet(in + 2 * X.n_vec + h0 + (q - 2) * NT, w[q][0], w[q][1], seq);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (want[q] && got[q]) {
                want[q] = false;
                if (q < 2) *(uint4*)((char*)src + 16 * (int)hdst[h0 + q * NT]) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
                else src[hdst[X.n_vec + h0 + (q - 2) * NT]] = Words<T>::make(w[q][0], w[q][1]);
              }
            if (!(want[0] || want[1] || want[2] || want[3])) break;
            if ((n & 63u) != 63u) continue;
            const uint64_t now = globaltimer_ns();
            if (t0 == 0) t0 = first = now;
            bool stop = ld_volatile_u32(a.err) != DEV_OK || n > (1u << 30);
            if (now - t0 > a.wait_ns) {
              // the limit counts from when every CTA has started: other streams'
              // kernels may still hold some of the SMs
              if (ld_acquire_u32(a.ctl + 2) < gridDim.x && now - first < kResStartNs) t0 = now;
              else stop = true;
            }
            if (stop) {
              atomicCAS(a.err, (uint32_t)DEV_OK, (uint32_t)DEV_TIMEOUT);
              *(volatile uint32_t*)a.host_err = DEV_TIMEOUT;
              ok = false;
              break;
            }
          }
        }
      }
      ok = __syncthreads_and(ok) != 0;
      if (!ok) break;
      const bool sends = t + 1 < a.n_iters;
      const uint32_t seq = base + (uint32_t)(t + 1);
      const int par = (int)((t + 1) & 1);
      if (sizeof(T) == 8 && emu) box_sweep<T, true>(G, X, tab, src, dst, a.packets, sends, seq, par);
      else box_sweep<T, false>(G, X, tab, src, dst, a.packets, sends, seq, par);
    }
    __syncthreads();
    // The last iterate to the blocks, and their faces into the neighbours' slots.
    if (ok) {
      const int pe = (int)((a.it0 + a.n_iters - GD.start_iter) & 1);
      const int pts = G.nx * G.ny * G.nz;
      const T* src = even + ((a.n_iters & 1) ? cells : 0);
      for (int e = tid; e < pts; e += NT) {
        const int r = e / G.nx, i = e - r * G.nx, k = r / G.ny, j = r - k * G.ny;
        const uint32_t tx = ax[i + 1], ty = ay[j + 1], tz = az[k + 1];
        const int li = tx & 0xFFFF, lj = ty & 0xFFFF, lk = tz & 0xFFFF;
        const BlockDev& B = a.blocks[R.block0 + ((int)(tz >> 16) * R.cnt[1] + (int)(ty >> 16)) * R.cnt[0] + (int)(tx >> 16)];
        const T val = src[(k + 1) * G.plane + (j + 1) * G.P + VEC + i];
        ((T*)B.u[pe])[(int64_t)lk * B.plane_pitch + (int64_t)lj * B.rx + li] = val;
        auto put = [&](int f, int64_t at) {
          T* d = (T*)B.send[f][pe];
          if (d) d[at] = val;
        };
        if (li == 0) put(XM, (int64_t)lk * B.ry + lj);
        if (li == B.nx - 1) put(XP, (int64_t)lk * B.ry + lj);
        if (lj == 0) put(YM, (int64_t)lk * B.rx + li);
        if (lj == B.ny - 1) put(YP, (int64_t)lk * B.rx + li);
        if (lk == 0) put(ZM, (int64_t)lj * B.rx + li);
        if (lk == B.nz - 1) put(ZP, (int64_t)lj * B.rx + li);
      }
    }
  }
  // the last CTA advances the sequence numbers for the next launch
  if (tid == 0 && atomicAdd(a.ctl + 1, 1u) == gridDim.x - 1) {
    a.ctl[1] = 0u;
    a.ctl[2] = 0u;
    a.ctl[0] = base + (uint32_t)a.n_iters;
  }
}

// The shared-memory opt-in, once per device.
template <typename T>
cudaError_t resident_attr() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  const uint64_t bit = 1ull << (dev & 63);
  if (e != cudaSuccess || (dev < 64 && (done.load() & bit))) return e;
  e = cudaFuncSetAttribute(k_resident<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem);
  if (e == cudaSuccess && dev < 64) done.fetch_or(bit);
  return e;
}

// ---- host: cutting grids into boxes -------------------------------------------

// Piece i of n cut into c near-equal pieces.
int piece_at(int n, int c, int i) { return i * (n / c) + (i < n % c ? i : n % c); }
int piece_len(int n, int c, int i) { return n / c + (i < n % c ? 1 : 0); }
int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Incoming entries of a box with extents n (nvx vectors wide) and these faces.
int vec_entries(const int* n, int nvx, int faces) {
  return n[1] * nvx * ((faces >> ZM & 1) + (faces >> ZP & 1)) + n[2] * nvx * ((faces >> YM & 1) + (faces >> YP & 1));
}
int one_entries(const int* n, int faces) { return n[1] * n[2] * ((faces >> XM & 1) + (faces >> XP & 1)); }

int64_t box_smem(const int* n, int nvx, int vec, int n_vec, int n_one) {
  const int64_t cells = (int64_t)(n[2] + 2) * (n[1] + 2) * (nvx + 2) * vec;
  return 2 * cells * (16 / vec) + 2 * ((nvx * n[1] * n[2] + n_vec + n_one + 1) / 2 * 2) + 4 * (n[0] + n[1] + n[2] + 6);
}

struct Cut {
  int c[3];
  double ns;  // estimated time of an iteration; < 0: does not fit
};

// Best cut of a grid into exactly or up to k boxes, for every k <= most.  The
// estimate of the largest box: its points at the arithmetic's rate of one SM
// (two-pipe FP64 1.0 ns, FP32 0.17 ns per point, the sweep measured alone), its
// surface entries (a packet each way through L2), and the trip and barrier.
std::vector<Cut> grid_cuts(const int* N, int dtype, int most) {
  const int vec = dtype == 0 ? 2 : 4;
  const double per_pt = dtype == 0 ? 1.0 : 0.17, per_vec = 0.5, per_one = 0.4, trip = 1000.0;
  std::vector<Cut> best(most + 1, Cut{{0, 0, 0}, -1.0});
  const int NV = ceil_div(N[0], vec);
  for (int cx = 1; cx <= std::min(NV, most); ++cx)
    for (int cy = 1; cy <= std::min(N[1], most / cx); ++cy)
      for (int cz = 1; cz <= std::min(N[2], most / cx / cy); ++cz) {
        const int nvx = ceil_div(NV, cx), n[3] = {nvx * vec, ceil_div(N[1], cy), ceil_div(N[2], cz)};
        int faces = 0;  // of a box in the middle
        if (cx > 1) faces |= 1 << XM | (cx > 2 ? 1 << XP : 0);
        if (cy > 1) faces |= 1 << YM | (cy > 2 ? 1 << YP : 0);
        if (cz > 1) faces |= 1 << ZM | (cz > 2 ? 1 << ZP : 0);
        const int64_t pts = (int64_t)n[0] * n[1] * n[2];
        if (pts > 1 << 16) continue;  // (keeps the products below in range; the table's 14-bit places hold any box that fits)
        const int nv = vec_entries(n, nvx, faces), no = one_entries(n, faces);
        if (box_smem(n, nvx, vec, nv, no) > kResSmem) continue;
        const double ns = pts * per_pt + nv * per_vec + no * per_one + (faces ? trip : 300.0);
        Cut& b = best[cx * cy * cz];
        if (b.ns < 0 || ns < b.ns) b = Cut{{cx, cy, cz}, ns};
      }
  for (int k = 1; k <= most; ++k)
    if (k > 1 && best[k - 1].ns >= 0 && (best[k].ns < 0 || best[k].ns >= best[k - 1].ns)) best[k] = best[k - 1];
  return best;
}

}  // namespace

bool resident_plan(const std::vector<ResGrid>& grids, int dtype, int n_ctas, ResPlan* P) {
  P->boxes.clear();
  const int vec = dtype == 0 ? 2 : 4, elem = 16 / vec, ng = (int)grids.size();
  if (ng < 1 || ng > n_ctas) return false;
  int64_t bytes = 0;
  for (const ResGrid& g : grids) {
    bytes += 2ll * elem * g.n[0] * g.n[1] * g.n[2];
    for (int d = 0; d < 3; ++d)
      if (g.cnt[d] > 0x7FFF) return false;  // the axis tables hold block numbers in 15 bits
    if (bytes > (int64_t)n_ctas * kResSmem) return false;
  }
  // Every grid starts at the fewest boxes that fit; then the slowest grid gets
  // more while there are CTAs left.
  std::vector<std::vector<Cut>> cuts(ng);
  std::vector<int> k(ng, 0);
  int total = 0;
  std::vector<int> most(ng);  // boxes considered for a grid: four times its share of the points
  for (int g = 0; g < ng; ++g) {
    const ResGrid& R = grids[g];
    const int64_t share = 2ll * elem * R.n[0] * R.n[1] * R.n[2] * n_ctas / bytes;
    most[g] = (int)std::min<int64_t>(n_ctas - (ng - 1), 4 * share + 4);
    int same = g;  // (grids of one size are cut once)
    for (int q = 0; q < g && same == g; ++q)
      if (std::equal(R.n, R.n + 3, grids[q].n)) same = q;
    cuts[g] = same == g ? grid_cuts(R.n, dtype, most[g]) : cuts[same];
    for (k[g] = 1; k[g] <= most[g] && cuts[g][k[g]].ns < 0; ++k[g]) {
    }
    if (k[g] > most[g]) return false;
    total += k[g];
  }
  if (total > n_ctas) return false;
  for (;;) {
    int s = 0;
    for (int g = 1; g < ng; ++g)
      if (cuts[g][k[g]].ns > cuts[s][k[s]].ns) s = g;
    int next = k[s] + 1;
    while (next <= most[s] && cuts[s][next].ns >= cuts[s][k[s]].ns) ++next;
    if (next > most[s] || total + next - k[s] > n_ctas) break;
    total += next - k[s];
    k[s] = next;
  }
  // the boxes, then where each sends its faces
  uint32_t units = 0;
  int smem = 0;
  std::vector<int> first(ng);
  for (int g = 0; g < ng; ++g) {
    const ResGrid& R = grids[g];
    const Cut& C = cuts[g][k[g]];
    const int NV = ceil_div(R.n[0], vec);
    first[g] = (int)P->boxes.size();
    for (int z = 0; z < C.c[2]; ++z)
      for (int y = 0; y < C.c[1]; ++y)
        for (int x = 0; x < C.c[0]; ++x) {
          ResBox b{};
          b.rgrid = g;
          b.o[0] = piece_at(NV, C.c[0], x) * vec;
          b.n[0] = std::min(piece_len(NV, C.c[0], x) * vec, R.n[0] - b.o[0]);
          b.o[1] = piece_at(R.n[1], C.c[1], y);
          b.n[1] = piece_len(R.n[1], C.c[1], y);
          b.o[2] = piece_at(R.n[2], C.c[2], z);
          b.n[2] = piece_len(R.n[2], C.c[2], z);
          b.faces = (x > 0) << XM | (x + 1 < C.c[0]) << XP | (y > 0) << YM | (y + 1 < C.c[1]) << YP | (z > 0) << ZM |
                    (z + 1 < C.c[2]) << ZP;
          const int nvx = ceil_div(b.n[0], vec);
          b.n_vec = vec_entries(b.n, nvx, b.faces);
          b.n_one = one_entries(b.n, b.faces);
          b.in_base = units;
          b.in_units = (uint32_t)(2 * b.n_vec + b.n_one);
          units += 2 * b.in_units;
          smem = std::max<int>(smem, (int)box_smem(b.n, nvx, vec, b.n_vec, b.n_one));
          P->boxes.push_back(b);
        }
  }
  // Offset of face f's entries in a box's incoming buffer (16-byte units):
  // vectors of zm, zp, ym, yp (two each), then values of xm, xp.
  auto region = [&](const ResBox& b, int f) {
    const int nvx = ceil_div(b.n[0], vec);
    int at = 0;
    for (int q : {(int)ZM, (int)ZP, (int)YM, (int)YP, (int)XM, (int)XP}) {
      if (q == f) break;
      if (!(b.faces >> q & 1)) continue;
      at += q >= ZM ? 2 * b.n[1] * nvx : q >= YM ? 2 * b.n[2] * nvx : b.n[1] * b.n[2];
    }
    return (uint32_t)at;
  };
  for (size_t q = 0; q < P->boxes.size(); ++q) {
    ResBox& b = P->boxes[q];
    const Cut& C = cuts[b.rgrid][k[b.rgrid]];
    const int step[3] = {1, C.c[0], C.c[0] * C.c[1]};
    for (int f = 0; f < 6; ++f) {
      if (!(b.faces >> f & 1)) continue;
      const ResBox& n = P->boxes[q + ((f & 1) ? step[f / 2] : -step[f / 2])];
      b.out_base[f] = n.in_base + region(n, opposite(f));
      b.out_units[f] = n.in_units;
    }
  }
  P->packet_units = units;
  P->smem = smem;
  P->iter_ns = 0.0;
  int64_t points = 0, largest = 0;
  for (int g = 0; g < ng; ++g) {
    P->iter_ns = std::max(P->iter_ns, cuts[g][k[g]].ns);
    points += (int64_t)grids[g].n[0] * grids[g].n[1] * grids[g].n[2];
  }
  for (const ResBox& b : P->boxes) largest = std::max<int64_t>(largest, (int64_t)b.n[0] * b.n[1] * b.n[2]);
  // the launch, its tables and the state's way in and out; an iteration as a
  // launch of its own
  P->once_ns = 14000.0 + 1.5 * (double)largest;
  P->launch_ns = 4300.0 + (double)points * (dtype == 0 ? 0.0066 : 0.00154);
  return true;
}

cudaError_t launch_resident(const ResLaunch& a, cudaStream_t s) {
  if (a.n_boxes <= 0 || a.n_iters <= 0) return cudaSuccess;
  cudaError_t e = a.dtype == 0 ? resident_attr<double>() : resident_attr<float>();
  if (e != cudaSuccess) return e;
  ResLaunch args = a;
  void* params[] = {&args};
  const void* fn = a.dtype == 0 ? (const void*)k_resident<double> : (const void*)k_resident<float>;
  return cudaLaunchCooperativeKernel(fn, dim3(a.n_boxes), dim3(a.dtype == 0 ? kResThreads<double> : kResThreads<float>), params, a.smem, s);
}

}  // namespace jgb
