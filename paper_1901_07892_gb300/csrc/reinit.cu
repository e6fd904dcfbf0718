// Reinitialisation of the flow level set (Sec. 4.1, the eikonal equation
// d phi/d tau + sgn(phi~)(|grad phi| - 1) = 0 marched to steady state).
//
// Per pseudo-time stage every cell evaluates, along each axis with more than
// one cell, the second-order ENO one-sided differences of phi; where phi~
// changes sign towards a neighbour the difference is taken across the
// interface instead (subcell fix of Min 2010: the interface sits at the zero
// of the quadratic through phi~ with the minmod second difference, and phi
// is 0 there).  The Godunov Hamiltonian of sgn(phi~) gives |grad phi|; the
// local step is cfl * min(h, subcell distances).  Two stages form one TVD
// Runge-Kutta step.  sgn(phi~) and the subcell distances come from phi~
// throughout (immobile interface, Son 2005).  Neumann mirror ghosts.
//
// phi~ enters through a one-byte code per cell (its sign and the axes along
// which it changes sign), made once per call.  Per stage phi is read once and
// written once (plus phi^m in the second stage) with the code byte: 9 or 13 bytes
// per cell in float32.  Two kernels march a z-chunk; use_pairs chooses.
//
// k_reinit: one cell per thread, tile 32 x 8, the subcell distances in the march,
// chunks down to one plane, so that a small grid still has blocks for every SM.
// Bound by the latency of a plane on small grids, by the float64 pipe in float64.
//
// k_reinit_pair: two neighbouring cells in x per thread; the planes of phi (tile of
// 64 x 8 cells with a two-cell halo, ghosts mirrored through the copies' source
// addresses) come through a ring in shared memory filled by cp.async two planes
// ahead.  The one-sided differences on the two sides of a cell face differ only in
// the sign of their second-order part, so each face's difference and minmod are
// formed once: the pair shares them in x, the march hands them on in z.  The cells
// next to the interface are listed with the code and a second launch per stage
// gives them their subcell distances (inside this march that path cost registers
// and instruction cache: 204 us per stage).  Bound by instruction issue (190 warp
// instructions per 32 cells, 76 % of the slots): 112 us per stage at 256^3 in
// float32 and 10 us for the listed cells; k_reinit 190 us.
#include <algorithm>

#include "internal.h"

namespace wsi {

static constexpr int RX = 32, RY = 8;  // threads
// k_reinit_pair: a staged plane (two cells per thread in x, two-cell halo) and its ring
static constexpr int RHX = 2 * RX + 4, RHY = RY + 4, RPL = RHX * RHY, RSLOT = 8;

__device__ __forceinline__ int mirror_cell(int m, int n) {
  if (m < 0) m = -m - 1;
  else if (m >= n) m = 2 * n - 1 - m;
  return clampi(m, 0, n - 1);
}

template <typename T>
struct ReinitAxes {
  T h[3], ih[3];
  int active[3];  // axis has more than one cell
  T cfl;
};

template <typename T>
__device__ __forceinline__ T minmod_(T a, T b) {
  return a * b > T(0) ? (fabs(a) < fabs(b) ? a : b) : T(0);
}

// fraction of the cell spacing from the centre holding a to the zero of the
// quadratic through a (at 0) and b (at 1) with second difference c, a*b < 0:
// local coordinate t = xi - 1/2, quadratic c0 + c1 t + c2 t^2; the zero in
// [-1/2, 1/2] is the root of smaller magnitude (stable form, linear limit
// for c = 0)
template <typename T>
__device__ __forceinline__ T iface_frac(T a, T b, T c) {
  const T c2 = T(0.5) * c, c1 = b - a, c0 = T(0.5) * (a + b) - T(0.125) * c;
  const T disc = fmax(c1 * c1 - T(4) * c2 * c0, T(0));
  return T(0.5) - T(2) * c0 / (c1 + copysign(sqrt(disc), c1));
}

template <typename T>
__device__ __forceinline__ double widen(T v);
template <>
__device__ __forceinline__ double widen<double>(double v) { return v; }
template <>
__device__ __forceinline__ double widen<float>(float v) { return f2d_fast(v); }

// Per-cell code of phi~, computed once per call (phi~ is fixed): bits 0-1
// the sign (0 zero, 1 positive, 2 negative); bit 2 + 2d (3 + 2d) set when
// phi~ changes sign towards the lower (upper) neighbour along axis d.  A
// mirror ghost equals its cell, so no crossing is flagged across a wall.
template <typename T>
__global__ void k_reinit_code(GridDev g, const T* __restrict__ q0, unsigned char* __restrict__ code, int* list,
                              int* count) {
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const size_t plane = (size_t)n0 * n1, n = plane * n2;
  for (size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x; id < n; id += (size_t)gridDim.x * blockDim.x) {
    const int row = (int)id / n0, i = (int)id - row * n0, k = row / n1, j = row - k * n1;
    const T q = q0[id];
    unsigned c = q > T(0) ? 1u : (q < T(0) ? 2u : 0u);
    const int cc[3] = {i, j, k}, nn[3] = {n0, n1, n2};
    const size_t sd[3] = {1, (size_t)n0, plane};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (cc[d] > 0 && q * q0[id - sd[d]] < T(0)) c |= 4u << (2 * d);
      if (cc[d] + 1 < nn[d] && q * q0[id + sd[d]] < T(0)) c |= 8u << (2 * d);
    }
    code[id] = (unsigned char)c;
    if (list && (c >> 2)) list[atomicAdd(count, 1)] = (int)id;  // next to the interface (any order will do)
  }
}

// subcell distances of one axis (rare path: the cell is next to the
// interface along this axis); taps of phi~ from global memory
template <typename T>
__device__ __forceinline__ void subcell_axis(const T* __restrict__ q0, size_t id, int c, int n, size_t stride,
                                             unsigned bits, const T p[5], T h, T ih, T mp, T mm, T& Dm, T& Dp,
                                             T& hloc) {
  T q[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) q[m] = q0[id + (ptrdiff_t)(mirror_cell(c - 2 + m, n) - c) * (ptrdiff_t)stride];
  const T qc = q[1] - T(2) * q[2] + q[3];
  if (bits & 2u) {
    const T qp = q[2] - T(2) * q[3] + q[4];
    const T hp = fmin(fmax(h * iface_frac(q[2], q[3], minmod_(qc, qp)), T(1e-10) * h), h);
    Dp = -p[2] / hp - T(0.5) * hp * mp * ih * ih;
    hloc = fmin(hloc, hp);
  }
  if (bits & 1u) {
    const T qm = q[0] - T(2) * q[1] + q[2];
    const T hm = fmin(fmax(h * iface_frac(q[2], q[1], minmod_(qc, qm)), T(1e-10) * h), h);
    Dm = p[2] / hm + T(0.5) * hm * mm * ih * ih;
    hloc = fmin(hloc, hm);
  }
}

// one stage (see k_reinit_pair) of the listed cells, those next to the interface:
// the three axes with subcell distances
template <typename T>
__global__ void __launch_bounds__(128) k_reinit_near(GridDev g, ReinitAxes<T> ax,
                                                     const unsigned char* __restrict__ code,
                                                     const int* __restrict__ list, const int* __restrict__ count,
                                                     const T* __restrict__ q0, const T* __restrict__ pin,
                                                     const T* pavg, T* pout, double* out64) {
  const int n0 = g.n[0], n1 = g.n[1];
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < count[0]; t += gridDim.x * blockDim.x) {
    const int id = list[t], row = id / n0, k = row / n1;
    const int cc[3] = {id - row * n0, row - k * n1, k};
    const unsigned cd = code[id];
    const T s = (cd & 3u) == 1u ? T(1) : ((cd & 3u) == 2u ? T(-1) : T(0));
    T g2 = T(0), hmin = T(0);
    bool any = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (!ax.active[d]) continue;
      const int c = cc[d], stride = d == 0 ? 1 : (d == 1 ? n0 : n0 * n1);
      T p[5];
#pragma unroll
      for (int m = 0; m < 5; ++m) p[m] = pin[id + (mirror_cell(c - 2 + m, g.n[d]) - c) * stride];
      const T pm = p[0] - T(2) * p[1] + p[2], pc = p[1] - T(2) * p[2] + p[3], pp = p[2] - T(2) * p[3] + p[4];
      const T mp = minmod_(pc, pp), mm = minmod_(pc, pm);
      T Dp = (p[3] - p[2]) * ax.ih[d] - T(0.5) * mp * ax.ih[d];
      T Dm = (p[2] - p[1]) * ax.ih[d] + T(0.5) * mm * ax.ih[d];
      T hloc = ax.h[d];
      const unsigned bits = (cd >> (2 + 2 * d)) & 3u;
      if (bits)
        subcell_axis(q0, (size_t)id, c, g.n[d], (size_t)stride, bits, p, ax.h[d], ax.ih[d], mp, mm, Dm, Dp, hloc);
      // Godunov: s > 0 takes max(D-, 0) and min(D+, 0), s < 0 min(D-, 0) and
      // max(D+, 0); both are max(s D-, -s D+, 0) in magnitude
      const T u = fmax(fmax(s * Dm, -s * Dp), T(0));
      g2 += u * u;
      hmin = any ? fmin(hmin, hloc) : hloc;
      any = true;
    }
    const T dtau = any ? ax.cfl * hmin : T(0);
    T v = pin[id] + dtau * (-s * (sqrt(g2) - T(1)));
    if (pavg) v = T(0.5) * pavg[id] + T(0.5) * v;
    if (out64) out64[id] = out64[id] + widen<T>(v - q0[id]);
    else pout[id] = v;
  }
}

template <typename T>
__device__ __forceinline__ void cp_elem(T* dst, const T* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// Godunov term of one axis from the difference q and second-order part h of the
// faces below (l) and above (u) the cell
template <typename T>
__device__ __forceinline__ T godunov(T s, T ih, T ql, T hl, T qu, T hu) {
  const T Dp = qu * ih - hu, Dm = ql * ih + hl;
  return fmax(fmax(s * Dm, -s * Dp), T(0));
}

// One stage: v = pin + dtau L(pin);  with pavg:  v = (pavg + v) / 2.
// Written to pout, or with out64 (float32 path, last stage) as the change
// v - phi~ added to the float64 level set in out64.
//
// One cell per thread: the plane's tile in shared memory, the next plane's values
// on their way in registers meanwhile, the z taps in a five-entry window.  In
// float64 the face below is handed on from the plane before: 7260 -> 6790 us for
// 16 stages of 128^3 (float32, bound by issue and latency: 0 to 2 % more).
template <typename T>
__global__ void __launch_bounds__(RX* RY) k_reinit(GridDev g, ReinitAxes<T> ax,
                                                   const unsigned char* __restrict__ code,
                                                   const T* __restrict__ q0, const T* __restrict__ pin,
                                                   const T* pavg, T* pout, double* out64, int zchunk) {
  constexpr int HX = RX + 4, HY = RY + 4, NS = (HX * HY + RX * RY - 1) / (RX * RY);
  __shared__ T sP[HY * HX];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * RX + tx;
  const int x0 = blockIdx.x * RX, y0 = blockIdx.y * RY;
  const int i = x0 + tx, j = y0 + ty;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const bool inside = i < n0 && j < n1;
  const int k0 = blockIdx.z * zchunk;
  const int k1 = min(k0 + zchunk, n2);
  const size_t plane = (size_t)n0 * n1;
  int soff[NS];
#pragma unroll
  for (int r = 0; r < NS; ++r) {
    const int t = tid + r * RX * RY;
    soff[r] = -1;
    if (t < HX * HY) {
      const int hy = t / HX, hx = t - hy * HX;
      soff[r] = mirror_cell(y0 - 2 + hy, n1) * n0 + mirror_cell(x0 - 2 + hx, n0);
    }
  }
  const size_t col = (size_t)min(j, n1 - 1) * n0 + min(i, n0 - 1);
  T zp[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) zp[m] = pin[(size_t)mirror_cell(k0 - 2 + m, n2) * plane + col];
  // software pipeline: the tile, code byte and next z tap of plane k + 1
  // are loaded while plane k is computed
  T nxt[NS];
#pragma unroll
  for (int r = 0; r < NS; ++r) nxt[r] = soff[r] >= 0 ? pin[(size_t)k0 * plane + soff[r]] : T(0);
  // z state (float64): the second difference at k, minmod and difference of the
  // face below
  constexpr bool CARRY = sizeof(T) == 8;
  T zz = T(0), zm = T(0), zd = T(0);
  if (CARRY && ax.active[2]) {
    zz = zp[1] - T(2) * zp[2] + zp[3];
    zm = minmod_(zz, zp[0] - T(2) * zp[1] + zp[2]);
    zd = zp[2] - zp[1];
  }
  unsigned cd_next = inside && k0 < k1 ? code[(size_t)k0 * plane + col] : 0u;
  for (int k = k0; k < k1; ++k) {
    const size_t id = (size_t)k * plane + col;
    const unsigned cd = cd_next;
#pragma unroll
    for (int r = 0; r < NS; ++r)
      if (soff[r] >= 0) sP[tid + r * RX * RY] = nxt[r];
    __syncthreads();
    if (k + 1 < k1) {
#pragma unroll
      for (int r = 0; r < NS; ++r)
        if (soff[r] >= 0) nxt[r] = pin[(size_t)(k + 1) * plane + soff[r]];
      cd_next = inside ? code[id + plane] : 0u;
    }
    const T z_in = pin[(size_t)mirror_cell(k + 3, n2) * plane + col];
    if (inside) {
      const T s = (cd & 3u) == 1u ? T(1) : ((cd & 3u) == 2u ? T(-1) : T(0));
      T g2 = T(0), hmin = T(0);
      bool any = false;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (!ax.active[d]) continue;
        T p[5];
#pragma unroll
        for (int m = 0; m < 5; ++m)
          p[m] = d == 2 ? zp[m] : (d == 0 ? sP[(ty + 2) * HX + tx + m] : sP[(ty + m) * HX + tx + 2]);
        T mp, mm, dp = p[3] - p[2], dm;
        const T pp = p[2] - T(2) * p[3] + p[4];
        if (CARRY && d == 2) {
          mp = minmod_(zz, pp);
          mm = zm;
          dm = zd;
          zz = pp;
          zm = mp;
          zd = dp;
        } else {
          const T pm = p[0] - T(2) * p[1] + p[2], pc = p[1] - T(2) * p[2] + p[3];
          mp = minmod_(pc, pp);
          mm = minmod_(pc, pm);
          dm = p[2] - p[1];
        }
        T Dp = dp * ax.ih[d] - T(0.5) * mp * ax.ih[d];
        T Dm = dm * ax.ih[d] + T(0.5) * mm * ax.ih[d];
        T hloc = ax.h[d];
        const unsigned bits = (cd >> (2 + 2 * d)) & 3u;
        if (bits) {
          const int c = d == 0 ? i : (d == 1 ? j : k);
          const size_t stride = d == 0 ? 1 : (d == 1 ? (size_t)n0 : plane);
          subcell_axis(q0, id, c, g.n[d], stride, bits, p, ax.h[d], ax.ih[d], mp, mm, Dm, Dp, hloc);
        }
        // Godunov: s > 0 takes max(D-, 0) and min(D+, 0), s < 0 min(D-, 0)
        // and max(D+, 0); both are max(s D-, -s D+, 0) in magnitude
        const T t = fmax(fmax(s * Dm, -s * Dp), T(0));
        g2 += t * t;
        hmin = any ? fmin(hmin, hloc) : hloc;
        any = true;
      }
      const T dtau = any ? ax.cfl * hmin : T(0);
      T v = zp[2] + dtau * (-s * (sqrt(g2) - T(1)));
      if (pavg) v = T(0.5) * pavg[id] + T(0.5) * v;
      if (out64) out64[id] = out64[id] + widen<T>(v - q0[id]);
      else pout[id] = v;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 4; ++m) zp[m] = zp[m + 1];
    zp[4] = z_in;
  }
}

// The same of the cells away from the interface, two per thread
template <typename T>
__global__ void __launch_bounds__(RX* RY, sizeof(T) == 4 ? 4 : 2) k_reinit_pair(GridDev g, ReinitAxes<T> ax,
                                                   const unsigned char* __restrict__ code,
                                                   const T* __restrict__ q0, const T* __restrict__ pin,
                                                   const T* pavg, T* pout, double* out64, int zchunk) {
  constexpr int NS = (RPL + RX * RY - 1) / (RX * RY);
  extern __shared__ __align__(16) unsigned char reinit_smem[];
  T* const sP = reinterpret_cast<T*>(reinit_smem);
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * RX + tx;
  const int x0 = blockIdx.x * 2 * RX, y0 = blockIdx.y * RY;
  const int i = x0 + 2 * tx, j = y0 + ty;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int k0 = blockIdx.z * zchunk;
  const int k1 = min(k0 + zchunk, n2);
  const size_t plane = (size_t)n0 * n1;
  int soff[NS];
#pragma unroll
  for (int r = 0; r < NS; ++r) {
    const int t = tid + r * RX * RY, hy = t / RHX, hx = t - hy * RHX;
    soff[r] = t < RPL ? mirror_cell(y0 - 2 + hy, n1) * n0 + mirror_cell(x0 - 2 + hx, n0) : -1;
  }
  auto slot = [&](int k) { return (k & (RSLOT - 1)) * RPL; };
  auto issue = [&](int k) {
    if (k <= k1 + 1) {
      const T* src = pin + (size_t)mirror_cell(k, n2) * plane;
      T* dst = sP + slot(k) + tid;
#pragma unroll
      for (int r = 0; r < NS; ++r)
        if (soff[r] >= 0) cp_elem(dst + r * RX * RY, src + soff[r]);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const bool in0 = i < n0 && j < n1, in1 = i + 1 < n0 && j < n1;
  const int own = (ty + 2) * RHX + 2 * tx + 2;
  const T ihx = ax.ih[0], ihy = ax.ih[1], ihz = ax.ih[2];
  // the step away from the interface (no subcell distance)
  T hmin = T(0);
  bool any = false;
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (ax.active[d]) {
      hmin = any ? fmin(hmin, ax.h[d]) : ax.h[d];
      any = true;
    }
  const T dtau0 = any ? ax.cfl * hmin : T(0);
#pragma unroll 1
  for (int k = k0 - 2; k <= k0 + 3; ++k) issue(k);
  // z state of the two cells: phi at k and k + 1, the second difference at k,
  // the face below
  T p0[2], p1[2], zz[2], ql[2], hl[2];
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();  // planes up to k + 2 staged
    issue(k + 4);
    // a row beyond the grid (a whole warp): its copies only.  (float64, where the
    // pipe is the time: 127 x 101 x 99 291 -> 277 us per stage; in float32 the test
    // costs 1 %)
    if (sizeof(T) == 8 && j >= n1) continue;
    const T* P = sP + slot(k) + own;
    const size_t id = (size_t)k * plane + (size_t)j * n0 + i;
    unsigned cd[2] = {0u, 0u};
    T av[2] = {T(0), T(0)};
    if (in0) {
      cd[0] = code[id];
      if (pavg) av[0] = pavg[id];
    }
    if (in1) {
      cd[1] = code[id + 1];
      if (pavg) av[1] = pavg[id + 1];
    }
    if (k == k0) {
      const T* Pm2 = sP + slot(k - 2) + own;
      const T* Pm = sP + slot(k - 1) + own;
      const T* Pp = sP + slot(k + 1) + own;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        p0[c] = P[c];
        p1[c] = Pp[c];
        zz[c] = Pm[c] - T(2) * p0[c] + p1[c];
        const T zm = Pm2[c] - T(2) * Pm[c] + p0[c];
        ql[c] = p0[c] - Pm[c];
        hl[c] = T(0.5) * minmod_(zz[c], zm) * ihz;
      }
    }
    const T* Pz = sP + slot(k + 2) + own;
    T v[2], g2[2], s[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      s[c] = (cd[c] & 3u) == 1u ? T(1) : ((cd[c] & 3u) == 2u ? T(-1) : T(0));
      g2[c] = T(0);
    }
    if (ax.active[0]) {
      T q[6];
#pragma unroll
      for (int m = 0; m < 6; ++m) q[m] = P[m - 2];
      T dd[4], df[3], hf[3];
#pragma unroll
      for (int m = 0; m < 4; ++m) dd[m] = q[m] - T(2) * q[m + 1] + q[m + 2];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        df[m] = q[m + 2] - q[m + 1];
        hf[m] = T(0.5) * minmod_(dd[m], dd[m + 1]) * ihx;
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const T t = godunov<T>(s[c], ihx, df[c], hf[c], df[c + 1], hf[c + 1]);
        g2[c] += t * t;
      }
    }
    if (ax.active[1]) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const T a = P[c - 2 * RHX], b = P[c - RHX], m = P[c], u = P[c + RHX], w = P[c + 2 * RHX];
        const T dm = a - T(2) * b + m, dc = b - T(2) * m + u, dp = m - T(2) * u + w;
        const T t = godunov<T>(s[c], ihy, m - b, T(0.5) * minmod_(dc, dm) * ihy, u - m,
                               T(0.5) * minmod_(dc, dp) * ihy);
        g2[c] += t * t;
      }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const T p2 = Pz[c];
      const T zp = p0[c] - T(2) * p1[c] + p2;
      const T qu = p1[c] - p0[c], hu = T(0.5) * minmod_(zz[c], zp) * ihz;
      if (ax.active[2]) {
        const T t = godunov<T>(s[c], ihz, ql[c], hl[c], qu, hu);
        g2[c] += t * t;
      }
      v[c] = p0[c] + dtau0 * (-s[c] * (sqrt(g2[c]) - T(1)));
      zz[c] = zp;
      ql[c] = qu;
      hl[c] = hu;
      p0[c] = p1[c];
      p1[c] = p2;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (!(c ? in1 : in0) || (cd[c] >> 2)) continue;  // (the listed cells: k_reinit_near)
      T r = v[c];
      if (pavg) r = T(0.5) * av[c] + T(0.5) * r;
      if (out64) out64[id + c] = out64[id + c] + widen<T>(r - q0[id + c]);
      else pout[id + c] = r;
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

__global__ void k_to_f32(const double* __restrict__ a, float* __restrict__ b, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    b[t] = d2f_fast(a[t]);
}

// Planes per march: halved from zc down to zmin while there are fewer than per_sm
// blocks per SM
static int reinit_chunk(const GridDev& g, int cells, int zc, int zmin, int per_sm) {
  const long long base = (long long)cdiv(g.n[0], cells * RX) * cdiv(g.n[1], RY);
  while (zc > zmin && base * cdiv(g.n[2], zc) < 152LL * per_sm) zc /= 2;
  return zc;
}
// k_reinit: in float64 down to single planes until eight blocks per SM share the
// pipe (32^3 950 -> 520 us for 16 stages, 64 x 128 x 128 4390 -> 3720); in float32
// marches of four planes where four blocks per SM have one (128 x 128 x 64: 320 us,
// two planes 330), else shorter (32^3 187 -> 152)
template <typename T>
static int one_chunk(const GridDev& g) {
  if (sizeof(T) == 8) return reinit_chunk(g, 1, 32, 1, 8);
  return reinit_chunk(g, 1, reinit_chunk(g, 1, 32, 4, 8), 1, 4);
}
static int pair_chunk(const GridDev& g) { return reinit_chunk(g, 2, 32, 4, 4); }

// Whether a grid takes k_reinit_pair: its estimated time against k_reinit's, in
// cells of k_reinit per SM (float32 11.5 ps, float64 0.2 ns a cell at 152 SMs).  A
// cell of the pair kernel's padded tiles costs 0.57 (0.85) of one, whole waves of
// blocks counted; a listed cell 1.5, up to two layers across the shortest axis;
// what the two launches and the long start of a march add came out as 9500
// (-150).  In a 2-D grid of float64 the z terms that the pair kernel forms and
// drops decide.  Measured, 16 stages, k_reinit and pair: float32 32^3 150 and 290 us, 128^3 475 and 515,
// 160^3 770 and 840, 256 x 128 x 128 787 and 753, 192^3 1250 and 1100, 256^3 3100
// and 2300, 2048 x 2048 x 3 3250 and 5330; float64 12 x 8 x 8 290 and 1150, 64^3
// 1340 and 1280, 128 x 128 x 64 3610 and 3930, 120^3 6150 and 5550, 128^3 6790 and
// 6420, 160^3 12700 and 13700, 2048 x 2048 x 1 9930 and 11600.
template <typename T>
static bool use_pairs(const GridDev& g) {
  if (sizeof(T) == 8 && g.n[2] == 1) return false;
  const int zc = pair_chunk(g);
  const long long blocks = (long long)cdiv(g.n[0], 2 * RX) * cdiv(g.n[1], RY) * cdiv(g.n[2], zc);
  const int shortest = std::min(std::min(g.n[0], g.n[1]), g.n[2] > 1 ? g.n[2] : g.n[1]);
  const double pair = (double)((blocks + 151) / 152) * (2 * RX * RY) * std::min(zc, g.n[2]);
  const double near = 1.5 * 2.0 * g.n[0] * g.n[1] * g.n[2] / shortest / 152;
  const double one = (double)cdiv(g.n[0], RX) * RX * g.n[1] * g.n[2] / 152;
  return near + (sizeof(T) == 4 ? 0.57 * pair + 9500 : 0.85 * pair - 150) < one;
}

template <typename T>
static void stage(const GridDev& g, const ReinitAxes<T>& ax, bool pairs, const unsigned char* code, const int* list,
                  const T* q0, const T* pin, const T* pavg, T* pout, double* out64, cudaStream_t st) {
  const int nc = pairs ? 2 : 1, zc = pairs ? pair_chunk(g) : one_chunk<T>(g);
  const dim3 grid(cdiv(g.n[0], nc * RX), cdiv(g.n[1], RY), cdiv(g.n[2], zc)), block(RX, RY);
  ktimer_begin(KC_REINIT, st);
  if (pairs) {
    constexpr int smem = RSLOT * RPL * (int)sizeof(T);
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_reinit_pair<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    { k_reinit_pair<T><<<grid, block, smem, st>>>(g, ax, code, q0, pin, pavg, pout, out64, zc); WSI_COUNT(); }
    const int nb = (int)std::min<long long>(((long long)g.n[0] * g.n[1] * g.n[2] + 127) / 128, 152 * 8);
    { k_reinit_near<T><<<nb, 128, 0, st>>>(g, ax, code, list + 2, list, q0, pin, pavg, pout, out64); WSI_COUNT(); }
  } else {
    { k_reinit<T><<<grid, block, 0, st>>>(g, ax, code, q0, pin, pavg, pout, out64, zc); WSI_COUNT(); }
  }
  ktimer_end(KC_REINIT, st);
}

template <typename T>
void reinit_levelset(const GridDev& g, double* phi, int iters, double cfl, void* scratch, cudaStream_t st) {
  if (iters <= 0) return;
  const size_t n = (size_t)g.n[0] * g.n[1] * g.n[2];
  ReinitAxes<T> ax;
  for (int d = 0; d < 3; ++d) {
    ax.h[d] = (T)g.h[d];
    ax.ih[d] = (T)g.ih[d];
    ax.active[d] = g.n[d] > 1;
  }
  ax.cfl = (T)cfl;
  T* q0 = (T*)scratch;  // phi~, fixed for the whole iteration
  T* B = q0 + n;        // first-stage result
  T* A = B + n;         // iterate (float32 path; the float64 path iterates in phi)
  // the per-cell code of phi~ after the three arrays (scratch: 3 n doubles;
  // the float64 path uses the third array's space, which it does not need)
  unsigned char* code = sizeof(T) == sizeof(double) ? (unsigned char*)A : (unsigned char*)(A + n);
  // then the list of cells next to the interface: its length, two ints in, n places
  int* list = (int*)(code + (n + 7) / 8 * 8);
  const bool pairs = use_pairs<T>(g);
  if (pairs) cudaMemsetAsync(list, 0, 2 * sizeof(int), st);
  const int blocks = std::max((int)std::min<size_t>((n + 255) / 256, 152 * 16), 1);
  if constexpr (sizeof(T) == sizeof(double)) {
    cudaMemcpyAsync(q0, phi, n * sizeof(double), cudaMemcpyDeviceToDevice, st);
  } else {
    { k_to_f32<<<blocks, 256, 0, st>>>(phi, (float*)q0, n); WSI_COUNT(); }
  }
  { k_reinit_code<T><<<blocks, 256, 0, st>>>(g, q0, code, pairs ? list + 2 : nullptr, list); WSI_COUNT(); }
  const T* cur = q0;
  for (int m = 0; m < iters; ++m) {
    stage<T>(g, ax, pairs, code, list, q0, cur, nullptr, B, nullptr, st);
    if constexpr (sizeof(T) == sizeof(double)) {
      stage<T>(g, ax, pairs, code, list, q0, B, cur, (T*)phi, nullptr, st);
      cur = (const T*)phi;
    } else if (m + 1 == iters) {
      stage<T>(g, ax, pairs, code, list, q0, B, cur, nullptr, phi, st);
    } else {
      stage<T>(g, ax, pairs, code, list, q0, B, cur, A, nullptr, st);
      cur = A;
    }
  }
}
template void reinit_levelset<double>(const GridDev&, double*, int, double, void*, cudaStream_t);
template void reinit_levelset<float>(const GridDev&, double*, int, double, void*, cudaStream_t);

}  // namespace wsi
