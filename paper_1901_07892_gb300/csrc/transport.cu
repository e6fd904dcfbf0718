// Consistent mass/momentum transport (Sec. 4.2.2) and level-set advection
// (Sec. 4.2.1), with the bounded cubic-upwind (CUI) limiter.
//
// Transport of the C-face density (and, for the convective term, of the C
// momentum) is a divergence over face-centred control volumes.  Each flux
// through a control-volume face is shared by the two C-faces on either side
// of it, so the kernel computes it once: a 32 x 8 block owns a tile of
// C-faces in (x, y) and marches up a chunk of z-planes; x-fluxes go to the next
// lane by shuffle and y-fluxes through shared memory (those through the tile's
// lower edges come from a ninth warp), the z-flux of the plane below is kept in a
// register.  The
// limiter's inputs are staged per plane in shared memory (see k_transport).
//
// Storage and arithmetic type T: float64 on the plain path; float32 on the
// mixed path, where the step keeps float32 shadow copies of the transported
// fields (an explicit stencil apply; reading float32 avoids a float64->float32
// conversion per load, which issues on GB300's narrow float64 pipe).
#include <math.h>

#include <algorithm>

#include "df.cuh"
#include "internal.h"

namespace wsi {

static constexpr int BX = 32, BY = 8;

// Division-free bounded CUI: with num = qC - qU and den = qD - qU,
// t = num/den lies in a branch interval iff num*sign(den) lies in den-scaled
// bounds, and qU + t_f den = qU + {3 num, 5 num/6 + den/3, den, num}.  The
// bounds 2/13 and 4/5 are tested as 6.5 a <= D and 1.25 a <= D (powers of two
// of 13 a <= 2 D and 5 a <= 4 D: the same roundings, two products less); none
// holds for NaN, which takes the last case.
// Without branches: neighbouring cells take different cases.  up: the flow is
// in the positive direction; there the steep case rounds once, against it the
// product by itself (float32 results are kept to the bit, whichever way the
// cases are told apart).
__device__ __forceinline__ float cui(float qU, float qC, float qD, bool up) {
  const float den = qD - qU, num = qC - qU;
  // num * sign(den), so that t = a / |den| (den = 0 is told apart below)
  const float a = __int_as_float(__float_as_int(num) ^ (__float_as_int(den) & 0x80000000)), D = fabsf(den);
  const bool p = a > 0.0f, c1 = p && 6.5f * a <= D, c2 = p && 1.25f * a <= D, c3 = p && a <= D;
  const float f = c1 ? 3.0f * num : (c2 ? num * (float)(5.0 / 6.0) + den * (float)(1.0 / 3.0) : (c3 ? den : num));
  const float q = c1 && up ? fmaf(3.0f, num, qU) : qU + f;
  return den == 0.0f ? qC : q;
}
// the cases written out, for differences that are subnormal, infinite or NaN
__device__ __forceinline__ double cui_cases(double qU, double num, double den) {
  const double a = den > 0.0 ? num : -num, D = fabs(den);
  if (a > 0.0 && 6.5 * a <= D) return qU + 3.0 * num;
  if (6.5 * a > D && 1.25 * a <= D) return qU + (num * (5.0 / 6.0) + den * (1.0 / 3.0));
  return qU + (1.25 * a > D && a <= D ? den : num);
}
// float64: the comparisons are made on the bit patterns (as signed integers a
// value of either sign orders correctly against a positive one, as unsigned ones a
// NaN of either sign lies above it), and the cases differ in two factors: seven
// operations on the narrow pipe.  A factor 0 makes a NaN of an infinite den, so
// that goes with the other special ones through a branch, which where the field is
// uniform skips the rest as well (transport of 128^3, 16 launches: 3310 us with a
// test of each by itself in the common path, which let infinities through; 3010).
__device__ __forceinline__ double cui(double qU, double qC, double qD, bool) {
  typedef unsigned long long ull;
  const double den = qD - qU, num = qC - qU;
  const long long TOP = (long long)0x8000000000000000ull;
  const long long bd = __double_as_longlong(den), bn = __double_as_longlong(num);
  if (((unsigned)(bd >> 32) & 0x7FF00000u) - 1u >= 0x7FEFFFFFu) {  // zero, subnormal, infinite or NaN
    if ((bd & ~TOP) == 0) return qC;
    return cui_cases(qU, num, den);
  }
  const bool pos = bd > 0;
  const long long D = pos ? bd : bd ^ TOP;
  const double a = __longlong_as_double(pos ? bn : bn ^ TOP);
  const long long i0 = pos ? bn : bn ^ TOP, i1 = __double_as_longlong(6.5 * a), i2 = __double_as_longlong(1.25 * a);
  const bool c1 = i0 > 0 && i1 <= D, c2 = i1 > D && (ull)i2 <= (ull)D, c3 = i2 > D && (ull)i0 <= (ull)D;
  const double A = c1 ? 3.0 : (c2 ? 5.0 / 6.0 : (c3 ? 0.0 : 1.0));
  const double B = c2 ? 1.0 / 3.0 : (c3 ? 1.0 : 0.0);
  return qU + fma(A, num, B * den);
}

// Entry m of the C-face array along axis D extended by two ghost layers: the
// stored index it maps to and the velocity ghost sign.  Density ghosts are
// even mirrors; velocity ghosts are odd about wall faces when C == D (the wall
// face itself is zero; even about an open top, where dw/dz = 0) and take the
// wall's tangential sign across D != C.
template <int C, int D, typename T>
__device__ __forceinline__ int mirror_index(const GridDev& g, int m, T& s) {
  const int n = g.n[D] + (C == D ? 1 : 0);
  int mm = m;
  s = T(1);
  if (m < 0) {
    const int gl = -m;
    if (C == D) {
      mm = gl;
      s = T(-1);
    } else {
      mm = gl - 1;
      s = gbc<T>(g, 2 * D);
    }
  } else if (m >= n) {
    const int gl = m - (n - 1);
    if (C == D) {
      mm = (n - 1) - gl;
      s = (D == 2 && g.open_top) ? T(1) : T(-1);
    } else {
      mm = n - gl;
      s = gbc<T>(g, 2 * D + 1);
    }
  }
  return clampi(mm, 0, n - 1);
}

// limited value from the four taps for advective velocity adv
template <typename T>
__device__ __forceinline__ T lim4(T t0, T t1, T t2, T t3, T adv) {
  const bool pos = adv > T(0);
  return cui(pos ? t0 : t3, pos ? t1 : t2, pos ? t2 : t1, pos);
}

// advective velocity at the D-direction CV face at position m of the C-face
// column through (i, j, k): C == D: mean of C-faces m and m+1; else mean of
// the two D-faces at D-index m adjacent along C
template <int C, int D, typename T>
__device__ __forceinline__ T adv_at(const GridDev& g, const CVel<T>& vel, int i, int j, int k, int m) {
  int a[3] = {i, j, k};
  a[D] = m;
  if (C == D) {
    const size_t id = fidx(g, C, a[0], a[1], a[2]);
    const size_t st = C == 0 ? 1 : (C == 1 ? (size_t)g.n[0] : (size_t)g.n[0] * g.n[1]);
    return T(0.5) * (vel.q[C][id] + vel.q[C][id + st]);
  }
  const size_t id1 = fidx(g, D, a[0], a[1], a[2]);
  const size_t sc = C == 0 ? 1 : (C == 1 ? (size_t)(g.n[0] + (D == 0)) : (size_t)(g.n[0] + (D == 0)) * (g.n[1] + (D == 1)));
  return T(0.5) * (vel.q[D][id1 - sc] + vel.q[D][id1]);
}

// Asynchronous 4- or 8-byte copies global -> shared (cp.async), grouped per
// staged plane
template <typename T>
__device__ __forceinline__ void cpa(T* dst, const T* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// What a launch does with the divergence R of the mass flux of rho, and that of
// the momentum flux:
// TR_STAGE  out = a base + b rho + c R (base null: rho + c R), a Runge-Kutta
//           stage of the density in T
// TR_CONV   conv = the momentum flux' divergence alone
// TR_LAST   both, with the velocity's limiter on the same mass flux: the last
//           stage in float64 (rho64 = a64 base64 + b64 rho + c64 R, beta64 its
//           reciprocal) and conv
enum { TR_STAGE, TR_CONV, TR_LAST };
template <typename T>
struct TransportOut {
  const T* base;
  T a, b, c;
  T* out;
  const double* base64;
  double a64, b64, c64;
  double *rho64, *beta64;
  T* conv;
};

// a x + b y + c z and y + c z with the roundings of the elementwise sums in
// float32 (the first product is the one that is fused) and float64 (the last)
__device__ __forceinline__ float stage_sum(float a, float x, float b, float y, float c, float z) {
  return fmaf(c, z, fmaf(a, x, __fmul_rn(b, y)));
}
__device__ __forceinline__ double stage_sum(double a, double x, double b, double y, double c, double z) {
  return fma(c, z, fma(b, y, a * x));
}
__device__ __forceinline__ float stage_sum(float y, float c, float z) { return __fadd_rn(y, __fmul_rn(c, z)); }
__device__ __forceinline__ double stage_sum(double y, double c, double z) { return fma(c, z, y); }

__device__ __forceinline__ double stage64(double a, double x, double b, float y, double c, float z) {
  return a * x + b * f2d_fast(y) + c * f2d_fast(z);
}
__device__ __forceinline__ double stage64(double a, double x, double b, double y, double c, double z) {
  return fma(c, z, fma(b, y, a * x));
}

// A block advances a tile of 32 x 8 faces up a z-chunk.  Per plane the tile of
// the transported field (and, for the convective term, of the velocity
// component) with a two-entry halo in x and y is in a ring of NPL plane slots in
// shared memory, filled by asynchronous copies up to NPL planes ahead (ghosts
// beyond walls are mirrored through the copies' source addresses; the velocity
// ghosts' signs, and the inlet data across a Dirichlet inlet, are applied by the
// thread that copied them once the copies have landed).  Every flux is formed
// once: a thread forms the three through the upper faces of its entry, a ninth
// warp those through the tile's lower x and y edges; the lower x-flux comes by
// shuffle, the lower y-flux through shared memory, the lower z-flux is the one of
// the plane before, as the z taps are carried in registers.  The raw advective
// velocities are loaded one plane ahead.  One barrier per plane: it publishes
// the edge and y-fluxes of plane k and the staged plane k + 3.  Faces of the last
// column (C = 0) or row (C = 1) lie on a wall, where R = 0: where they would
// start a tile of their own their neighbours' threads write them.
// Bound by instruction issue (82 % of the slots at 256 x 256 x 64, the limiters'
// compares and selects a third of the instructions).  At 256^3 in float32 a stage
// takes 166 us per component with its sum, the last stage 345 us with the
// momentum flux, its sum and the reciprocal.  One launch per flux kind, edges by
// the first lane and row and two branches per limiter took 240-274 and 400 us,
// formed the last stage's mass flux twice, and the sums took 26, 106 and 50 us
// more.  In float64 (128 x 64 x 64): 76 and 151 us, before 217 and 456.
static constexpr int TNT = BX * (BY + 1);

// inl (C == 2 with the velocity only, else null): tangential data of w on
// the x- plane of a Dirichlet inlet, (nz+1) x ny; the ghosts of w across it
// are then 2 inl - (mirror image)
template <int C, int MODE, typename T>
__global__ void __launch_bounds__(TNT, sizeof(T) == 4 ? (MODE == TR_STAGE ? 4 : 3) : 2)
    k_transport(GridDev g, CVel<T> vel, const T* __restrict__ rho, TransportOut<T> o, int zchunk,
                const T* __restrict__ inl) {
  constexpr bool V = MODE != TR_STAGE;
  constexpr int NF = MODE == TR_LAST ? 2 : 1;   // fluxes handed on: mass, momentum
  constexpr int NPL = sizeof(T) == 4 ? 8 : 4;   // ring slots
  constexpr int HX = BX + 4, HY = BY + 4, PL = HX * HY, NS = (PL + TNT - 1) / TNT;
  __shared__ __align__(16) T sR[NPL][PL];
  __shared__ __align__(16) T sQ[V ? NPL : 1][V ? PL : 1];
  __shared__ T sFy[2][NF][BY + 1][BX];
  __shared__ T sXe[2][NF][BY];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * BX + tx;
  const bool edge = ty == BY;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
  const int i = x0 + tx, j = y0 + ty;
  const int e0 = ext(g, C, 0), e1 = ext(g, C, 1), e2 = ext(g, C, 2);
  const bool inside = !edge && i < e0 && j < e1;
  const int k0 = blockIdx.z * zchunk;
  const int k1 = min(k0 + zchunk, e2);
  const size_t plane = (size_t)e0 * e1;
  const T* __restrict__ qc = vel.q[C];
  // staged entries of this thread: in-plane offset (mirrored) and velocity sign
  int soff[NS];
  T ssg[NS];
  constexpr bool INL = C == 2 && V;
  int sinl[INL ? NS : 1];  // inlet data row of an x-ghost entry, else -1
#pragma unroll
  for (int r = 0; r < NS; ++r) {
    const int t = tid + r * TNT;
    soff[r] = -1;
    ssg[r] = T(1);
    if (INL) sinl[r] = -1;
    if (t < PL) {
      const int hy = t / HX, hx = t - hy * HX;
      T sx, sy;
      const int mx = mirror_index<C, 0, T>(g, x0 - 2 + hx, sx);
      const int my = mirror_index<C, 1, T>(g, y0 - 2 + hy, sy);
      soff[r] = my * e0 + mx;
      ssg[r] = sx * sy;
      if (INL && inl && x0 - 2 + hx < 0) sinl[r] = my;
    }
  }
  // copies of plane p (k0 <= p; above the array its mirror image) into its slot;
  // one group per call
  auto issue = [&](int p) {
    if (p <= k1 + 1) {
      const int s = (p - k0) & (NPL - 1);
      T sz;
      const size_t pz = (size_t)mirror_index<C, 2, T>(g, p, sz) * plane;
#pragma unroll
      for (int r = 0; r < NS; ++r) {
        const int t = tid + r * TNT;
        if (soff[r] >= 0) {
          cpa<T>(&sR[s][t], rho + pz + soff[r]);
          if (V) cpa<T>(&sQ[V ? s : 0][V ? t : 0], qc + pz + soff[r]);
        }
      }
    }
    cpa_commit();
  };
  // signs and inlet data of this thread's entries of plane p, once landed
  // (planes above the array: only their inner columns are read)
  auto fix = [&](int p) {
    if (!V || p >= e2 || p > k1 + 1) return;
    const int s = (p - k0) & (NPL - 1);
#pragma unroll
    for (int r = 0; r < NS; ++r) {
      const int t = tid + r * TNT;
      if (soff[r] < 0) continue;
      const bool inl_here = INL && sinl[INL ? r : 0] >= 0;
      if (ssg[r] == T(1) && !inl_here) continue;
      T q = ssg[r] * sQ[V ? s : 0][V ? t : 0];
      if (inl_here) q += T(2) * inl[(size_t)p * e1 + sinl[INL ? r : 0]];
      sQ[V ? s : 0][V ? t : 0] = q;
    }
  };
  // The entries whose upper x- and y-fluxes this thread forms: its own, in the
  // ninth warp those below the tile's edges; whether there is a flux at all (not
  // through a wall, nor for a face on a wall), and where its two advective
  // velocities are: offsets at level k0 that move by one level of their array
  // per plane (32-bit: every array holds fewer than 2^31 entries)
  const int xi = edge ? x0 - 1 : i, xj = edge ? y0 + (tx & (BY - 1)) : j, yj = edge ? y0 - 1 : j;
  const int mx = xi + (C == 0 ? 0 : 1), my = yj + (C == 1 ? 0 : 1);
  const bool wi = i == 0 || i == n0, wj = j == 0 || j == n1;
  const bool fx = (edge ? tx < BY : i < e0) && xj < e1 && (C != 0 || (mx >= 0 && mx < n0)) &&
                  (C != 1 || (xj != 0 && xj != n1));
  const bool fy = i < e0 && yj < e1 && (C != 1 || (my >= 0 && my < n1)) && (C != 0 || !wi);
  const bool fz = inside && (C != 0 || !wi) && (C != 1 || !wj);
  const int lx = (n0 + 1) * n1, ly = n0 * (n1 + 1), lz = n0 * n1;  // one z-level of u, v, w
  const int dx = C == 0 ? 1 : (C == 1 ? -(n0 + 1) : -lx);
  const int dy = C == 1 ? n0 : (C == 0 ? -1 : -ly);
  const int dz = C == 2 ? lz : (C == 0 ? -1 : -n0);
  int ax = fx ? (int)fidx(g, 0, mx, xj, k0) : 0;
  int ay = fy ? (int)fidx(g, 1, i, my, k0) : 0;
  int az = fz ? (int)fidx(g, 2, i, j, k0 + (C == 2 ? 0 : 1)) : 0;
  const T* __restrict__ U_ = vel.q[0];
  const T* __restrict__ V_ = vel.q[1];
  const T* __restrict__ W_ = vel.q[2];
  T u0 = T(0), u1 = T(0), v0 = T(0), v1 = T(0), w0 = T(0), w1 = T(0);
  auto load = [&](int k) {  // of plane k; called for consecutive planes
    const bool kw = C == 2 && (k == 0 || k == n2);
    u0 = u1 = v0 = v1 = w0 = w1 = T(0);
    if (fx && !kw) {
      u0 = U_[ax];
      u1 = U_[ax + dx];
    }
    if (fy && !kw) {
      v0 = V_[ay];
      v1 = V_[ay + dy];
    }
    if (fz && (C != 2 || k < n2)) {
      w0 = W_[az];
      w1 = W_[az + dz];
    }
    ax += lx;
    ay += ly;
    az += lz;
  };
  const int own = (ty + 2) * HX + tx + 2;
  const int ox = edge ? ((tx & (BY - 1)) + 2) * HX + 1 : own;
  const int oy = edge ? HX + tx + 2 : own;

#pragma unroll 1
  for (int p = k0; p < k0 + NPL; ++p) issue(p);
  load(k0);
  // own column: planes k0 - 2 and k0 - 1 from memory
  const size_t col = (size_t)min(j, e1 - 1) * e0 + min(i, e0 - 1);
  T ra, rm, qa = T(0), qm = T(0);
  {
    T sa, sm;
    const size_t pa = (size_t)mirror_index<C, 2, T>(g, k0 - 2, sa) * plane + col;
    const size_t pm = (size_t)mirror_index<C, 2, T>(g, k0 - 1, sm) * plane + col;
    ra = rho[pa];
    rm = rho[pm];
    if (V) {
      qa = sa * qc[pa];
      qm = sm * qc[pm];
    }
  }
  cpa_wait<NPL - 3>();  // planes k0 .. k0 + 2
#pragma unroll 1
  for (int p = k0; p <= k0 + 2; ++p) fix(p);
  __syncthreads();
  T rc = sR[0][own], rp = sR[1][own], qo = T(0), qp = T(0);
  if (V) {
    T sp;
    mirror_index<C, 2, T>(g, k0 + 1, sp);
    qo = sQ[0][V ? own : 0];
    qp = sp * sQ[V ? 1 : 0][V ? own : 0];
  }
  T zlo[2] = {T(0), T(0)};
  if (fz && (C != 2 || k0 > 0)) {
    const T adv = adv_at<C, 2, T>(g, vel, i, j, k0, C == 2 ? k0 - 1 : k0);
    if (adv != T(0)) {
      zlo[0] = adv * lim4<T>(ra, rm, rc, rp, adv);
      if (V) zlo[1] = zlo[0] * lim4<T>(qa, qm, qo, qp, adv);
    }
  }
  size_t id = (size_t)k0 * plane + (size_t)j * e0 + i;
  // face through the last column or row, next to this one
  const bool twin = inside && ((C == 0 && tx == BX - 1 && i == n0 - 1) || (C == 1 && ty == BY - 1 && j == n1 - 1));
  auto emit = [&](size_t at, T self, T R, T M, T base, double base64) {
    if (MODE == TR_STAGE) {
      o.out[at] = o.base ? stage_sum(o.a, base, o.b, self, o.c, R) : stage_sum(self, o.c, R);
    } else if (MODE == TR_LAST) {
      const double v = stage64(o.a64, base64, o.b64, self, o.c64, R);
      o.rho64[at] = v;
      o.beta64[at] = recip_df(v);
    }
    if (V) o.conv[at] = M;
  };
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const T axv = T(0.5) * (u0 + u1), ayv = T(0.5) * (v0 + v1), azv = T(0.5) * (w0 + w1);
    if (k + 1 < k1) load(k + 1);
    T base = T(0);
    double base64 = 0.0;
    if (MODE == TR_STAGE && o.base && inside) base = o.base[id];
    if (MODE == TR_LAST && inside) base64 = o.base64[id];
    const int s = (k - k0) & (NPL - 1), s2 = (k + 2 - k0) & (NPL - 1), par = k & 1;
    const T* R_ = sR[s];
    const T* Q_ = sQ[V ? s : 0];
    const T rq = sR[s2][own];
    T qq = T(0);
    if (V) {
      T sz;
      mirror_index<C, 2, T>(g, k + 2, sz);
      qq = sz * sQ[V ? s2 : 0][V ? own : 0];
    }
    // fluxes: [0] mass, [1] momentum
    T xf[2], yf[2], zf[2];
    xf[0] = axv * lim4<T>(R_[ox - 1], R_[ox], R_[ox + 1], R_[ox + 2], axv);
    yf[0] = ayv * lim4<T>(R_[oy - HX], R_[oy], R_[oy + HX], R_[oy + 2 * HX], ayv);
    zf[0] = azv * lim4<T>(rm, rc, rp, rq, azv);
    if (axv == T(0)) xf[0] = T(0);
    if (ayv == T(0)) yf[0] = T(0);
    if (azv == T(0)) zf[0] = T(0);
    xf[1] = yf[1] = zf[1] = T(0);
    if (V) {
      if (axv != T(0)) xf[1] = xf[0] * lim4<T>(Q_[ox - 1], Q_[ox], Q_[ox + 1], Q_[ox + 2], axv);
      if (ayv != T(0)) yf[1] = yf[0] * lim4<T>(Q_[oy - HX], Q_[oy], Q_[oy + HX], Q_[oy + 2 * HX], ayv);
      if (azv != T(0)) zf[1] = zf[0] * lim4<T>(qm, qo, qp, qq, azv);
    }
    constexpr int F0 = MODE == TR_CONV ? 1 : 0;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      sFy[par][f][edge ? 0 : ty + 1][tx] = yf[F0 + f];
      if (edge && tx < BY) sXe[par][f][tx] = xf[F0 + f];
    }
    cpa_wait<NPL - 4>();  // planes up to k + 3 have landed (this thread's copies)
    fix(k + 3);
    __syncthreads();
    T res[2] = {T(0), T(0)};
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      T xl = __shfl_up_sync(0xffffffffu, xf[F0 + f], 1);
      if (tx == 0) xl = sXe[par][f][edge ? 0 : ty];
      const T yl = sFy[par][f][edge ? 0 : ty][tx];
      res[F0 + f] = (xf[F0 + f] - xl) * ginv<T>(g, 0) + (yf[F0 + f] - yl) * ginv<T>(g, 1) +
                    (zf[F0 + f] - zlo[F0 + f]) * ginv<T>(g, 2);
      zlo[F0 + f] = zf[F0 + f];
    }
    if (C == 0 ? wi : (C == 1 ? wj : (k == 0 || k == n2))) res[0] = res[1] = T(0);
    if (inside) emit(id, rc, res[0], res[1], base, base64);
    if (twin) {
      const size_t at = id + (C == 0 ? 1 : e0);
      emit(at, rho[at], T(0), T(0), MODE == TR_STAGE && o.base ? o.base[at] : T(0),
           MODE == TR_LAST ? o.base64[at] : 0.0);
    }
    issue(k + NPL);  // into plane k's slot
    rm = rc;
    rc = rp;
    rp = rq;
    if (V) {
      qm = qo;
      qo = qp;
      qp = qq;
    }
    id += plane;
  }
  cpa_wait<0>();  // no copies in flight when the block ends
}

// z-chunk of the transport kernels: long marches amortise the chunk start,
// but the grid must still fill the GPU (about 8 blocks per SM)
int transport_chunk(int ex, int ey, int ez) {
  const long long base = (long long)cdiv(ex, BX) * cdiv(ey, BY);
  int c = 32;
  while (c > 4 && base * cdiv(ez, c) < 152LL * 8) c /= 2;
  return c;
}

template <int C, int MODE, typename T>
static void transport_one(const GridDev& g, const CVel<T>& v, const T* rho, const TransportOut<T>& o, const T* inl,
                          cudaStream_t st) {
  // (the last column or row, see k_transport, gets no tile of its own)
  const int ex = C == 0 && g.n[0] % BX == 0 ? g.n[0] : ext(g, C, 0);
  const int ey = C == 1 && g.n[1] % BY == 0 ? g.n[1] : ext(g, C, 1);
  const int ez = ext(g, C, 2), zc = transport_chunk(ex, ey, ez);
  { k_transport<C, MODE, T><<<dim3(cdiv(ex, BX), cdiv(ey, BY), cdiv(ez, zc)), dim3(BX, BY + 1), 0, st>>>(g, v, rho, o, zc,
                                                                                                       inl); WSI_COUNT(); }
}

template <int MODE, typename T>
static void transport_all(const GridDev& g, const T* const vel[3], const T* const rho[3], const TransportOut<T> o[3],
                          const T* inlet_w, cudaStream_t st) {
  CVel<T> v{{vel[0], vel[1], vel[2]}};
  ktimer_begin(KC_TRANSPORT, st);
  {
    // algorithmic bytes: per component rho_C, u, v, w (advective velocities),
    // q_C and the result with the momentum flux; the stage's other input and
    // its results
    const double F = (double)(fsize(g, 0) + fsize(g, 1) + fsize(g, 2));
    const double b = sizeof(T) * (MODE == TR_STAGE ? (o[0].base ? 6.0 : 5.0) : 6.0) + (MODE == TR_LAST ? 24.0 : 0.0);
    ktimer_bytes(KC_TRANSPORT, F * b);
  }
  transport_one<0, MODE, T>(g, v, rho[0], o[0], nullptr, st);
  transport_one<1, MODE, T>(g, v, rho[1], o[1], nullptr, st);
  transport_one<2, MODE, T>(g, v, rho[2], o[2], inlet_w, st);
  ktimer_end(KC_TRANSPORT, st);
}

template <typename T>
void launch_transport_stage(const GridDev& g, const T* const vel[3], const T* const rho[3], double a,
                            const T* const base[3], double b, double c, T* const out[3], cudaStream_t st) {
  TransportOut<T> o[3] = {};
  for (int d = 0; d < 3; ++d) {
    o[d].base = base ? base[d] : nullptr;
    o[d].a = (T)a;
    o[d].b = (T)b;
    o[d].c = (T)c;
    o[d].out = out[d];
  }
  transport_all<TR_STAGE, T>(g, vel, rho, o, nullptr, st);
}

template <typename T>
void launch_transport_last(const GridDev& g, const T* const vel[3], const T* const rho[3], double a,
                           const double* const base[3], double b, double c, double* const rho_out[3],
                           double* const beta_out[3], T* const conv[3], cudaStream_t st, const T* inlet_w) {
  TransportOut<T> o[3] = {};
  for (int d = 0; d < 3; ++d) {
    o[d].base64 = base[d];
    o[d].a64 = a;
    o[d].b64 = b;
    o[d].c64 = c;
    o[d].rho64 = rho_out[d];
    o[d].beta64 = beta_out[d];
    o[d].conv = conv[d];
  }
  transport_all<TR_LAST, T>(g, vel, rho, o, inlet_w, st);
}

template <typename T>
void launch_transport_conv(const GridDev& g, const T* const vel[3], const T* const rho[3], T* const conv[3],
                           cudaStream_t st, const T* inlet_w) {
  TransportOut<T> o[3] = {};
  for (int d = 0; d < 3; ++d) o[d].conv = conv[d];
  transport_all<TR_CONV, T>(g, vel, rho, o, inlet_w, st);
}
#define INST_TRANSPORT(T)                                                                                              \
  template void launch_transport_stage<T>(const GridDev&, const T* const[3], const T* const[3], double,                \
                                          const T* const[3], double, double, T* const[3], cudaStream_t);               \
  template void launch_transport_last<T>(const GridDev&, const T* const[3], const T* const[3], double,                 \
                                         const double* const[3], double, double, double* const[3], double* const[3],   \
                                         T* const[3], cudaStream_t, const T*);                                         \
  template void launch_transport_conv<T>(const GridDev&, const T* const[3], const T* const[3], T* const[3],            \
                                         cudaStream_t, const T*);
INST_TRANSPORT(double)
INST_TRANSPORT(float)
#undef INST_TRANSPORT

template <typename Ti, typename To>
__global__ void k_lincomb(size_t n, double a, const Ti* __restrict__ x, double b, const Ti* __restrict__ y, double c,
                          const Ti* __restrict__ z, To* out) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  // coefficients of +-1 and 0 skip their multiplication (float64 operations
  // are scarce); the common forms are x - y and x + c z
  const bool a1 = a == 1.0, b1 = b == 1.0, bm1 = b == -1.0, c1 = c == 1.0, cm1 = c == -1.0;
  for (; t < n; t += stride) {
    double s = a1 ? (double)x[t] : a * (double)x[t];
    if (y) s = b1 ? s + (double)y[t] : (bm1 ? s - (double)y[t] : fma(b, (double)y[t], s));
    if (z) s = c1 ? s + (double)z[t] : (cm1 ? s - (double)z[t] : fma(c, (double)z[t], s));
    out[t] = (To)s;
  }
}

// float64 inputs, float32 arithmetic and output: the inputs are rounded by
// integer operations (d2f_fast), keeping the float64 pipe idle
__global__ void k_lincomb_tof(size_t n, float a, const double* __restrict__ x, float b, const double* __restrict__ y,
                              float c, const double* __restrict__ z, float* out) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (; t < n; t += stride) {
    float s = a * d2f_fast(x[t]);
    if (y) s += b * d2f_fast(y[t]);
    if (z) s += c * d2f_fast(z[t]);
    out[t] = s;
  }
}

// the two SSP-RK3 stage velocities of Sec. 4.2.2 in float32 from one pass over
// u^n, u^{n-1} (and u^{n+1,k} in later cycles), and optionally the float32
// copy of u^n; the same arithmetic as k_lincomb_tof for each output
__global__ void k_rk_vel_tof(size_t n, const double* __restrict__ un, const double* __restrict__ unm1,
                             const double* __restrict__ uk, float* u1, float* u2, float* un32) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    const float a = d2f_fast(un[t]), b = d2f_fast(unm1[t]);
    if (uk) {
      const float q = d2f_fast(uk[t]);
      u1[t] = 1.0f * q;
      u2[t] = 0.375f * q + 0.75f * a + -0.125f * b;
    } else {
      u1[t] = 2.0f * a + -1.0f * b;
      u2[t] = 1.5f * a + -0.5f * b;
    }
    if (un32) un32[t] = 1.0f * a;
  }
}

// same in float32 arithmetic (float32 inputs and outputs)
__global__ void k_lincomb_f(size_t n, float a, const float* __restrict__ x, float b, const float* __restrict__ y,
                            float c, const float* __restrict__ z, float* out) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (; t < n; t += stride) {
    float s = a * x[t];
    if (y) s += b * y[t];
    if (z) s += c * z[t];
    out[t] = s;
  }
}

static int lc_blocks(size_t n) {
  int blocks = (int)std::min<size_t>((n + 255) / 256, 152 * 16);
  return blocks < 1 ? 1 : blocks;
}

void launch_rk_velocities_f32(size_t n, const double* un, const double* unm1, const double* uk, float* u1, float* u2,
                              float* un32, cudaStream_t st) {
  { k_rk_vel_tof<<<lc_blocks(n), 256, 0, st>>>(n, un, unm1, uk, u1, u2, un32); WSI_COUNT(); }
}

void launch_lincomb(size_t n, double a, const double* x, double b, const double* y, double c, const double* z,
                    double* out, cudaStream_t st) {
  { k_lincomb<double, double><<<lc_blocks(n), 256, 0, st>>>(n, a, x, b, y, c, z, out); WSI_COUNT(); }
}
void launch_lincomb_to_f32(size_t n, double a, const double* x, double b, const double* y, double c,
                           const double* z, float* out, cudaStream_t st) {
  { k_lincomb_tof<<<lc_blocks(n), 256, 0, st>>>(n, (float)a, x, (float)b, y, (float)c, z, out); WSI_COUNT(); }
}
void launch_lincomb_f32(size_t n, float a, const float* x, float b, const float* y, float c, const float* z,
                        float* out, cudaStream_t st) {
  { k_lincomb_f<<<lc_blocks(n), 256, 0, st>>>(n, a, x, b, y, c, z, out); WSI_COUNT(); }
}
// out = a*x64 + b*y32 + c*z32 in float64
__global__ void k_lincomb_mix(size_t n, double a, const double* __restrict__ x, double b, const float* __restrict__ y,
                              double c, const float* __restrict__ z, double* out) {
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (; t < n; t += stride) out[t] = a * x[t] + b * f2d_fast(y[t]) + c * f2d_fast(z[t]);
}
void launch_lincomb_mix(size_t n, double a, const double* x, double b, const float* y, double c, const float* z,
                        double* out, cudaStream_t st) {
  { k_lincomb_mix<<<lc_blocks(n), 256, 0, st>>>(n, a, x, b, y, c, z, out); WSI_COUNT(); }
}

__global__ void k_widen(const float* __restrict__ x, size_t n, double* out) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    out[t] = f2d_fast(x[t]);
}
void launch_widen(const float* x, size_t n, double* out, cudaStream_t st) {
  { k_widen<<<lc_blocks(n), 256, 0, st>>>(x, n, out); WSI_COUNT(); }
}

// The mean is taken off in float32 pairs and the scale is a power of two, so
// the result carries one rounding and no float64 operation (1/64 of the
// float32 rate) is spent.
__global__ void k_shift_scale_f(size_t n, const double* __restrict__ x, dfl m, float f, float* y) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
    const dfl a = df_split(x[t]);
    float s, e;
    two_sum(a.h, -m.h, s, e);
    y[t] = f * (s + (e + (a.l - m.l)));
  }
}
void launch_shift_scale_f32(size_t n, const double* x, double m, int e, float* y, cudaStream_t st) {
  dfl d;
  d.h = (float)m;
  d.l = (float)(m - (double)d.h);
  { k_shift_scale_f<<<lc_blocks(n), 256, 0, st>>>(n, x, d, ldexpf(1.0f, -e), y); WSI_COUNT(); }
}
__global__ void k_axpy_f(size_t n, double a, const float* __restrict__ y, double* x) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    x[t] = fma(a, f2d_fast(y[t]), x[t]);
}
void launch_axpy_f32(size_t n, double a, const float* y, double* x, cudaStream_t st) {
  { k_axpy_f<<<lc_blocks(n), 256, 0, st>>>(n, a, y, x); WSI_COUNT(); }
}
__global__ void k_shift(size_t n, double* x, double m) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) x[t] -= m;
}
void launch_shift(size_t n, double* x, double m, cudaStream_t st) {
  { k_shift<<<lc_blocks(n), 256, 0, st>>>(n, x, m); WSI_COUNT(); }
}

// ================================================================ level set
// Same staging as k_transport: per z-plane the tile of phi^{n+1/2} with a
// halo of H cells (Neumann mirror ghosts applied while staging) in shared
// memory, the z taps in a 2H-entry register window, the face velocities
// loaded before the staging barrier.  H = 2 for the CUI limiter, 4 for
// xsPPM7 (seven-cell upwind-biased stencils).
template <typename T>
__device__ __forceinline__ int ls_mirror(int m, int n) {
  // repeated even reflection (grids thinner than the halo reflect again)
  for (int it = 0; it < 8; ++it) {
    if (m < 0) m = -m - 1;
    else if (m >= n) m = 2 * n - 1 - m;
  }
  return clampi(m, 0, n - 1);
}

template <typename T>
__device__ __forceinline__ T mm2(T a, T b) {
  return (a > T(0) && b > T(0)) ? fmin(a, b) : ((a < T(0) && b < T(0)) ? fmax(a, b) : T(0));
}
template <typename T>
__device__ __forceinline__ T mm4(T a, T b, T c, T d) {
  if (a > T(0) && b > T(0) && c > T(0) && d > T(0)) return fmin(fmin(a, b), fmin(c, d));
  if (a < T(0) && b < T(0) && c < T(0) && d < T(0)) return fmax(fmax(a, b), fmax(c, d));
  return T(0);
}

// xsPPM7 face value between q0 and p1 (cells ordered along the flow): the
// seventh-order upwind-biased interpolant, accepted when it lies between q0
// and the monotonicity-preserving value, otherwise moved into the
// curvature-widened bounds of Suresh and Huynh (alpha = 4)
template <typename T>
__device__ __forceinline__ T xsppm7_face(T m3, T m2, T m1, T q0, T p1, T p2, T p3) {
  const T u7 = (T(-3) * m3 + T(25) * m2 - T(101) * m1 + T(319) * q0 + T(214) * p1 - T(38) * p2 + T(4) * p3) *
               T(1.0 / 420.0);
  const T alpha = T(4);
  const T ump = q0 + mm2<T>(p1 - q0, alpha * (q0 - m1));
  if ((u7 - q0) * (u7 - ump) <= T(0)) return u7;
  const T dm1 = m2 - T(2) * m1 + q0, d0 = m1 - T(2) * q0 + p1, dp1 = q0 - T(2) * p1 + p2;
  const T dp = mm4<T>(T(4) * d0 - dp1, T(4) * dp1 - d0, d0, dp1);
  const T dm = mm4<T>(T(4) * dm1 - d0, T(4) * d0 - dm1, dm1, d0);
  const T uul = q0 + alpha * (q0 - m1);
  const T umd = T(0.5) * (q0 + p1) - T(0.5) * dp;
  const T ulc = q0 + T(0.5) * (q0 - m1) + T(4.0 / 3.0) * dm;
  const T umin = fmax(fmin(fmin(q0, p1), umd), fmin(fmin(q0, uul), ulc));
  const T umax = fmin(fmax(fmax(q0, p1), umd), fmax(fmax(q0, uul), ulc));
  return u7 + mm2<T>(umin - u7, umax - u7);
}

// upwind face value from the 2H cells around the face (c[H-1] | c[H])
template <typename T, int H>
struct LsLim;
template <typename T>
struct LsLim<T, 2> {
  static __device__ __forceinline__ T face(const T* c, T adv) { return lim4<T>(c[0], c[1], c[2], c[3], adv); }
};
template <typename T>
struct LsLim<T, 4> {
  static __device__ __forceinline__ T face(const T* c, T adv) {
    return adv > T(0) ? xsppm7_face<T>(c[0], c[1], c[2], c[3], c[4], c[5], c[6])
                      : xsppm7_face<T>(c[7], c[6], c[5], c[4], c[3], c[2], c[1]);
  }
};

template <typename T, int H>
__global__ void __launch_bounds__(BX* BY) k_ls_advect(GridDev g, CVel<T> vel,
                                                      const double* __restrict__ phi_n, const T* __restrict__ phi_h,
                                                      double dt, double* out, int zchunk) {
  constexpr int HX = BX + 2 * H, HY = BY + 2 * H, NS = (HX * HY + BX * BY - 1) / (BX * BY);
  __shared__ T sP[HY][HX];
  __shared__ T sFx[BY][BX + 1];
  __shared__ T sFy[BY + 1][BX];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * BX + tx;
  const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
  const int i = x0 + tx, j = y0 + ty;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const bool inside = i < n0 && j < n1;
  const int k0 = blockIdx.z * zchunk;
  const int k1 = min(k0 + zchunk, n2);
  const size_t plane = (size_t)n0 * n1;
  int soff[NS];
#pragma unroll
  for (int r = 0; r < NS; ++r) {
    const int t = tid + r * BX * BY;
    soff[r] = -1;
    if (t < HX * HY) {
      const int hy = t / HX, hx = t - hy * HX;
      soff[r] = ls_mirror<T>(y0 - H + hy, n1) * n0 + ls_mirror<T>(x0 - H + hx, n0);
    }
  }
  const size_t col = (size_t)min(j, n1 - 1) * n0 + min(i, n0 - 1);
  // z window: the 2H cells around the current bottom face (k - H .. k + H - 1)
  T zp[2 * H];
#pragma unroll
  for (int q = 0; q < 2 * H; ++q) zp[q] = phi_h[(size_t)ls_mirror<T>(k0 - H + q, n2) * plane + col];
  T Fz_lo = T(0);
  for (int k = k0; k < k1; ++k) {
    T ux = T(0), uxl = T(0), vy = T(0), vyl = T(0), wz = T(0), wzl = T(0);
    if (inside) {
      ux = vel.q[0][fidx(g, 0, i + 1, j, k)];
      if (tx == 0) uxl = vel.q[0][fidx(g, 0, i, j, k)];
      vy = vel.q[1][fidx(g, 1, i, j + 1, k)];
      if (ty == 0) vyl = vel.q[1][fidx(g, 1, i, j, k)];
      wz = vel.q[2][fidx(g, 2, i, j, k + 1)];
      if (k == k0) wzl = vel.q[2][fidx(g, 2, i, j, k)];
    }
#pragma unroll
    for (int r = 0; r < NS; ++r) {
      const int t = tid + r * BX * BY;
      if (soff[r] >= 0) {
        const int hy = t / HX, hx = t - hy * HX;
        sP[hy][hx] = phi_h[(size_t)k * plane + soff[r]];
      }
    }
    __syncthreads();
    if (inside) {
      const int hy = ty + H, hx = tx + H;
      T c[2 * H];
      // right x-face of cell i: cells i + 1 - H .. i + H
#pragma unroll
      for (int q = 0; q < 2 * H; ++q) c[q] = sP[hy][tx + 1 + q];
      sFx[ty][tx + 1] = ux * LsLim<T, H>::face(c, ux);
      if (tx == 0) {
#pragma unroll
        for (int q = 0; q < 2 * H; ++q) c[q] = sP[hy][tx + q];
        sFx[ty][0] = uxl * LsLim<T, H>::face(c, uxl);
      }
#pragma unroll
      for (int q = 0; q < 2 * H; ++q) c[q] = sP[ty + 1 + q][hx];
      sFy[ty + 1][tx] = vy * LsLim<T, H>::face(c, vy);
      if (ty == 0) {
#pragma unroll
        for (int q = 0; q < 2 * H; ++q) c[q] = sP[ty + q][hx];
        sFy[0][tx] = vyl * LsLim<T, H>::face(c, vyl);
      }
    }
    __syncthreads();
    if (k == k0) Fz_lo = wzl * LsLim<T, H>::face(zp, wzl);
#pragma unroll
    for (int q = 0; q < 2 * H - 1; ++q) zp[q] = zp[q + 1];
    zp[2 * H - 1] = phi_h[(size_t)ls_mirror<T>(k + H, n2) * plane + col];
    if (inside) {
      const T Fz_hi = wz * LsLim<T, H>::face(zp, wz);
      const T Q = (sFx[ty][tx + 1] - sFx[ty][tx]) * ginv<T>(g, 0) + (sFy[ty + 1][tx] - sFy[ty][tx]) * ginv<T>(g, 1) +
                  (Fz_hi - Fz_lo) * ginv<T>(g, 2);
      const size_t id = (size_t)k * plane + (size_t)j * n0 + i;
      out[id] = phi_n[id] - dt * cvt<double, T>(Q);
      Fz_lo = Fz_hi;
    }
    __syncthreads();
  }
}

template <typename T>
void launch_levelset_advect(const GridDev& g, const T* const vel[3], const double* phi_n, const T* phi_half, double dt,
                            double* out, cudaStream_t st, int limiter) {
  CVel<T> v{{vel[0], vel[1], vel[2]}};
  const int zc = transport_chunk(g.n[0], g.n[1], g.n[2]);
  dim3 grid(cdiv(g.n[0], BX), cdiv(g.n[1], BY), cdiv(g.n[2], zc));
  if (limiter == WSI_LIMIT_XSPPM7) {
    k_ls_advect<T, 4><<<grid, dim3(BX, BY), 0, st>>>(g, v, phi_n, phi_half, dt, out, zc);
  } else {
    k_ls_advect<T, 2><<<grid, dim3(BX, BY), 0, st>>>(g, v, phi_n, phi_half, dt, out, zc);
  }
  WSI_COUNT();
}
template void launch_levelset_advect<double>(const GridDev&, const double* const[3], const double*, const double*,
                                             double, double*, cudaStream_t, int);
template void launch_levelset_advect<float>(const GridDev&, const float* const[3], const double*, const float*,
                                            double, double*, cudaStream_t, int);

__global__ void k_box_sdf(GridDev g, const double* __restrict__ xc, double hx_, double hy_, double hz_, double* psi) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= g.n[0] || j >= g.n[1]) return;
  double x = (i + 0.5) * g.h[0], y = (j + 0.5) * g.h[1], z = (k + 0.5) * g.h[2];
  double qx = fabs(x - xc[0]) - hx_, qy = fabs(y - xc[1]) - hy_, qz = fabs(z - xc[2]) - hz_;
  double ox = fmax(qx, 0.0), oy = fmax(qy, 0.0), oz = fmax(qz, 0.0);
  double outside = sqrt(ox * ox + oy * oy + oz * oz);
  double inside = fmin(fmax(fmax(qx, qy), qz), 0.0);
  psi[fidx(g, 3, i, j, k)] = outside + inside;
}

// capped cylinder with its axis along y (radius r, half length hl) about xc
__global__ void k_cyl_sdf(GridDev g, const double* __restrict__ xc, double r, double hl, double* psi) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= g.n[0] || j >= g.n[1]) return;
  double x = (i + 0.5) * g.h[0], y = (j + 0.5) * g.h[1], z = (k + 0.5) * g.h[2];
  double dx = x - xc[0], dz = z - xc[2];
  double qr = sqrt(dx * dx + dz * dz) - r, qy = fabs(y - xc[1]) - hl;
  double or_ = fmax(qr, 0.0), oy = fmax(qy, 0.0);
  psi[fidx(g, 3, i, j, k)] = sqrt(or_ * or_ + oy * oy) + fmin(fmax(qr, qy), 0.0);
}

void launch_cyl_sdf(const GridDev& g, const double* xcom_dev, double radius, double half_length, double* psi,
                    cudaStream_t st) {
  { k_cyl_sdf<<<dim3(cdiv(g.n[0], BX), cdiv(g.n[1], BY), g.n[2]), dim3(BX, BY), 0, st>>>(g, xcom_dev, radius,
                                                                                          half_length, psi); WSI_COUNT(); }
}

void launch_box_sdf(const GridDev& g, const double* xcom_dev, const double half[3], double* psi, cudaStream_t st) {
  { k_box_sdf<<<dim3(cdiv(g.n[0], BX), cdiv(g.n[1], BY), g.n[2]), dim3(BX, BY), 0, st>>>(g, xcom_dev, half[0], half[1],
                                                                                         half[2], psi); WSI_COUNT(); }
}

}  // namespace wsi
