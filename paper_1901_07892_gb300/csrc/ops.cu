// Field kernels of libwsi: material coefficients (Sec. 4.1) and the staggered
// operators of the implicit Stokes system (Sec. 3.1, 4.2.2); transport and
// level-set advection live in transport.cu.
//
// Every kernel walks its output array in x-fastest order with one thread per
// entry (blocks of 32 x 8 in x, y; one z-plane per grid row), so warps read
// and write contiguous rows of the unghosted MAC arrays.
#include <math.h>

#include <algorithm>
#include <cmath>
#include <limits>

#include "internal.h"

namespace wsi {

static constexpr int BX = 32, BY = 8;

static inline dim3 grid3(int nx, int ny, int nz) { return dim3(cdiv(nx, BX), cdiv(ny, BY), nz); }

// =========================================================== materials
// Smoothed Heaviside of Sec. 2 with t = phi / eps: 0 for t <= -1, 1 for
// t >= 1, the sine ramp between.  The band test runs on a float32 copy of t
// made by integer operations (float64 comparisons issue on GB300's narrow
// float64 pipe); where that copy is ambiguous, |t| within 2^-24 of 1, the
// ramp differs from its limit by ~(1 - |t|)^3, far below float64 resolution.
// code: 0 or 1 away from the band (value exactly 0 or 1), 2 inside.
// Float32 pre-test: tf, a float32 estimate of t = phi/eps whose error is at
// most `bound` (a few units in the last float32 place of the magnitudes that
// formed it), decides the code without any float64 operation when it lies
// beyond the band edges by more than that bound; otherwise 2 (undecided:
// the float64 path runs).
__device__ __forceinline__ int band_code_f(float tf, float bound) {
  if (tf < -1.0f - bound) return 0;
  if (tf > 1.0f + bound) return 1;
  return 2;
}

// FUSED: 1 + phi/eps with one rounding, else the quotient by itself (each caller
// keeps to one of the two, so that its results are kept to the bit).
template <bool FUSED>
__device__ __forceinline__ double heav(double phi, double inv_eps, int& code) {
  const double t = phi * inv_eps;
  const float tf = d2f_fast(t);
  if (tf <= -1.0f) {
    code = 0;
    return 0.0;
  }
  if (tf >= 1.0f) {
    code = 1;
    return 1.0;
  }
  code = 2;
  const double q = FUSED ? fma(phi, inv_eps, 1.0) : __dadd_rn(1.0, t);
  return 0.5 * __dadd_rn(q, sin(M_PI * t) / M_PI);
}

// two-stage blend (Sec. 2): fluid value from phi, then solid from psi; away
// from both bands the value comes from the table (same expression, host)
__device__ __forceinline__ double two_stage(double h1, int c1, double h2, int c2, double zl, double zg, double zs,
                                            const double* tab) {
  if (c1 < 2 && c2 < 2) return tab[c1 + 2 * c2];
  const double zf = zl + (zg - zl) * h1;
  return zs + (zf - zs) * h2;
}

// inside a band: the cell's density and viscosity, a face's density and flow
// density with their reciprocals (rare: out of line, one copy of the code)
__device__ __noinline__ void cell_band(const PhaseConst& pc, double a, double b, double* rho, double* mu, double* imu) {
  int c1, c2;
  const double h1 = heav<true>(a, pc.inv_eps, c1), h2 = heav<true>(b, pc.inv_eps, c2);
  if (rho) *rho = two_stage(h1, c1, h2, c2, pc.rho_l, pc.rho_g, pc.rho_s, pc.rho_tab);
  const double m = two_stage(h1, c1, h2, c2, pc.mu_l, pc.mu_g, pc.mu_s, pc.mu_tab);
  *mu = m;
  if (imu) *imu = (c1 < 2 && c2 < 2) ? pc.imu_tab[c1 + 2 * c2] : 1.0 / m;
}
__device__ __noinline__ void face_band(const PhaseConst& pc, double pl, double ph, double sl, double sh, double* rho,
                                       double* beta, double* flow) {
  int c1, c2;
  const double pa = 0.5 * (pl + ph);
  const double h1 = heav<true>(pa, pc.inv_eps, c1);
  const double sa = 0.5 * (sl + sh);
  const double h2 = heav<false>(sa, pc.inv_eps, c2);
  const double r = two_stage(h1, c1, h2, c2, pc.rho_l, pc.rho_g, pc.rho_s, pc.rho_tab);
  *rho = r;
  if (beta) *beta = (c1 < 2 && c2 < 2) ? pc.beta_tab[c1 + 2 * c2] : 1.0 / r;
  if (flow) *flow = c1 < 2 ? pc.flow_tab[c1] : pc.rho_l + (pc.rho_g - pc.rho_l) * h1;
}

// Any of the pointers but rho_face may be null.
struct MatOut {
  double *rho_cc, *mu_cc;
  double *rho_face[3], *beta[3], *rho_flow[3];
};

// Cell densities and viscosities and the face densities (from face-averaged
// level sets; wall faces: the interior cell) of all three components in one
// pass: a thread owns a cell and its lower faces, and the upper one at the end of
// each axis.  Every level-set value is read once from memory: 144 us at 250 x
// 126 x 130, with a pass for the cells and one per component 195 us.  Latency and
// the float64 pipe share the time (530 warp instructions per 32 cells, the bands
// included).
__global__ void __launch_bounds__(BX* BY, 4) k_materials(GridDev g, const __grid_constant__ PhaseConst pc,
                                                      const double* __restrict__ phi, const double* __restrict__ psi,
                                                      const __grid_constant__ MatOut o) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  if (i >= n0 || j >= n1) return;
  // (32-bit offsets: every array holds fewer than 2^31 entries)
  const int pl = n0 * n1, id = (k * n1 + j) * n0 + i;
  const int lo[3] = {id - (i > 0 ? 1 : 0), id - (j > 0 ? n0 : 0), id - (k > 0 ? pl : 0)};
  const double a = phi[id], b = psi[id];
  double an[3], bn[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    an[d] = phi[lo[d]];
    bn[d] = psi[lo[d]];
  }
  const float ie = pc.inv_eps_f, eb = 9.5367431640625e-07f;
  const float af = d2f_fast(a), bf = d2f_fast(b);
  if (o.mu_cc) {
    // bound: 2^-20 |t|, far above the float32 rounding of phi and of phi/eps
    const int c1 = band_code_f(af * ie, eb * fabsf(af * ie)), c2 = band_code_f(bf * ie, eb * fabsf(bf * ie));
    if (c1 < 2 && c2 < 2) {
      if (o.rho_cc) o.rho_cc[id] = pc.rho_tab[c1 + 2 * c2];
      o.mu_cc[id] = pc.mu_tab[c1 + 2 * c2];
      if (pc.inv_mu) pc.inv_mu[id] = pc.imu_tab[c1 + 2 * c2];
    } else {
      cell_band(pc, a, b, o.rho_cc ? o.rho_cc + id : nullptr, o.mu_cc + id, pc.inv_mu ? pc.inv_mu + id : nullptr);
    }
  }
  const int fid[3] = {id + k * n1 + j, id + k * n0, id}, up[3] = {1, n0, pl};
  const bool last[3] = {i == n0 - 1, j == n1 - 1, k == n2 - 1};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    auto face = [&](int f, double pm, double sm) {
      // bound: 2^-20 (|phi_lo| + |phi_hi|)/eps, far above the float32 rounding of
      // the two values, their mean and the scaling
      const float pf = d2f_fast(pm), sf = d2f_fast(sm);
      const int c1 = band_code_f(0.5f * (pf + af) * ie, eb * (fabsf(pf) + fabsf(af)) * ie);
      const int c2 = band_code_f(0.5f * (sf + bf) * ie, eb * (fabsf(sf) + fabsf(bf)) * ie);
      if (c1 < 2 && c2 < 2) {  // away from both bands: table values only
        o.rho_face[d][f] = pc.rho_tab[c1 + 2 * c2];
        if (o.beta[d]) o.beta[d][f] = pc.beta_tab[c1 + 2 * c2];
        if (o.rho_flow[d]) o.rho_flow[d][f] = pc.flow_tab[c1];
      } else {
        face_band(pc, pm, a, sm, b, o.rho_face[d] + f, o.beta[d] ? o.beta[d] + f : nullptr,
                  o.rho_flow[d] ? o.rho_flow[d] + f : nullptr);
      }
    };
    face(fid[d], an[d], bn[d]);
    if (last[d]) face(fid[d] + up[d], a, b);
  }
}

// Harmonic mean 4 / sum(1/mu) of the 4 cells around an edge (mirror ghosts
// at walls).  The reciprocals come precomputed once per cell when inv_mu is
// given: a float64 division costs tens of instructions at GB300's float64
// rate, and each cell feeds twelve edges.  Where the four reciprocals are
// bit-identical table values the mean comes from the table as well.
// All three edge families in one pass (80 bytes per cell less than three): the
// seven cells around a corner are read by the corner's thread: 39 us at 250 x
// 126 x 130, by three passes 62 us.
__global__ void __launch_bounds__(BX* BY) k_mat_edges(GridDev g, const __grid_constant__ PhaseConst pc,
                                                      const double* __restrict__ mu_cc,
                                                      const double* __restrict__ inv_mu, double* e0, double* e1,
                                                      double* e2) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  if (i > n0 || j > n1) return;
  // the cells above (1) and below (0) the corner along each axis, mirrored at walls
  const int id = (min(k, n2 - 1) * n1 + min(j, n1 - 1)) * n0 + min(i, n0 - 1);
  const int dx = i > 0 && i < n0 ? 1 : 0, dy = j > 0 && j < n1 ? n0 : 0, dz = k > 0 && k < n2 ? n0 * n1 : 0;
  auto at = [&](int o) { return inv_mu ? inv_mu[id - o] : 1.0 / mu_cc[id - o]; };
  const double v = at(0), vx = at(dx), vy = at(dy), vz = at(dz), vxy = at(dx + dy), vxz = at(dx + dz), vyz = at(dy + dz);
  auto edge = [&](double* out, double a, double b, double c, double d) {
    const long long b0 = __double_as_longlong(a);
    if (b0 == __double_as_longlong(b) && b0 == __double_as_longlong(c) && b0 == __double_as_longlong(d)) {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (b0 == __double_as_longlong(pc.imu_tab[t])) {
          *out = pc.mue_tab[t];
          return;
        }
    }
    *out = 4.0 / (((a + b) + c) + d);
  };
  if (k < n2) edge(e0 + ((k * (n1 + 1) + j) * (n0 + 1) + i), v, vy, vx, vxy);
  if (j < n1) edge(e1 + ((k * n1 + j) * (n0 + 1) + i), v, vz, vx, vxz);
  if (i < n0) edge(e2 + ((k * (n1 + 1) + j) * n0 + i), v, vz, vy, vyz);
}

void phase_tables(PhaseConst& pc) {
  pc.inv_eps = 1.0 / pc.eps;
  pc.inv_eps_f = (float)pc.inv_eps;
  for (int h2 = 0; h2 < 2; ++h2)
    for (int h1 = 0; h1 < 2; ++h1) {
      const int t = h1 + 2 * h2;
      const double rf = pc.rho_l + (pc.rho_g - pc.rho_l) * (double)h1;
      pc.rho_tab[t] = pc.rho_s + (rf - pc.rho_s) * (double)h2;
      pc.beta_tab[t] = 1.0 / pc.rho_tab[t];
      const double mf = pc.mu_l + (pc.mu_g - pc.mu_l) * (double)h1;
      pc.mu_tab[t] = pc.mu_s + (mf - pc.mu_s) * (double)h2;
      pc.imu_tab[t] = 1.0 / pc.mu_tab[t];
      const double x = pc.imu_tab[t];
      pc.mue_tab[t] = 4.0 / (((x + x) + x) + x);
    }
  for (int h1 = 0; h1 < 2; ++h1) pc.flow_tab[h1] = pc.rho_l + (pc.rho_g - pc.rho_l) * (double)h1;
}

void launch_materials(const GridDev& g, const PhaseConst& pc, const double* phi, const double* psi, double* rho_cc,
                      double* mu_cc, double* const rho_face[3], double* const beta[3], double* const rho_flow[3],
                      double* const mu_e[3], cudaStream_t st) {
  MatOut o = {rho_cc, mu_cc, {}, {}, {}};
  for (int d = 0; d < 3; ++d) {
    o.rho_face[d] = rho_face[d];
    o.beta[d] = beta[d];
    o.rho_flow[d] = rho_flow[d];
  }
  { k_materials<<<grid3(g.n[0], g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, pc, phi, psi, o); WSI_COUNT(); }
  { k_mat_edges<<<grid3(g.n[0] + 1, g.n[1] + 1, g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, pc, mu_cc, pc.inv_mu, mu_e[0],
                                                                                  mu_e[1], mu_e[2]); WSI_COUNT(); }
}

void launch_face_density(const GridDev& g, const PhaseConst& pc, const double* phi, const double* psi,
                         double* const rho_face[3], cudaStream_t st) {
  MatOut o = {nullptr, nullptr, {rho_face[0], rho_face[1], rho_face[2]}, {}, {}};
  { k_materials<<<grid3(g.n[0], g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, pc, phi, psi, o); WSI_COUNT(); }
}

// =========================================================== strain-rate operator
// (L_mu q)_C at the interior C-face (i,j,k):
//   d/dx_C (2 mu dq_C/dx_C) + sum_{D != C} d/dx_D [ mu_e (dq_C/dx_D + dq_D/dx_C) ]
// diag (optional): coefficient of q_C(i,j,k) itself in L_mu q.
template <int C, typename T>
__device__ __forceinline__ T strain_at(const GridDev& g, const Coef<T>& cf, const T* const* q, int i, int j, int k,
                                       T* diag) {
  const T* qc = q[C];
  const T ihC = ginv<T>(g, C);
  int id3[3] = {i, j, k};
  T q0 = qc[fidx(g, C, i, j, k)];
  // the top row of an open top: the cell above is a ghost whose normal stress
  // is minus the one below (w mirrors evenly) and whose tangential
  // velocities are -1 times those below
  const bool top = C == 2 && k == g.n[2];
  // normal stress: cells hi = face index along C, lo = index - 1
  int lo3[3] = {i, j, k};
  lo3[C] -= 1;
  int hi3[3] = {i, j, k};
  hi3[C] += 1;
  T mu_lo = cf.mu_cc[fidx(g, 3, lo3[0], lo3[1], lo3[2])];
  T qm = qc[fidx(g, C, lo3[0], lo3[1], lo3[2])];
  T mu_hi = top ? mu_lo : cf.mu_cc[fidx(g, 3, i, j, k)];
  T qp = top ? qm : qc[fidx(g, C, hi3[0], hi3[1], hi3[2])];
  const T w = sizeof(T) == 8 ? T(2) * ginv2<T>(g, C) : T(2) * ihC * ihC;
  T L = w * (mu_hi * (qp - q0) - mu_lo * (q0 - qm));
  T dg = -T(2) * ihC * ihC * (mu_hi + mu_lo);
#pragma unroll
  for (int D = 0; D < 3; ++D) {
    if (D == C) continue;
    const int E = edge_id(C, D);
    const T ihD = ginv<T>(g, D);
    const T* qd = q[D];
    // neighbours along D (ghosts beyond walls mirror with the wall sign)
    int a3[3] = {id3[0], id3[1], id3[2]};
    int b3[3] = {id3[0], id3[1], id3[2]};
    a3[D] += 1;
    b3[D] -= 1;
    T q_hi, q_lo, s_hi = T(0), s_lo = T(0);
    if (a3[D] >= g.n[D]) {
      s_hi = gbc<T>(g, 2 * D + 1);
      q_hi = s_hi * q0;
    } else {
      q_hi = qc[fidx(g, C, a3[0], a3[1], a3[2])];
    }
    if (b3[D] < 0) {
      s_lo = gbc<T>(g, 2 * D);
      q_lo = s_lo * q0;
    } else {
      q_lo = qc[fidx(g, C, b3[0], b3[1], b3[2])];
    }
    // edges: along C at the face index, along D at j_D (lo) and j_D + 1 (hi)
    int eh[3] = {id3[0], id3[1], id3[2]};
    eh[D] += 1;
    T mue_hi = cf.mu_e[E][eidx(g, E, eh[0], eh[1], eh[2])];
    T mue_lo = cf.mu_e[E][eidx(g, E, id3[0], id3[1], id3[2])];
    // q_D on D-faces adjacent along C: cells (index along C) id-1 and id
    int d1[3] = {id3[0], id3[1], id3[2]};  // hi edge, cell id
    d1[D] += 1;
    int d0[3] = {d1[0], d1[1], d1[2]};
    d0[C] -= 1;
    const T qd_d0 = qd[fidx(g, D, d0[0], d0[1], d0[2])];
    const T qd_d1 = top ? gbc<T>(g, 5) * qd_d0 : qd[fidx(g, D, d1[0], d1[1], d1[2])];
    T dqd_hi = (qd_d1 - qd_d0) * ihC;
    int c1[3] = {id3[0], id3[1], id3[2]};  // lo edge
    int c0[3] = {id3[0], id3[1], id3[2]};
    c0[C] -= 1;
    const T qd_c0 = qd[fidx(g, D, c0[0], c0[1], c0[2])];
    const T qd_c1 = top ? gbc<T>(g, 5) * qd_c0 : qd[fidx(g, D, c1[0], c1[1], c1[2])];
    T dqd_lo = (qd_c1 - qd_c0) * ihC;
    T f_hi = mue_hi * ((q_hi - q0) * ihD + dqd_hi);
    T f_lo = mue_lo * ((q0 - q_lo) * ihD + dqd_lo);
    L += (f_hi - f_lo) * ihD;
    dg += (mue_hi * (s_hi - T(1)) - mue_lo * (T(1) - s_lo)) * ihD * ihD;
  }
  if (diag) *diag = dg;
  return L;
}

template <int C, typename T>
__global__ void k_viscous(GridDev g, Coef<T> cf, T inv_dt, T theta, CVel<T> q, T* out, const T* b, bool strain_only) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  int e0 = ext(g, C, 0), e1 = ext(g, C, 1);
  if (i >= e0 || j >= e1) return;
  int id3[3] = {i, j, k};
  size_t id = fidx(g, C, i, j, k);
  if (!face_row(g, C, id3[C])) {
    out[id] = T(0);
    return;
  }
  T L = strain_at<C, T>(g, cf, q.q, i, j, k, nullptr);
  T a;
  if (strain_only)
    a = L;
  else
    a = cf.rho_face[C][id] * inv_dt * q.q[C][id] - theta * L;
  out[id] = b ? b[id] - a : a;
}

template <typename T>
void launch_viscous(const GridDev& g, const Coef<T>& cf, T inv_dt, T theta, const T* const q[3], T* const out[3],
                    cudaStream_t st, bool strain_only) {
  CVel<T> cq{{q[0], q[1], q[2]}};
  { k_viscous<0, T><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, cq, out[0],
                                                                              nullptr, strain_only); WSI_COUNT(); }
  { k_viscous<1, T><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, cq, out[1],
                                                                              nullptr, strain_only); WSI_COUNT(); }
  { k_viscous<2, T><<<grid3(g.n[0], g.n[1], g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, cq, out[2],
                                                                              nullptr, strain_only); WSI_COUNT(); }
}

template <typename T>
void launch_viscous_residual(const GridDev& g, const Coef<T>& cf, T inv_dt, T theta, const T* const q[3],
                             const T* const b[3], T* const r[3], cudaStream_t st) {
  CVel<T> cq{{q[0], q[1], q[2]}};
  { k_viscous<0, T><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, cq, r[0], b[0],
                                                                              false); WSI_COUNT(); }
  { k_viscous<1, T><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, cq, r[1], b[1],
                                                                              false); WSI_COUNT(); }
  { k_viscous<2, T><<<grid3(g.n[0], g.n[1], g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, cq, r[2], b[2],
                                                                              false); WSI_COUNT(); }
}

// red-black Gauss-Seidel on component C of the viscous block: the other
// components and the other colour are read as they stand.
template <int C, typename T>
__global__ void k_viscous_rbgs(GridDev g, Coef<T> cf, T inv_dt, T theta, Vel<T> q, const T* __restrict__ b,
                               int color) {
  // thread t of a row owns the t-th face of the colour: i = 2t + ((j + k + color) & 1)
  const int j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  const int i = 2 * (blockIdx.x * BX + threadIdx.x) + ((j + k + color) & 1);
  int e0 = ext(g, C, 0), e1 = ext(g, C, 1);
  if (i >= e0 || j >= e1) return;
  int id3[3] = {i, j, k};
  if (!face_row(g, C, id3[C])) return;
  size_t id = fidx(g, C, i, j, k);
  T dg;
  const T* cq[3] = {q.q[0], q.q[1], q.q[2]};
  T L = strain_at<C, T>(g, cf, cq, i, j, k, &dg);
  T rf = cf.rho_face[C][id] * inv_dt;
  T a = rf * q.q[C][id] - theta * L;
  T d = rf - theta * dg;
  q.q[C][id] += (b[id] - a) / d;
}

// The same with the inverse diagonals from memory: the float64 pipe bounds the
// update, and the diagonal and its division were 25 of its 60 operations (at 128
// x 64 x 64 36 -> 22 us per component and half sweep).
template <int C>
__global__ void k_viscous_rbgs_d(GridDev g, Coef<double> cf, double inv_dt, double theta, Vel<double> q,
                                 const double* __restrict__ b, const double* __restrict__ vd, int color) {
  const int j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  const int i = 2 * (blockIdx.x * BX + threadIdx.x) + ((j + k + color) & 1);
  if (i >= ext(g, C, 0) || j >= ext(g, C, 1)) return;
  int id3[3] = {i, j, k};
  if (!face_row(g, C, id3[C])) return;
  const size_t id = fidx(g, C, i, j, k);
  const double* cq[3] = {q.q[0], q.q[1], q.q[2]};
  const double L = strain_at<C, double>(g, cf, cq, i, j, k, nullptr);
  const double q0 = q.q[C][id], r = fma(-(cf.rho_face[C][id] * inv_dt), q0, b[id]);
  q.q[C][id] = fma(fma(theta, L, r), vd[id], q0);
}

// (q: arrays of the velocity's shape; the operator's value is not used)
template <int C>
__global__ void k_viscous_diag(GridDev g, Coef<double> cf, double inv_dt, double theta, CVel<double> q, double* vd) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ext(g, C, 0) || j >= ext(g, C, 1)) return;
  int id3[3] = {i, j, k};
  const size_t id = fidx(g, C, i, j, k);
  double dg = 0.0;
  if (face_row(g, C, id3[C])) {
    strain_at<C, double>(g, cf, q.q, i, j, k, &dg);
    dg = 1.0 / (cf.rho_face[C][id] * inv_dt - theta * dg);
  }
  vd[id] = dg;
}

void launch_viscous_diag(const GridDev& g, const Coef<double>& cf, double inv_dt, double theta,
                         const double* const q[3], double* const vd[3], cudaStream_t st) {
  const CVel<double> v{{q[0], q[1], q[2]}};
  const dim3 blk(BX, BY);
  { k_viscous_diag<0><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), blk, 0, st>>>(g, cf, inv_dt, theta, v, vd[0]); WSI_COUNT(); }
  { k_viscous_diag<1><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), blk, 0, st>>>(g, cf, inv_dt, theta, v, vd[1]); WSI_COUNT(); }
  { k_viscous_diag<2><<<grid3(g.n[0], g.n[1], g.n[2] + 1), blk, 0, st>>>(g, cf, inv_dt, theta, v, vd[2]); WSI_COUNT(); }
}

template <int C, typename T>
static void viscous_rbgs_one(const GridDev& g, const Coef<T>& cf, T inv_dt, T theta, const Vel<T>& q, const T* b,
                             const T* vd, int color, cudaStream_t st) {
  const dim3 grid = grid3((ext(g, C, 0) + 1) / 2, ext(g, C, 1), ext(g, C, 2)), blk(BX, BY);
  if constexpr (sizeof(T) == 8) {
    if (vd) {
      { k_viscous_rbgs_d<C><<<grid, blk, 0, st>>>(g, cf, inv_dt, theta, q, b, vd, color); WSI_COUNT(); }
      return;
    }
  }
  { k_viscous_rbgs<C, T><<<grid, blk, 0, st>>>(g, cf, inv_dt, theta, q, b, color); WSI_COUNT(); }
}

template <typename T>
void launch_viscous_rbgs(const GridDev& g, const Coef<T>& cf, T inv_dt, T theta, T* const q[3], const T* const b[3],
                         int color, cudaStream_t st, T* const* vd) {
  Vel<T> vq{{q[0], q[1], q[2]}};
  ktimer_begin(KC_RBGS_V, st);
  viscous_rbgs_one<0, T>(g, cf, inv_dt, theta, vq, b[0], vd ? vd[0] : nullptr, color, st);
  viscous_rbgs_one<1, T>(g, cf, inv_dt, theta, vq, b[1], vd ? vd[1] : nullptr, color, st);
  if (g.n[2] > 1) viscous_rbgs_one<2, T>(g, cf, inv_dt, theta, vq, b[2], vd ? vd[2] : nullptr, color, st);
  ktimer_end(KC_RBGS_V, st);
}

// =========================================================== pressure, grad, div
template <typename T>
__global__ void k_pressure(GridDev g, const T* __restrict__ bx, const T* __restrict__ by, const T* __restrict__ bz,
                           const T* __restrict__ p, T* out) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= g.n[0] || j >= g.n[1]) return;
  size_t id = fidx(g, 3, i, j, k);
  T pc = p[id];
  T s = T(0);
  T ihx2 = ginv2<T>(g, 0), ihy2 = ginv2<T>(g, 1), ihz2 = ginv2<T>(g, 2);
  if (i + 1 < g.n[0]) s += bx[fidx(g, 0, i + 1, j, k)] * (p[id + 1] - pc) * ihx2;
  if (i > 0) s -= bx[fidx(g, 0, i, j, k)] * (pc - p[id - 1]) * ihx2;
  if (j + 1 < g.n[1]) s += by[fidx(g, 1, i, j + 1, k)] * (p[id + g.n[0]] - pc) * ihy2;
  if (j > 0) s -= by[fidx(g, 1, i, j, k)] * (pc - p[id - g.n[0]]) * ihy2;
  size_t pl = (size_t)g.n[0] * g.n[1];
  if (k + 1 < g.n[2]) s += bz[fidx(g, 2, i, j, k + 1)] * (p[id + pl] - pc) * ihz2;
  else if (g.open_top) s -= T(2) * bz[fidx(g, 2, i, j, k + 1)] * pc * ihz2;  // ghost -p above the open top
  if (k > 0) s -= bz[fidx(g, 2, i, j, k)] * (pc - p[id - pl]) * ihz2;
  out[id] = s;
}

template <typename T>
void launch_pressure(const GridDev& g, const T* const beta[3], const T* p, T* out, cudaStream_t st) {
  { k_pressure<T><<<grid3(g.n[0], g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, beta[0], beta[1], beta[2], p, out); WSI_COUNT(); }
}

// r = y - D beta G x in float64 with the partials of its sum and square sum.
// Float64-pipe bound, so every flux beta dx is formed once: along x the upper
// face comes from the next lane, along y from the next row through shared
// memory, along z it is carried up the march; a ninth warp forms the fluxes
// through the tile's upper edges (x: one lane per row, y: one per column).  14
// operations per cell where five passes (k_pressure, the difference, its sum,
// the removal of its mean, its norm) took 23, 562 us in k_pressure alone: 495 us at
// 256^3 (at the float64 rate 14.5 operations take 450).
static constexpr int QX = 32, QY = 8, QZ = 16;
// the block's barrier, met from two places of the code (the ninth warp's loop and
// the others')
__device__ __forceinline__ void tile_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * (QY + 1)) : "memory"); }

__global__ void __launch_bounds__(32 * (QY + 1)) k_pressure_residual(GridDev g, const double* __restrict__ bx,
                                                                     const double* __restrict__ by,
                                                                     const double* __restrict__ bz,
                                                                     const double* __restrict__ x,
                                                                     const double* __restrict__ y, double* r,
                                                                     int zchunk, double* part) {
  __shared__ double sF[2][QY + 1][32];  // flux through the lower y face
  __shared__ double sX[2][QY];          // flux through the tile's upper x edge
  __shared__ double sh[2][QY];
  const int lane = threadIdx.x, ty = threadIdx.y;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const int x0 = blockIdx.x * QX, y0 = blockIdx.y * QY;
  const int k0 = blockIdx.z * zchunk, k1 = min(k0 + zchunk, nz);
  const int i = x0 + lane, j = y0 + ty;
  const double wx = g.ih2[0], wy = g.ih2[1], wz = g.ih2[2];
  const size_t pl = (size_t)nx * ny, px = (size_t)(nx + 1) * ny, py = (size_t)nx * (ny + 1);
  double s1 = 0.0, s2 = 0.0;
  if (ty == QY) {
    // upper edges: the row j = y0 + QY, and column x0 + QX of rows y0 + lane
    const bool row = i < nx && j < ny, col = lane < QY && y0 + lane < ny && x0 + QX < nx;
    size_t id = row ? (size_t)k0 * pl + (size_t)j * nx + i : 0, iy = row ? fidx(g, 1, i, j, k0) : 0;
    size_t ic = col ? (size_t)k0 * pl + (size_t)(y0 + lane) * nx + x0 + QX : 0;
    size_t ix = col ? fidx(g, 0, x0 + QX, y0 + lane, k0) : 0;
    for (int k = k0; k < k1; ++k) {
      sF[k & 1][QY][lane] = row ? by[iy] * (x[id] - x[id - nx]) : 0.0;
      if (lane < QY) sX[k & 1][lane] = col ? bx[ix] * (x[ic] - x[ic - 1]) : 0.0;
      id += pl;
      iy += py;
      ic += pl;
      ix += px;
      tile_sync();
    }
    tile_sync();
    if (lane >= 2) return;
    double a = 0.0;
    for (int w = 0; w < QY; ++w) a += sh[lane][w];
    part[2 * (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) + lane] = a;
    return;
  }
  const bool cell = i < nx && j < ny;
  size_t id = cell ? (size_t)k0 * pl + (size_t)j * nx + i : 0;
  size_t ix = cell ? fidx(g, 0, i, j, k0) : 0, iy = cell ? fidx(g, 1, i, j, k0) : 0;
  double xc = cell ? x[id] : 0.0, fz = 0.0;
  if (cell && k0 > 0) fz = bz[id] * (xc - x[id - pl]);
  for (int k = k0; k < k1; ++k) {
    const double xn = cell && k + 1 < nz ? x[id + pl] : 0.0;
    double fx = 0.0, fy = 0.0;
    if (cell && i > 0) fx = bx[ix] * (xc - x[id - 1]);
    if (cell && j > 0) fy = by[iy] * (xc - x[id - nx]);
    sF[k & 1][ty][lane] = fy;
    double fxr = __shfl_down_sync(0xffffffffu, fx, 1);  // (zero beyond the grid)
    tile_sync();
    if (cell) {
      if (lane == 31) fxr = sX[k & 1][ty];
      const double fyr = sF[k & 1][ty + 1][lane];
      double fzr = 0.0;
      if (k + 1 < nz) fzr = bz[id + pl] * (xn - xc);
      else if (g.open_top) fzr = -2.0 * bz[id + pl] * xc;  // ghost -p above the open top
      const double v = fma(fx - fxr, wx, fma(fy - fyr, wy, fma(fz - fzr, wz, y[id])));
      r[id] = v;
      s1 += v;
      s2 = fma(v, v, s2);
      fz = fzr;
      xc = xn;
    }
    id += pl;
    ix += px;
    iy += py;
  }
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_down_sync(0xffffffffu, s1, o);
    s2 += __shfl_down_sync(0xffffffffu, s2, o);
  }
  if (lane == 0) {
    sh[0][ty] = s1;
    sh[1][ty] = s2;
  }
  tile_sync();
}

__global__ void __launch_bounds__(1024) k_reduce_pairs(const double* __restrict__ part, size_t n, double* out) {
  __shared__ double sh[2][32];
  double a = 0.0, b = 0.0;
  for (size_t t = threadIdx.x; t < n; t += 1024) {
    a += part[2 * t];
    b += part[2 * t + 1];
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    sh[0][threadIdx.x >> 5] = a;
    sh[1][threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int w = 0; w < 32; ++w) s += sh[threadIdx.x][w];
    out[threadIdx.x] = s;
  }
}

double host_pressure_residual(const GridDev& g, const double* const beta[3], const double* x, const double* y, double* r,
                              double* scratch, double* mean, cudaStream_t st) {
  const int bx = cdiv(g.n[0], QX), by = cdiv(g.n[1], QY);
  int zc = QZ;  // shorter marches where the grid is small
  while (zc > 2 && (long long)bx * by * cdiv(g.n[2], zc) < 152 * 4) zc /= 2;
  const dim3 grid(bx, by, cdiv(g.n[2], zc));
  const size_t nb = (size_t)grid.x * grid.y * grid.z;
  { k_pressure_residual<<<grid, dim3(32, QY + 1), 0, st>>>(g, beta[0], beta[1], beta[2], x, y, r, zc, scratch + 2); WSI_COUNT(); }
  { k_reduce_pairs<<<1, 1024, 0, st>>>(scratch + 2, nb, scratch); WSI_COUNT(); }
  double h[2] = {0.0, 0.0};
  cudaMemcpyAsync(h, scratch, sizeof(h), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  if (!mean) return sqrt(h[1]);
  const double n = (double)g.n[0] * g.n[1] * g.n[2];
  *mean = h[0] / n;
  // (sums that overflow or hold a NaN are no small residual: inf - inf below)
  if (!std::isfinite(h[0]) || !std::isfinite(h[1])) return std::numeric_limits<double>::infinity();
  return sqrt(std::max(h[1] - h[0] * *mean, 0.0));
}

template <int C, typename T>
__global__ void k_grad(GridDev g, const T* __restrict__ p, T* out) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ext(g, C, 0) || j >= ext(g, C, 1)) return;
  int id3[3] = {i, j, k};
  size_t id = fidx(g, C, i, j, k);
  if (!face_row(g, C, id3[C])) {
    out[id] = T(0);
    return;
  }
  int lo3[3] = {i, j, k};
  lo3[C] -= 1;
  const T plo = p[fidx(g, 3, lo3[0], lo3[1], lo3[2])];
  const T phi = (C == 2 && k == g.n[2]) ? -plo : p[fidx(g, 3, i, j, k)];  // open top: ghost -p
  out[id] = (phi - plo) * ginv<T>(g, C);
}

template <typename T>
void launch_grad(const GridDev& g, const T* p, T* const out[3], cudaStream_t st) {
  { k_grad<0, T><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, p, out[0]); WSI_COUNT(); }
  { k_grad<1, T><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), dim3(BX, BY), 0, st>>>(g, p, out[1]); WSI_COUNT(); }
  { k_grad<2, T><<<grid3(g.n[0], g.n[1], g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, p, out[2]); WSI_COUNT(); }
}

template <typename T>
__global__ void k_div(GridDev g, const T* __restrict__ u, const T* __restrict__ v, const T* __restrict__ w, T* out,
                      T scale) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= g.n[0] || j >= g.n[1]) return;
  T d = (u[fidx(g, 0, i + 1, j, k)] - u[fidx(g, 0, i, j, k)]) * ginv<T>(g, 0) +
        (v[fidx(g, 1, i, j + 1, k)] - v[fidx(g, 1, i, j, k)]) * ginv<T>(g, 1) +
        (w[fidx(g, 2, i, j, k + 1)] - w[fidx(g, 2, i, j, k)]) * ginv<T>(g, 2);
  out[fidx(g, 3, i, j, k)] = scale * d;
}

template <typename T>
void launch_div(const GridDev& g, const T* const q[3], T* out, T scale, cudaStream_t st) {
  { k_div<T><<<grid3(g.n[0], g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, q[0], q[1], q[2], out, scale); WSI_COUNT(); }
}

// packed Stokes matvec: momentum rows A u + G p (zero on wall faces)
template <int C>
__device__ __forceinline__ void stokes_row(const GridDev& g, const Coef<double>& cf, double inv_dt, double theta,
                                           const CVel<double>& q, const double* __restrict__ p, double* out, int i,
                                           int j, int k) {
  int id3[3] = {i, j, k};
  size_t id = fidx(g, C, i, j, k);
  if (!face_row(g, C, id3[C])) {
    out[id] = 0.0;
    return;
  }
  double L = strain_at<C, double>(g, cf, q.q, i, j, k, nullptr);
  int lo3[3] = {i, j, k};
  lo3[C] -= 1;
  const double plo = p[fidx(g, 3, lo3[0], lo3[1], lo3[2])];
  const double phi = (C == 2 && k == g.n[2]) ? -plo : p[fidx(g, 3, i, j, k)];  // open top: ghost -p
  double gp = (phi - plo) * g.ih[C];
  out[id] = cf.rho_face[C][id] * inv_dt * q.q[C][id] - theta * L + gp;
}

// One launch covers the whole packed vector: blockIdx.z walks the z-planes of
// the u, v and w momentum rows, then the continuity rows.
__global__ void k_stokes(GridDev g, Coef<double> cf, double inv_dt, double theta, CVel<double> q,
                         const double* __restrict__ p, double* yu, double* yv, double* yw, double* yp) {
  int z = blockIdx.z;
  int nz = g.n[2];
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y;
  if (z < nz) {
    if (i < g.n[0] + 1 && j < g.n[1]) stokes_row<0>(g, cf, inv_dt, theta, q, p, yu, i, j, z);
  } else if (z < 2 * nz) {
    if (i < g.n[0] && j < g.n[1] + 1) stokes_row<1>(g, cf, inv_dt, theta, q, p, yv, i, j, z - nz);
  } else if (z < 3 * nz + 1) {
    if (i < g.n[0] && j < g.n[1]) stokes_row<2>(g, cf, inv_dt, theta, q, p, yw, i, j, z - 2 * nz);
  } else {
    int k = z - (3 * nz + 1);
    if (i < g.n[0] && j < g.n[1]) {
      double d = (q.q[0][fidx(g, 0, i + 1, j, k)] - q.q[0][fidx(g, 0, i, j, k)]) * g.ih[0] +
                 (q.q[1][fidx(g, 1, i, j + 1, k)] - q.q[1][fidx(g, 1, i, j, k)]) * g.ih[1] +
                 (q.q[2][fidx(g, 2, i, j, k + 1)] - q.q[2][fidx(g, 2, i, j, k)]) * g.ih[2];
      yp[fidx(g, 3, i, j, k)] = -d;
    }
  }
}

void launch_stokes(const GridDev& g, const Coef<double>& cf, double inv_dt, double theta, const double* x, double* y,
                   cudaStream_t st) {
  Packing pk = packing(g);
  CVel<double> q{{x + pk.off[0], x + pk.off[1], x + pk.off[2]}};
  const double* p = x + pk.off[3];
  dim3 grid(cdiv(g.n[0] + 1, BX), cdiv(g.n[1] + 1, BY), 4 * g.n[2] + 1);
  ktimer_begin(KC_STOKES, st);
  { k_stokes<<<grid, dim3(BX, BY), 0, st>>>(g, cf, inv_dt, theta, q, p, y + pk.off[0], y + pk.off[1],
                                            y + pk.off[2], y + pk.off[3]); WSI_COUNT(); }
  ktimer_end(KC_STOKES, st);
}

template <int C>
__global__ void k_zero_walls(GridDev g, double* q) {
  // walls normal to C: planes index 0 and n along C
  int a = blockIdx.x * BX + threadIdx.x, b = blockIdx.y * BY + threadIdx.y, side = blockIdx.z;
  constexpr int A = (C == 0) ? 1 : 0;
  constexpr int B = (C == 2) ? 1 : 2;
  if (a >= g.n[A] || b >= g.n[B]) return;
  if (C == 2 && side && g.open_top) return;  // the open top's faces are unknowns
  int c3[3];
  c3[C] = side ? g.n[C] : 0;
  c3[A] = a;
  c3[B] = b;
  q[fidx(g, C, c3[0], c3[1], c3[2])] = 0.0;
}

void launch_zero_walls(const GridDev& g, double* const q[3], cudaStream_t st) {
  { k_zero_walls<0><<<dim3(cdiv(g.n[1], BX), cdiv(g.n[2], BY), 2), dim3(BX, BY), 0, st>>>(g, q[0]); WSI_COUNT(); }
  { k_zero_walls<1><<<dim3(cdiv(g.n[0], BX), cdiv(g.n[2], BY), 2), dim3(BX, BY), 0, st>>>(g, q[1]); WSI_COUNT(); }
  { k_zero_walls<2><<<dim3(cdiv(g.n[0], BX), cdiv(g.n[1], BY), 2), dim3(BX, BY), 0, st>>>(g, q[2]); WSI_COUNT(); }
}

// =========================================================== momentum RHS
template <int C, typename T>
__global__ void k_rhs_base(GridDev g, Coef<T> cf_n, CVel<T> uT, const double* __restrict__ rho_n,
                           const double* __restrict__ un, double inv_dt, double theta, double* b0) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ext(g, C, 0) || j >= ext(g, C, 1)) return;
  int id3[3] = {i, j, k};
  size_t id = fidx(g, C, i, j, k);
  if (!face_row(g, C, id3[C])) {
    b0[id] = 0.0;
    return;
  }
  T L = strain_at<C, T>(g, cf_n, uT.q, i, j, k, nullptr);
  b0[id] = rho_n[id] * un[id] * inv_dt + (1.0 - theta) * (double)L;
}

template <typename T>
void launch_rhs_base(const GridDev& g, const Coef<T>& cf_n, const T* const uT[3], const double* const rho_n[3],
                     const double* const u_n[3], double inv_dt, double theta, double* const b0[3], cudaStream_t st) {
  CVel<T> u{{uT[0], uT[1], uT[2]}};
  { k_rhs_base<0, T><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, cf_n, u, rho_n[0], u_n[0], inv_dt,
                                                                               theta, b0[0]); WSI_COUNT(); }
  { k_rhs_base<1, T><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), dim3(BX, BY), 0, st>>>(g, cf_n, u, rho_n[1], u_n[1], inv_dt,
                                                                               theta, b0[1]); WSI_COUNT(); }
  { k_rhs_base<2, T><<<grid3(g.n[0], g.n[1], g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, cf_n, u, rho_n[2], u_n[2], inv_dt,
                                                                               theta, b0[2]); WSI_COUNT(); }
}

// b = b0 - C + rho_g g over the packed velocity vector; wall faces are zero
// in b0, C and on output
// (one component per blockIdx.y; gmask: those with gravity, as bits.  The others
// have a loop of their own without the density and its two float64 operations,
// which even predicated off bound the pass: 300 -> 232 us at 256^3.)
struct RhsParts {
  size_t off[3], n[3];
  const double* rg[3];
  double g[3];
  int gmask;
};
template <typename TC>
__global__ void k_rhs_cycle(RhsParts p, const double* __restrict__ b0, const TC* __restrict__ Cc, double* b) {
  const int c = blockIdx.y;
  const size_t stride = (size_t)gridDim.x * blockDim.x, n = p.n[c], o = p.off[c];
  const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p.gmask >> c & 1) {
    const double* __restrict__ rg = p.rg[c];
    const double g = p.g[c];
    for (size_t t = t0; t < n; t += stride)
      b[o + t] = __dadd_rn(b0[o + t] - cvt<double, TC>(Cc[o + t]), __dmul_rn(rg[t], g));
  } else {
    for (size_t t = t0; t < n; t += stride) b[o + t] = b0[o + t] - cvt<double, TC>(Cc[o + t]);
  }
}

template <typename TC>
void launch_rhs_cycle(const GridDev& g, const double* b0, const TC* C, const double* const rho_g[3],
                      const double grav[3], double* b, cudaStream_t st) {
  size_t n0 = fsize(g, 0), n1 = fsize(g, 1), n2 = fsize(g, 2);
  RhsParts p = {{0, n0, n0 + n1}, {n0, n1, n2}, {rho_g[0], rho_g[1], rho_g[2]}, {grav[0], grav[1], grav[2]}, 0};
  for (int d = 0; d < 3; ++d) p.gmask |= (grav[d] != 0.0) << d;
  const int blocks = (int)std::min<size_t>((std::max(n0, std::max(n1, n2)) + 255) / 256, 152 * 16);
  { k_rhs_cycle<TC><<<dim3(blocks, 3), 256, 0, st>>>(p, b0, C, b); WSI_COUNT(); }
  double* q[3] = {b, b + n0, b + n0 + n1};
  launch_zero_walls(g, q, st);
}

// Non-conservative form (Sec. 4.2.3): b = b0 + rho (u^n/dt - N) + rho_g g with
// b0 = (1 - theta) L_mu^n u^n and rho = rho^{n+1,k+1} the face density of the
// level sets; wall faces are zero on output
template <typename TN>
__global__ void k_rhs_nc(size_t n0, size_t n1, size_t n2, const double* __restrict__ b0, const TN* __restrict__ N,
                         const double* __restrict__ r0, const double* __restrict__ r1, const double* __restrict__ r2,
                         const double* __restrict__ un, double inv_dt, const double* __restrict__ rg0,
                         const double* __restrict__ rg1, const double* __restrict__ rg2, double g0, double g1,
                         double g2, double* b) {
  size_t stride = (size_t)gridDim.x * blockDim.x;
  size_t n = n0 + n1 + n2;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    double rho, grav = 0.0;
    if (t < n0) {
      rho = r0[t];
      if (g0 != 0.0) grav = rg0[t] * g0;
    } else if (t < n0 + n1) {
      rho = r1[t - n0];
      if (g1 != 0.0) grav = rg1[t - n0] * g1;
    } else {
      rho = r2[t - n0 - n1];
      if (g2 != 0.0) grav = rg2[t - n0 - n1] * g2;
    }
    b[t] = b0[t] + rho * (un[t] * inv_dt - cvt<double, TN>(N[t])) + grav;
  }
}

template <typename TN>
void launch_rhs_nc(const GridDev& g, const double* b0, const TN* N, const double* const rho[3], const double* u_n,
                   double inv_dt, const double* const rho_g[3], const double grav[3], double* b, cudaStream_t st) {
  size_t n0 = fsize(g, 0), n1 = fsize(g, 1), n2 = fsize(g, 2);
  int blocks = (int)std::min<size_t>((n0 + n1 + n2 + 255) / 256, 152 * 16);
  { k_rhs_nc<TN><<<blocks, 256, 0, st>>>(n0, n1, n2, b0, N, rho[0], rho[1], rho[2], u_n, inv_dt, rho_g[0], rho_g[1],
                                         rho_g[2], grav[0], grav[1], grav[2], b); WSI_COUNT(); }
  double* q[3] = {b, b + n0, b + n0 + n1};
  launch_zero_walls(g, q, st);
}
template void launch_rhs_nc<double>(const GridDev&, const double*, const double*, const double* const[3],
                                    const double*, double, const double* const[3], const double[3], double*,
                                    cudaStream_t);
template void launch_rhs_nc<float>(const GridDev&, const double*, const float*, const double* const[3],
                                   const double*, double, const double* const[3], const double[3], double*,
                                   cudaStream_t);

template void launch_rhs_base<double>(const GridDev&, const Coef<double>&, const double* const[3],
                                      const double* const[3], const double* const[3], double, double,
                                      double* const[3], cudaStream_t);
template void launch_rhs_base<float>(const GridDev&, const Coef<float>&, const float* const[3],
                                     const double* const[3], const double* const[3], double, double,
                                     double* const[3], cudaStream_t);
template void launch_rhs_cycle<double>(const GridDev&, const double*, const double*, const double* const[3],
                                       const double[3], double*, cudaStream_t);
template void launch_rhs_cycle<float>(const GridDev&, const double*, const float*, const double* const[3],
                                      const double[3], double*, cudaStream_t);

// explicit instantiations
template void launch_viscous<double>(const GridDev&, const Coef<double>&, double, double, const double* const[3],
                                     double* const[3], cudaStream_t, bool);
template void launch_viscous<float>(const GridDev&, const Coef<float>&, float, float, const float* const[3],
                                    float* const[3], cudaStream_t, bool);
template void launch_viscous_residual<double>(const GridDev&, const Coef<double>&, double, double,
                                              const double* const[3], const double* const[3], double* const[3],
                                              cudaStream_t);
template void launch_viscous_residual<float>(const GridDev&, const Coef<float>&, float, float, const float* const[3],
                                             const float* const[3], float* const[3], cudaStream_t);
template void launch_viscous_rbgs<double>(const GridDev&, const Coef<double>&, double, double, double* const[3],
                                          const double* const[3], int, cudaStream_t, double* const*);
template void launch_viscous_rbgs<float>(const GridDev&, const Coef<float>&, float, float, float* const[3],
                                         const float* const[3], int, cudaStream_t, float* const*);
template void launch_pressure<double>(const GridDev&, const double* const[3], const double*, double*, cudaStream_t);
template void launch_pressure<float>(const GridDev&, const float* const[3], const float*, float*, cudaStream_t);
template void launch_grad<double>(const GridDev&, const double*, double* const[3], cudaStream_t);
template void launch_grad<float>(const GridDev&, const float*, float* const[3], cudaStream_t);
template void launch_div<double>(const GridDev&, const double* const[3], double*, double, cudaStream_t);
template void launch_div<float>(const GridDev&, const float* const[3], float*, float, cudaStream_t);

}  // namespace wsi
