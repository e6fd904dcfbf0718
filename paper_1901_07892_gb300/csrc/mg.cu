// Projection preconditioner of the implicit Stokes system (Sec. 4.2.4; the
// paper cites the variable-coefficient projection method without printing
// it) with a cell-centred geometric multigrid for the pressure operator
// D(beta G).  Templated on the arithmetic type T: float64 for the plain
// path, float32 inside float64 FGMRES for the mixed path.
//
// One application  z = P^{-1} r  (r = (r_u, r_p)):
//   u~ = A^{-1} r_u      by red-black Gauss-Seidel sweeps on the viscous block
//   y  = r_p + D u~      (mean removed: closed box)
//   phi = L_beta^{-1} y   by V-cycles
//   p  = phi/dt - theta mu y,    u = u~ - beta G phi
// which is the block factorisation of K with the Schur complement
// D A^{-1} G approximated by dt D beta G plus the local-viscosity term.
//
// Multigrid: coarsening by 2 along every axis whose extent is even and >= 4,
// until <= 64 cells; coarse face beta = mean of the coplanar fine faces;
// restriction = mean of the 2^d children (fused with the residual);
// prolongation = (bi/tri)linear on cell centres (fused with the correction);
// smoother = red-black Gauss-Seidel; coarsest = dense float64 inverse of the
// operator regularised on its constant null space.
#include <math.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "df.cuh"
#include "internal.h"

namespace wsi {

static constexpr int BX = 32, BY = 8;
static inline dim3 grid3(int nx, int ny, int nz) { return dim3(cdiv(nx, BX), cdiv(ny, BY), nz); }

template <typename T>
__global__ void k_coarse_inverse(GridDev g, const T* __restrict__ bx, const T* __restrict__ by,
                                 const T* __restrict__ bz, int n, double* inv);
static constexpr int INV_MAX = 160;  // cells of a coarsest level that is inverted on the device
template <typename T>
struct CoarseCycle;
template <typename T, int NT>
__global__ void k_coarse_cycle(const __grid_constant__ CoarseCycle<T> c);
// Cells of a level that one block works on in shared memory, and of one that the
// fused lower cycle takes at all.  float64 updates are bound by the narrow pipe of
// the SMs that take part, so there the whole GPU wins earlier.  Measured per V-cycle
// in float64, fused from 512, 4096 and 32768 cells down: 16^3 121, 110 and 110 us, 32 x 16 x 16
// 167, 148 and 136, 32^3 178, 166 and 180, 64^2 161, 132 and 132, 128^2 212, 183 and
// 176; one block up to 256, 512 and 1024 cells: 16^3 119, 110 and 110, 64^2 132, 132
// and 124 (float32 16^3 80, 71 and 71, 64^2 82, 82 and 72).
template <typename T>
static constexpr int coarse_smem_cells() { return 512; }
template <typename T>
static constexpr int coarse_max_cells() { return sizeof(T) == 4 ? 65536 : 4096; }
template <typename T>
static constexpr int coarse_threads() { return 512; }

template <typename T>
static T* dalloc(std::vector<void*>& allocs, size_t n, std::string& err) {
  void* p = nullptr;
  if (cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(T)) != cudaSuccess) {
    err = "cudaMalloc failed in preconditioner";
    return nullptr;
  }
  allocs.push_back(p);
  return (T*)p;
}

template <typename T>
static int vlev_alloc(Precond<T>& P, std::string& err) {
  P.vlev.assign(P.lev.size(), VLevel<T>{});
  for (int c = 0; c < 3; ++c) {
    P.vres0[c] = dalloc<T>(P.allocs, fsize(P.lev[0].g, c), err);
    if (!P.vres0[c]) return WSI_ERR_OOM;
  }
  for (size_t l = 1; l < P.lev.size(); ++l) {
    const GridDev& g = P.lev[l].g;
    VLevel<T>& V = P.vlev[l];
    for (int c = 0; c < 3; ++c) {
      V.rho_face[c] = dalloc<T>(P.allocs, fsize(g, c), err);
      V.u[c] = dalloc<T>(P.allocs, fsize(g, c), err);
      V.b[c] = dalloc<T>(P.allocs, fsize(g, c), err);
      V.res[c] = dalloc<T>(P.allocs, fsize(g, c), err);
      V.mu_e[c] = dalloc<T>(P.allocs, esize(g, c), err);
      if (!V.rho_face[c] || !V.u[c] || !V.b[c] || !V.res[c] || !V.mu_e[c]) return WSI_ERR_OOM;
    }
    V.mu_cc = dalloc<T>(P.allocs, fsize(g, 3), err);
    if (!V.mu_cc) return WSI_ERR_OOM;
  }
  return WSI_OK;
}

template <typename T>
int precond_alloc(Precond<T>& P, const GridDev& g0, bool visc, std::string& err) {
  precond_free(P);
  GridDev g = g0;
  for (;;) {
    MGLevel<T> L;
    L.g = g;
    for (int c = 0; c < 3; ++c) {
      L.beta[c] = dalloc<T>(P.allocs, fsize(g, c), err);
      if (!L.beta[c]) return WSI_ERR_OOM;
    }
    size_t nc = fsize(g, 3);
    L.x = dalloc<T>(P.allocs, nc, err);
    L.b = dalloc<T>(P.allocs, nc, err);
    L.res = dalloc<T>(P.allocs, nc, err);
    L.cd = dalloc<T>(P.allocs, nc, err);
    L.cx2 = dalloc<T>(P.allocs, nc, err);
    L.cd2 = dalloc<T>(P.allocs, nc, err);
    L.id = sizeof(T) == 8 ? dalloc<T>(P.allocs, nc, err) : nullptr;
    if (!L.x || !L.b || !L.res || !L.cd || !L.cx2 || !L.cd2 || (sizeof(T) == 8 && !L.id)) return WSI_ERR_OOM;
    // Semi-coarsening on anisotropic grids: an axis coarsens only while its
    // spacing is within 1.5x of the finest active spacing, so a grid with
    // hx = 2 hy = 2 hz first coarsens y and z and then all three (point
    // smoothers damp the weakly coupled direction poorly).
    double hmin = 1e300;
    for (int a = 0; a < 3; ++a)
      if (g.n[a] > 1) hmin = std::min(hmin, g.h[a]);
    bool any = false;
    for (int a = 0; a < 3; ++a) {
      L.r[a] = (g.n[a] % 2 == 0 && g.n[a] >= 4 && g.h[a] <= 1.5 * hmin) ? 2 : 1;
      any |= L.r[a] == 2;
    }
    if (!any && nc > 64) {
      // strongly anisotropic grids whose fine axes can no longer coarsen
      // (wave tanks with long cells): coarsen every axis that still can
      for (int a = 0; a < 3; ++a) {
        L.r[a] = (g.n[a] % 2 == 0 && g.n[a] >= 4) ? 2 : 1;
        any |= L.r[a] == 2;
      }
    }
    if (nc <= 64 || !any) {
      for (int a = 0; a < 3; ++a) L.r[a] = 1;
      P.lev.push_back(L);
      break;
    }
    P.lev.push_back(L);
    for (int a = 0; a < 3; ++a) {
      g.n[a] /= L.r[a];
      g.h[a] *= L.r[a];
    }
    grid_finalize(g);
  }
  P.ncoarse = (int)fsize(P.lev.back().g, 3);
  if (P.ncoarse > 1024) {
    err = "coarsest multigrid level too large (grid extents need more factors of 2)";
    return WSI_ERR_INVALID_ARG;
  }
  P.coarse_inv = dalloc<double>(P.allocs, (size_t)P.ncoarse * P.ncoarse, err);
  for (int c = 0; c < 3; ++c) {
    P.rho_face[c] = dalloc<T>(P.allocs, fsize(g0, c), err);
    P.ut[c] = dalloc<T>(P.allocs, fsize(g0, c), err);
  }
  P.mu_cc = dalloc<T>(P.allocs, fsize(g0, 3), err);
  for (int e = 0; e < 3; ++e) P.mu_e[e] = dalloc<T>(P.allocs, esize(g0, e), err);
  if (!std::is_same<T, double>::value) P.pv = dalloc<T>(P.allocs, fsize(g0, 3), err);
  if (std::is_same<T, double>::value && !visc)
    for (int c = 0; c < 3; ++c) {
      P.vd[c] = dalloc<T>(P.allocs, fsize(g0, c), err);
      if (!P.vd[c]) return WSI_ERR_OOM;
    }
  cudaFuncSetAttribute(k_coarse_inverse<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (INV_MAX + 1) * INV_MAX * (int)sizeof(double));
  // the fused lower cycle's shared memory: x and b of its small levels (each at
  // most half the cells of the one above) and the dense solve's vector
  cudaFuncSetAttribute(k_coarse_cycle<T, coarse_threads<T>()>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       4 * std::max(coarse_smem_cells<T>(), 1024) * (int)sizeof(T) + 1024 * 8);
  P.coarse_ctas = 8;
  if (cudaFuncSetAttribute(k_coarse_cycle<T, coarse_threads<T>()>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
      cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(coarse_threads<T>());
    cfg.dynamicSmemBytes = 4 * std::max(coarse_smem_cells<T>(), 1024) * (int)sizeof(T) + 1024 * 8;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 16;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, k_coarse_cycle<T, coarse_threads<T>()>, &cfg) == cudaSuccess && ncl > 0)
      P.coarse_ctas = 16;
  }
  cudaGetLastError();
  P.dscratch = dalloc<double>(P.allocs, 4096, err);
  P.dsum = dalloc<double>(P.allocs, 8, err);
  if (!P.coarse_inv || !P.mu_cc || (!P.pv && !std::is_same<T, double>::value) || !P.dscratch || !P.dsum) return WSI_ERR_OOM;
  if (visc) return vlev_alloc(P, err);
  P.vlev.assign(P.lev.size(), VLevel<T>{});
  return WSI_OK;
}

template <typename T>
void precond_free(Precond<T>& P) {
  for (void* p : P.allocs) cudaFree(p);
  P.allocs.clear();
  P.lev.clear();
  for (int c = 0; c < 3; ++c) P.vd[c] = nullptr;
  P.vd_set = false;
  P.built = false;
  P.learn.lrho.clear();
  P.learn.phi.clear();
  P.learn.diag = nullptr;
  P.learn.e = nullptr;
  P.learn.t1 = P.learn.t2 = P.learn.t3 = nullptr;
  P.learn.ss = nullptr;
  P.learn.ready = false;
}

// ------------------------------------------------------------ coefficients
template <int C, typename T>
__device__ __forceinline__ void coarsen_face(const GridDev& gf, const GridDev& gc, int r0, int r1, int r2,
                                             const T* __restrict__ bf, T* bc, int i, int j, int k) {
  if (i >= ext(gc, C, 0) || j >= ext(gc, C, 1) || k >= ext(gc, C, 2)) return;
  int r[3] = {r0, r1, r2};
  int base[3] = {i * r[0], j * r[1], k * r[2]};
  int span[3] = {r[0], r[1], r[2]};
  span[C] = 1;  // the coplanar block only
  T s = T(0);
  for (int c = 0; c < span[2]; ++c)
    for (int b = 0; b < span[1]; ++b)
      for (int a = 0; a < span[0]; ++a) s += bf[fidx(gf, C, base[0] + a, base[1] + b, base[2] + c)];
  bc[fidx(gc, C, i, j, k)] = s / T(span[0] * span[1] * span[2]);
}

// the three face arrays in one launch, one after another along blockIdx.x (y and z
// of a grid end at 65535, and the planes of one array may use all of that)
template <typename T>
__global__ void k_coarsen_faces(GridDev gf, GridDev gc, int r0, int r1, int r2, CVel<T> f, Vel<T> c) {
  const int nb = gridDim.x / 3, q = blockIdx.x / nb;
  const int i = (blockIdx.x - q * nb) * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (q == 0) coarsen_face<0, T>(gf, gc, r0, r1, r2, f.q[0], c.q[0], i, j, k);
  else if (q == 1) coarsen_face<1, T>(gf, gc, r0, r1, r2, f.q[1], c.q[1], i, j, k);
  else coarsen_face<2, T>(gf, gc, r0, r1, r2, f.q[2], c.q[2], i, j, k);
}

template <typename T>
static void coarsen_faces(const MGLevel<T>& F, const GridDev& gc, const T* const f[3], T* const c[3], cudaStream_t st) {
  const dim3 grid(3 * cdiv(gc.n[0] + 1, BX), cdiv(gc.n[1] + 1, BY), gc.n[2] + 1);
  { k_coarsen_faces<T><<<grid, dim3(BX, BY), 0, st>>>(F.g, gc, F.r[0], F.r[1], F.r[2], CVel<T>{{f[0], f[1], f[2]}},
                                                      Vel<T>{{c[0], c[1], c[2]}}); WSI_COUNT(); }
}

// coarse cell viscosity: mean of the children
template <typename T>
__global__ void k_vmu_down(GridDev gf, GridDev gc, int r0, int r1, int r2, const T* __restrict__ mf, T* mc) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= gc.n[0] || j >= gc.n[1]) return;
  T s = T(0);
  for (int c = 0; c < r2; ++c)
    for (int b = 0; b < r1; ++b)
      for (int a = 0; a < r0; ++a) s += mf[fidx(gf, 3, i * r0 + a, j * r1 + b, k * r2 + c)];
  mc[fidx(gc, 3, i, j, k)] = s / T(r0 * r1 * r2);
}

// coarse edge viscosity: harmonic mean of the four coarse cells around the
// edge (indices clamped at walls), the fine-grid rule on the coarse grid
template <int E, typename T>
__global__ void k_vedges(GridDev g, const T* __restrict__ mu, T* mu_e) {
  constexpr int A1 = (E == 2) ? 1 : 0;
  constexpr int A2 = (E == 0) ? 1 : 2;
  const int ex = g.n[0] + (A1 == 0 || A2 == 0), ey = g.n[1] + (A1 == 1 || A2 == 1);
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ex || j >= ey) return;
  T s = T(0);
  for (int o1 = 0; o1 < 2; ++o1)
    for (int o2 = 0; o2 < 2; ++o2) {
      int c[3] = {i, j, k};
      c[A1] -= o1;
      c[A2] -= o2;
      for (int a = 0; a < 3; ++a) c[a] = clampi(c[a], 0, g.n[a] - 1);
      s += T(1) / mu[fidx(g, 3, c[0], c[1], c[2])];
    }
  mu_e[eidx(g, E, i, j, k)] = T(4) / s;
}

// Face restriction of component C: full weighting (1/4, 1/2, 1/4) across the
// coarse face along C where that axis coarsens, the mean of the children
// across it; wall faces of the coarse grid are not unknowns (0)
template <int C, typename T>
__global__ void k_vrestrict(GridDev gf, GridDev gc, int r0, int r1, int r2, const T* __restrict__ rf, T* bc) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ext(gc, C, 0) || j >= ext(gc, C, 1)) return;
  const int I3[3] = {i, j, k};
  const size_t id = fidx(gc, C, i, j, k);
  if (I3[C] == 0 || I3[C] == gc.n[C]) {
    bc[id] = T(0);
    return;
  }
  const int r[3] = {r0, r1, r2};
  int span[3] = {r0, r1, r2};
  span[C] = 1;
  T s = T(0);
  for (int c = 0; c < span[2]; ++c)
    for (int b = 0; b < span[1]; ++b)
      for (int a = 0; a < span[0]; ++a) {
        int f[3] = {i * r[0] + a, j * r[1] + b, k * r[2] + c};
        if (r[C] == 2) {
          f[C] = 2 * I3[C];
          T v = T(0.5) * rf[fidx(gf, C, f[0], f[1], f[2])];
          f[C] -= 1;
          v += T(0.25) * rf[fidx(gf, C, f[0], f[1], f[2])];
          f[C] += 2;
          v += T(0.25) * rf[fidx(gf, C, f[0], f[1], f[2])];
          s += v;
        } else {
          f[C] = I3[C];
          s += rf[fidx(gf, C, f[0], f[1], f[2])];
        }
      }
  bc[id] = s / T(span[0] * span[1] * span[2]);
}

// Face prolongation of component C, added to the fine iterate: linear along
// C where that axis coarsens (coincident faces take the coarse value, the
// faces between two coarse faces their mean), constant across it
template <int C, typename T>
__global__ void k_vprolong(GridDev gf, GridDev gc, int r0, int r1, int r2, const T* __restrict__ uc, T* uf) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ext(gf, C, 0) || j >= ext(gf, C, 1)) return;
  const int i3[3] = {i, j, k};
  if (i3[C] == 0 || i3[C] == gf.n[C]) return;
  const int r[3] = {r0, r1, r2};
  int I[3];
  for (int a = 0; a < 3; ++a) I[a] = a == C ? i3[a] : i3[a] / r[a];
  T v;
  if (r[C] == 2) {
    if ((i3[C] & 1) == 0) {
      I[C] = i3[C] / 2;
      v = uc[fidx(gc, C, I[0], I[1], I[2])];
    } else {
      I[C] = (i3[C] - 1) / 2;
      v = uc[fidx(gc, C, I[0], I[1], I[2])];
      I[C] += 1;
      v = T(0.5) * (v + uc[fidx(gc, C, I[0], I[1], I[2])]);
    }
  } else {
    v = uc[fidx(gc, C, I[0], I[1], I[2])];
  }
  uf[fidx(gf, C, i, j, k)] += v;
}

// up to sixteen arrays cast in one launch (blockIdx.y selects the array)
template <typename Ts, typename Td>
struct CastSet {
  const Ts* a[16];
  Td* b[16];
  size_t n[16];
  int count;
};

template <typename Ts, typename Td>
__global__ void k_cast_set(CastSet<Ts, Td> s) {
  const int q = blockIdx.y;
  if (q >= s.count) return;
  const Ts* __restrict__ a = s.a[q];
  Td* b = s.b[q];
  const size_t n = s.n[q];
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    b[t] = cvt<Td, Ts>(a[t]);
}

template <typename Ts, typename Td>
static void cast_set(const CastSet<Ts, Td>& s, cudaStream_t st) {
  size_t nmax = 0;
  for (int q = 0; q < s.count; ++q) nmax = std::max(nmax, s.n[q]);
  if (!nmax) return;
  const int blocks = (int)std::min<size_t>((nmax + 255) / 256, 152 * 4);
  { k_cast_set<Ts, Td><<<dim3(blocks, s.count), 256, 0, st>>>(s); WSI_COUNT(); }
}

// Gauss-Jordan inverse (host, float64) of an SPD matrix, no pivoting needed
static void spd_inverse(std::vector<double>& A, int n) {
  std::vector<double> I((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i) I[(size_t)i * n + i] = 1.0;
  for (int p = 0; p < n; ++p) {
    double d = A[(size_t)p * n + p];
    double id = 1.0 / d;
    for (int c = 0; c < n; ++c) {
      A[(size_t)p * n + c] *= id;
      I[(size_t)p * n + c] *= id;
    }
    for (int r = 0; r < n; ++r) {
      if (r == p) continue;
      double f = A[(size_t)r * n + p];
      if (f == 0.0) continue;
      for (int c = 0; c < n; ++c) {
        A[(size_t)r * n + c] -= f * A[(size_t)p * n + c];
        I[(size_t)r * n + c] -= f * I[(size_t)p * n + c];
      }
    }
  }
  A.swap(I);
}

// The dense coarsest operator M = -L + c 1 1^T of the level and its inverse
// (Gauss-Jordan in place, no pivoting: M is symmetric positive definite), one
// block, the matrix in shared memory; the same operations as the host form
// below, in a launch that the host doesn't wait for (read back, inverted there and
// sent down it costs two synchronisations).  Bound by the float64 pipe of one SM and
// the chain of n pivots (a division, three barriers and n^2 multiply-adds each), so
// only what the pivots need goes to that pipe: the reciprocal by one thread (by all
// of them 73 us more at 64 cells), the test for zero on the bits, and the columns of
// a row in whole warps (unrolled by lane, the last chunk split the warp: 1140 us at
// 125 cells).  154 us at 64 cells, 757 at 125 (232 and 900 before).  A set-up and one
// cycle of 4 x 4 x 4 cells 317 us (404; inverted on the host 330), of 8^3 340 (430,
// 455), 40^3 1120 (1276, 1460), 44 x 28 x 8 1620 (1790, 1800).
template <typename T>
__global__ void __launch_bounds__(1024) k_coarse_inverse(GridDev g, const T* __restrict__ bx, const T* __restrict__ by,
                                                         const T* __restrict__ bz, int n, double* inv) {
  extern __shared__ double W[];  // n x n, then a column
  double* col = W + n * n;
  __shared__ double dmax_w[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int t = tid; t < n * n; t += 1024) W[t] = 0.0;
  __syncthreads();
  double dg = 0.0;
  for (int row = tid; row < n; row += 1024) {
    const int i = row % g.n[0], j = row / g.n[0] % g.n[1], k = row / (g.n[0] * g.n[1]);
    const int c3[3] = {i, j, k}, sd[3] = {1, g.n[0], g.n[0] * g.n[1]};
    double d = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T* b = a == 0 ? bx : (a == 1 ? by : bz);
      const double ih2 = 1.0 / (g.h[a] * g.h[a]);
      const double hi = (double)b[fidx(g, a, i + (a == 0), j + (a == 1), k + (a == 2))];
      if (c3[a] + 1 < g.n[a]) {
        W[row * n + row + sd[a]] -= hi * ih2;
        d += hi * ih2;
      }
      if (c3[a] > 0) {
        const double lo = (double)b[fidx(g, a, i, j, k)];
        W[row * n + row - sd[a]] -= lo * ih2;
        d += lo * ih2;
      }
      if (a == 2 && k + 1 == g.n[2] && g.open_top) d += 2.0 * hi * ih2;  // p = 0 on the open top: ghost -p
    }
    W[row * n + row] = d;
    dg = d;
  }
  for (int o = 16; o > 0; o >>= 1) dg = fmax(dg, __shfl_xor_sync(0xffffffffu, dg, o));
  if (lane == 0) dmax_w[warp] = dg;
  __syncthreads();
  double dmax = 0.0;
  for (int w = 0; w < 32; ++w) dmax = fmax(dmax, dmax_w[w]);
  const double creg = g.open_top ? 0.0 : dmax / n;
  for (int t = tid; t < n * n; t += 1024) W[t] += creg;
  __shared__ double rpiv;  // reciprocal of the pivot
  for (int p = 0; p < n; ++p) {
    __syncthreads();
    if (tid < n) col[tid] = W[tid * n + p];
    if (tid == 1023) rpiv = 1.0 / W[p * n + p];  // (a warp of its own)
    __syncthreads();
    if (tid < n) W[p * n + tid] = tid == p ? rpiv : W[p * n + tid] * rpiv;
    __syncthreads();
    for (int r = warp; r < n; r += 32) {
      const double f = col[r];
      if (r == p || (__double_as_longlong(f) << 1) == 0) continue;
      for (int c0 = 0; c0 < n; c0 += 32) {
        const int c = c0 + lane;
        if (c < n) W[r * n + c] = fma(-f, W[p * n + c], c == p ? 0.0 : W[r * n + c]);
      }
    }
  }
  __syncthreads();
  for (int t = tid; t < n * n; t += 1024) inv[t] = W[t];
}

template <typename T>
int precond_setup(Precond<T>& P, const GridDev& g, const Coef<double>& fine, bool visc, bool beta_only,
                  cudaStream_t st, std::string& err) {
  // fine coefficients in T (one launch for the arrays)
  {
    CastSet<double, T> cs;
    cs.count = 0;
    auto add = [&](const double* a, T* b, size_t n) {
      cs.a[cs.count] = a;
      cs.b[cs.count] = b;
      cs.n[cs.count] = n;
      ++cs.count;
    };
    for (int c = 0; c < 3; ++c) {
      if (!beta_only) add(fine.rho_face[c], P.rho_face[c], fsize(g, c));
      add(fine.beta[c], P.lev[0].beta[c], fsize(g, c));
    }
    if (!beta_only) {
      add(fine.mu_cc, P.mu_cc, fsize(g, 3));
      for (int e = 0; e < 3; ++e) add(fine.mu_e[e], P.mu_e[e], esize(g, e));
    }
    cast_set(cs, st);
  }
  for (size_t l = 0; l + 1 < P.lev.size(); ++l) {
    MGLevel<T>& F = P.lev[l];
    MGLevel<T>& Cl = P.lev[l + 1];
    const GridDev& gc = Cl.g;
    const T* bf[3] = {F.beta[0], F.beta[1], F.beta[2]};
    coarsen_faces<T>(F, gc, bf, Cl.beta, st);
    if (!visc) continue;  // the viscous hierarchy is used by viscous V-cycles only
    // viscous coefficients: face density like beta (coplanar mean), cell
    // viscosity the mean of the children, edge viscosity harmonic again
    const T* rf[3] = {l == 0 ? P.rho_face[0] : P.vlev[l].rho_face[0], l == 0 ? P.rho_face[1] : P.vlev[l].rho_face[1],
                      l == 0 ? P.rho_face[2] : P.vlev[l].rho_face[2]};
    const T* mf = l == 0 ? P.mu_cc : P.vlev[l].mu_cc;
    VLevel<T>& VC = P.vlev[l + 1];
    coarsen_faces<T>(F, gc, rf, VC.rho_face, st);
    { k_vmu_down<T><<<grid3(gc.n[0], gc.n[1], gc.n[2]), dim3(BX, BY), 0, st>>>(F.g, gc, F.r[0], F.r[1], F.r[2], mf,
                                                                             VC.mu_cc); WSI_COUNT(); }
    { k_vedges<0, T><<<grid3(gc.n[0] + 1, gc.n[1] + 1, gc.n[2]), dim3(BX, BY), 0, st>>>(gc, VC.mu_cc, VC.mu_e[0]); WSI_COUNT(); }
    { k_vedges<1, T><<<grid3(gc.n[0] + 1, gc.n[1], gc.n[2] + 1), dim3(BX, BY), 0, st>>>(gc, VC.mu_cc, VC.mu_e[1]); WSI_COUNT(); }
    { k_vedges<2, T><<<grid3(gc.n[0], gc.n[1] + 1, gc.n[2] + 1), dim3(BX, BY), 0, st>>>(gc, VC.mu_cc, VC.mu_e[2]); WSI_COUNT(); }
  }
  inv_diag_levels(P.lev, st);
  P.vd_set = false;
  // dense coarsest operator: M = -L + c 1 1^T (SPD), inverted in float64
  const MGLevel<T>& Lc = P.lev.back();
  const GridDev& gc = Lc.g;
  int n = P.ncoarse;
  if (n <= INV_MAX) {
    { k_coarse_inverse<T><<<1, 1024, (size_t)(n + 1) * n * sizeof(double), st>>>(gc, Lc.beta[0], Lc.beta[1], Lc.beta[2], n,
                                                                              P.coarse_inv); WSI_COUNT(); }
    P.built = true;
    return WSI_OK;
  }
  std::vector<T> hb[3];
  for (int c = 0; c < 3; ++c) {
    hb[c].resize(fsize(gc, c));
    cudaMemcpyAsync(hb[c].data(), Lc.beta[c], fsize(gc, c) * sizeof(T), cudaMemcpyDeviceToHost, st);
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) {
    err = "CUDA error while building the coarse operator";
    return WSI_ERR_CUDA;
  }
  std::vector<double> M((size_t)n * n, 0.0);
  double dmax = 0.0;
  for (int k = 0; k < gc.n[2]; ++k)
    for (int j = 0; j < gc.n[1]; ++j)
      for (int i = 0; i < gc.n[0]; ++i) {
        int row = (int)fidx(gc, 3, i, j, k);
        int c3[3] = {i, j, k};
        for (int a = 0; a < 3; ++a) {
          double ih2 = 1.0 / (gc.h[a] * gc.h[a]);
          // face hi
          if (c3[a] + 1 < gc.n[a]) {
            int f3[3] = {i, j, k};
            f3[a] += 1;
            double b = (double)hb[a][fidx(gc, a, f3[0], f3[1], f3[2])] * ih2;
            int nb3[3] = {i, j, k};
            nb3[a] += 1;
            int col = (int)fidx(gc, 3, nb3[0], nb3[1], nb3[2]);
            M[(size_t)row * n + col] -= b;
            M[(size_t)row * n + row] += b;
          }
          if (c3[a] > 0) {
            double b = (double)hb[a][fidx(gc, a, i, j, k)] * ih2;
            int nb3[3] = {i, j, k};
            nb3[a] -= 1;
            int col = (int)fidx(gc, 3, nb3[0], nb3[1], nb3[2]);
            M[(size_t)row * n + col] -= b;
            M[(size_t)row * n + row] += b;
          }
          if (a == 2 && k + 1 == gc.n[2] && gc.open_top)  // p = 0 on the open top: ghost -p
            M[(size_t)row * n + row] += 2.0 * (double)hb[2][fidx(gc, 2, i, j, k + 1)] * ih2;
        }
        dmax = std::max(dmax, M[(size_t)row * n + row]);
      }
  // a closed box leaves constants in the null space: M = -L + c 1 1^T is SPD
  // and its inverse gives the mean-free solution; with an open top -L is SPD
  const double creg = gc.open_top ? 0.0 : dmax / n;
  for (size_t t = 0; t < M.size(); ++t) M[t] += creg;
  spd_inverse(M, n);
  cudaMemcpyAsync(P.coarse_inv, M.data(), M.size() * sizeof(double), cudaMemcpyHostToDevice, st);
  if (cudaStreamSynchronize(st) != cudaSuccess) {
    err = "CUDA error in preconditioner setup";
    return WSI_ERR_CUDA;
  }
  P.built = true;
  return WSI_OK;
}

// ------------------------------------------------------------ V-cycle kernels
static inline dim3 grid_rb(const GridDev& g) { return dim3(cdiv(cdiv(g.n[0], 2), BX), cdiv(g.n[1], BY), g.n[2]); }

// The pressure operator of one level as the smoothing kernels use it
template <typename T>
struct PLevel {
  int n[3], open_top;
  T ih2[3];
  const T *bx, *by, *bz, *b;
  const T* id;  // float64: the inverse diagonal (0: a cell without any face)
};

template <typename T>
static PLevel<T> plevel(const MGLevel<T>& L) {
  PLevel<T> p;
  for (int a = 0; a < 3; ++a) {
    p.n[a] = L.g.n[a];
    p.ih2[a] = ginv2<T>(L.g, a);
  }
  p.open_top = L.g.open_top;
  p.bx = L.beta[0];
  p.by = L.beta[1];
  p.bz = L.beta[2];
  p.b = L.b;
  p.id = L.id;
  return p;
}

// face coefficients around cell (i, j, k); those of walls are not used
template <typename T>
struct Faces {
  T xh, xl, yh, yl, zh, zl;
};
template <typename T>
__device__ __forceinline__ Faces<T> load_faces(const PLevel<T>& p, int i, int j, int k) {
  const int r = k * p.n[1] + j, ox = r * (p.n[0] + 1) + i, oy = (r + k) * p.n[0] + i, oz = r * p.n[0] + i;
  Faces<T> f{p.bx[ox + 1], p.bx[ox], p.by[oy + p.n[0]], p.by[oy], T(0), T(0)};
  if (k + 1 < p.n[2] || p.open_top) f.zh = p.bz[oz + p.n[0] * p.n[1]];  // (a 2-D grid reads neither)
  if (k > 0) f.zl = p.bz[oz];
  return f;
}

// Gauss-Seidel value of cell (i, j, k): x(di, dj, dk) returns the neighbours;
// a cell without any face keeps x(0, 0, 0).  In float64 the pipe bounds the
// update (29 operations with the diagonal and its division: 11 with the inverse
// diagonal from memory and one weight per axis; 9.8 -> 5.8 us per half sweep,
// the mean over the levels of 128 x 64 x 64).
template <typename T, typename X>
__device__ __forceinline__ T gs_value(const PLevel<T>& p, const Faces<T>& f, int i, int j, int k, T b, T id, X x) {
  if constexpr (sizeof(T) == 8) {
    T sx = T(0), sy = T(0), sz = T(0);
    if (i + 1 < p.n[0]) sx = f.xh * x(1, 0, 0);
    if (i > 0) sx = fma(f.xl, x(-1, 0, 0), sx);
    if (j + 1 < p.n[1]) sy = f.yh * x(0, 1, 0);
    if (j > 0) sy = fma(f.yl, x(0, -1, 0), sy);
    if (k + 1 < p.n[2]) sz = f.zh * x(0, 0, 1);
    if (k > 0) sz = fma(f.zl, x(0, 0, -1), sz);
    const T s = fma(sx, p.ih2[0], fma(sy, p.ih2[1], fma(sz, p.ih2[2], -b)));
    return __double_as_longlong(id) == 0 ? x(0, 0, 0) : s * id;
  }
  T s = T(0), d = T(0);
  if (i + 1 < p.n[0]) { T c = f.xh * p.ih2[0]; s += c * x(1, 0, 0); d += c; }
  if (i > 0) { T c = f.xl * p.ih2[0]; s += c * x(-1, 0, 0); d += c; }
  if (j + 1 < p.n[1]) { T c = f.yh * p.ih2[1]; s += c * x(0, 1, 0); d += c; }
  if (j > 0) { T c = f.yl * p.ih2[1]; s += c * x(0, -1, 0); d += c; }
  if (k + 1 < p.n[2]) { T c = f.zh * p.ih2[2]; s += c * x(0, 0, 1); d += c; }
  else if (p.open_top) d += T(2) * f.zh * p.ih2[2];  // ghost -x above the open top
  if (k > 0) { T c = f.zl * p.ih2[2]; s += c * x(0, 0, -1); d += c; }
  if (d > T(0)) return (s - b) / d;
  return x(0, 0, 0);
}

template <typename T>
__device__ __forceinline__ T inv_diag(const PLevel<T>& p, int id) {
  if constexpr (sizeof(T) == 8) return p.id[id];
  else return T(0);
}

// the inverse diagonals of all levels in one launch
static constexpr int DIAG_LEVELS = 24;
struct DiagLevels {
  PLevel<double> p[DIAG_LEVELS];
  double* out[DIAG_LEVELS];
};
__global__ void k_inv_diag(const __grid_constant__ DiagLevels d) {
  const PLevel<double>& p = d.p[blockIdx.y];
  const int n = p.n[0] * p.n[1] * p.n[2];
  for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < n; id += gridDim.x * blockDim.x) {
    const int r = id / p.n[0], i = id - r * p.n[0], k = r / p.n[1], j = r - k * p.n[1];
    const Faces<double> f = load_faces<double>(p, i, j, k);
    double s = 0.0;
    if (i + 1 < p.n[0]) s += f.xh * p.ih2[0];
    if (i > 0) s += f.xl * p.ih2[0];
    if (j + 1 < p.n[1]) s += f.yh * p.ih2[1];
    if (j > 0) s += f.yl * p.ih2[1];
    if (k + 1 < p.n[2]) s += f.zh * p.ih2[2];
    else if (p.open_top) s += 2.0 * f.zh * p.ih2[2];
    if (k > 0) s += f.zl * p.ih2[2];
    d.out[blockIdx.y][id] = s > 0.0 ? 1.0 / s : 0.0;
  }
}
static void inv_diag_levels(const std::vector<MGLevel<double>>& lev, cudaStream_t st) {
  for (size_t l0 = 0; l0 < lev.size(); l0 += DIAG_LEVELS) {
    DiagLevels d;
    const int m = (int)std::min<size_t>(lev.size() - l0, DIAG_LEVELS);
    for (int l = 0; l < m; ++l) {
      d.p[l] = plevel(lev[l0 + l]);
      d.out[l] = lev[l0 + l].id;
    }
    const size_t n = fsize(lev[l0].g, 3);
    { k_inv_diag<<<dim3((unsigned)std::min<size_t>((n + 255) / 256, 152 * 8), m), 256, 0, st>>>(d); WSI_COUNT(); }
  }
}
static void inv_diag_levels(const std::vector<MGLevel<float>>&, cudaStream_t) {}

// L x at cell (i, j, k), x as above
template <typename T, typename X>
__device__ __forceinline__ T lap_value(const PLevel<T>& p, const Faces<T>& f, int i, int j, int k, X x) {
  const T xc = x(0, 0, 0);
  T s = T(0);
  if constexpr (sizeof(T) == 8) {  // one weight per axis: 15 operations instead of 18
    T sx = T(0), sy = T(0), sz = T(0);
    if (i + 1 < p.n[0]) sx = f.xh * (x(1, 0, 0) - xc);
    if (i > 0) sx = fma(f.xl, x(-1, 0, 0) - xc, sx);
    if (j + 1 < p.n[1]) sy = f.yh * (x(0, 1, 0) - xc);
    if (j > 0) sy = fma(f.yl, x(0, -1, 0) - xc, sy);
    if (k + 1 < p.n[2]) sz = f.zh * (x(0, 0, 1) - xc);
    else if (p.open_top) sz = T(-2) * f.zh * xc;
    if (k > 0) sz = fma(f.zl, x(0, 0, -1) - xc, sz);
    return fma(sx, p.ih2[0], fma(sy, p.ih2[1], sz * p.ih2[2]));
  }
  if (i + 1 < p.n[0]) s += f.xh * (x(1, 0, 0) - xc) * p.ih2[0];
  if (i > 0) s -= f.xl * (xc - x(-1, 0, 0)) * p.ih2[0];
  if (j + 1 < p.n[1]) s += f.yh * (x(0, 1, 0) - xc) * p.ih2[1];
  if (j > 0) s -= f.yl * (xc - x(0, -1, 0)) * p.ih2[1];
  if (k + 1 < p.n[2]) s += f.zh * (x(0, 0, 1) - xc) * p.ih2[2];
  else if (p.open_top) s -= T(2) * f.zh * xc * p.ih2[2];
  if (k > 0) s -= f.zl * (xc - x(0, 0, -1)) * p.ih2[2];
  return s;
}

// prolongation (linear in cell centres along coarsened axes) at fine cell
// (i, j, k): xc(I, J, K) returns the coarse values; m: the coarse extents
template <typename T, typename X>
__device__ __forceinline__ T prolong_value(const int r[3], const int m[3], int i, int j, int k, X xc) {
  const int f3[3] = {i, j, k};
  int c0[3], c1[3];
  T w0[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (r[a] == 2) {
      c0[a] = f3[a] >> 1;
      int nb = (f3[a] & 1) ? c0[a] + 1 : c0[a] - 1;
      c1[a] = clampi(nb, 0, m[a] - 1);
      w0[a] = T(0.75);
    } else {
      c0[a] = f3[a];
      c1[a] = f3[a];
      w0[a] = T(1);
    }
  }
  if (r[0] == 2 && r[1] == 2 && r[2] == 2) {  // the weights' products as constants
    T v = T(0);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int cx = m & 1, cy = (m >> 1) & 1, cz = m >> 2, e = cx + cy + cz;
      v += T(e == 0 ? 27.0 / 64 : (e == 1 ? 9.0 / 64 : (e == 2 ? 3.0 / 64 : 1.0 / 64))) *
           xc(cx ? c1[0] : c0[0], cy ? c1[1] : c0[1], cz ? c1[2] : c0[2]);
    }
    return v;
  }
  T s = T(0);
#pragma unroll
  for (int cz = 0; cz < 2; ++cz)
#pragma unroll
    for (int cy = 0; cy < 2; ++cy)
#pragma unroll
      for (int cx = 0; cx < 2; ++cx) {
        T wx = cx ? T(1) - w0[0] : w0[0];
        T wy = cy ? T(1) - w0[1] : w0[1];
        T wz = cz ? T(1) - w0[2] : w0[2];
        T w = wx * wy * wz;
        if (w == T(0)) continue;
        int a = cx ? c1[0] : c0[0], b = cy ? c1[1] : c0[1], c = cz ? c1[2] : c0[2];
        s += w * xc(a, b, c);
      }
  return s;
}

// one colour of a red-black Gauss-Seidel sweep: thread t of a row owns the
// t-th cell of that colour, i = 2t + ((j + k + color) & 1)
template <typename T>
__global__ void k_rbgs_p(PLevel<T> p, T* x, int color) {
  const int j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  const int i = 2 * (blockIdx.x * BX + threadIdx.x) + ((j + k + color) & 1);
  if (i >= p.n[0] || j >= p.n[1]) return;
  const int id = (k * p.n[1] + j) * p.n[0] + i, pl = p.n[0] * p.n[1];
  x[id] = gs_value<T>(p, load_faces<T>(p, i, j, k), i, j, k, p.b[id], inv_diag(p, id),
                      [&](int a, int b, int c) { return x[id + a + b * p.n[0] + c * pl]; });
}

// Four neighbouring cells at a time (rows of a multiple of four cells, so that
// every row of a cell or y/z-face array starts on a 16-byte boundary; x-face
// rows have one element more and are read one by one).  float32 only, as the three
// kernels that use them: in float64 the pipe bounds an update, and two in a row per
// thread cost 5 % more.
struct Quad {
  float v[4];
};
__device__ __forceinline__ Quad load4(const float* a) {
  const float4 f = *reinterpret_cast<const float4*>(a);
  return Quad{{f.x, f.y, f.z, f.w}};
}
__device__ __forceinline__ void store4(float* a, const Quad& q) {
  *reinterpret_cast<float4*>(a) = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
}

// One colour of a red-black sweep, four cells (two of the colour) per thread:
// 15 loads for two updates instead of 28, and whole sectors written (the other
// colour's values go back as they were read).  ZERO: x is zero on entry and not
// read.  HBM-bound: x, b and the three coefficient arrays stream once per half
// sweep, 24 bytes per cell; at 256^3 58.6 us, 6.9 TB/s (one cell per
// thread, 64-bit indices: 98 us).
template <bool ZERO>
__global__ void __launch_bounds__(256) k_rbgs_p4(PLevel<float> p, float* x, int color) {
  const int nx = p.n[0], ny = p.n[1], nz = p.n[2], nq = nx >> 2;
  const int t = blockIdx.x * 256 + threadIdx.x, k = blockIdx.y;
  const int j = t / nq;
  if (j >= ny) return;
  const int i0 = 4 * (t - j * nq), pl = nx * ny;
  const int r = k * ny + j, id = r * nx + i0, oy = id + k * nx, ox = id + r;
  const int q = (j + k + color) & 1;  // cells i0 + q and i0 + q + 2
  const Quad b = load4(p.b + id);
  Quad xc, xyl, xyh, xzl, xzh, yl, yh, zl, zh;
  float xe = 0.0f, fx[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) fx[a] = p.bx[ox + q + a];
  yl = load4(p.by + oy);
  yh = load4(p.by + oy + nx);
  zl = load4(p.bz + id);
  zh = load4(p.bz + id + pl);
  if (!ZERO) {
    xc = load4(x + id);
    if (j > 0) xyl = load4(x + id - nx);
    if (j + 1 < ny) xyh = load4(x + id + nx);
    if (k > 0) xzl = load4(x + id - pl);
    if (k + 1 < nz) xzh = load4(x + id + pl);
    if (q ? i0 + 4 < nx : i0 > 0) xe = q ? x[id + 4] : x[id - 1];
  } else {
#pragma unroll
    for (int a = 0; a < 4; ++a) xc.v[a] = 0.0f;
  }
  auto update = [&](auto QC) {
    constexpr int Q = decltype(QC)::value;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = Q + 2 * h;  // place in the quad
      const Faces<float> f{fx[2 * h + 1], fx[2 * h], yh.v[m], yl.v[m], zh.v[m], zl.v[m]};
      xc.v[m] = gs_value<float>(p, f, i0 + m, j, k, b.v[m], 0.0f, [&](int a, int c, int d) {
        if (ZERO) return 0.0f;
        if (a == 1) return m == 3 ? xe : xc.v[m < 3 ? m + 1 : 3];
        if (a == -1) return m == 0 ? xe : xc.v[m > 0 ? m - 1 : 0];
        if (c == 1) return xyh.v[m];
        if (c == -1) return xyl.v[m];
        if (d == 1) return xzh.v[m];
        if (d == -1) return xzl.v[m];
        return xc.v[m];
      });
    }
  };
  if (q) update(std::integral_constant<int, 1>{});
  else update(std::integral_constant<int, 0>{});
  store4(x + id, xc);
}

// 1 / (r0 r1 r2), each 1 or 2 (no division)
template <typename T>
__device__ __forceinline__ T mean_scale(int r0, int r1, int r2) {
  const int e = (r0 >> 1) + (r1 >> 1) + (r2 >> 1);
  return e == 0 ? T(1) : (e == 1 ? T(0.5) : (e == 2 ? T(0.25) : T(0.125)));
}

// coarse b = mean over children of (b - L x) on the fine grid
template <typename T>
__global__ void k_restrict_res(PLevel<T> p, int m0, int m1, int r0, int r1, int r2, const T* __restrict__ x,
                               T* bcoarse) {
  int I = blockIdx.x * BX + threadIdx.x, J = blockIdx.y * BY + threadIdx.y, K = blockIdx.z;
  if (I >= m0 || J >= m1) return;
  const int pl = p.n[0] * p.n[1];
  T s = T(0);
  for (int c = 0; c < r2; ++c)
    for (int bb = 0; bb < r1; ++bb)
      for (int a = 0; a < r0; ++a) {
        const int i = I * r0 + a, j = J * r1 + bb, k = K * r2 + c, id = (k * p.n[1] + j) * p.n[0] + i;
        s += p.b[id] - lap_value<T>(p, load_faces<T>(p, i, j, k), i, j, k,
                                    [&](int da, int db, int dc) { return x[id + da + db * p.n[0] + dc * pl]; });
      }
  bcoarse[(K * m1 + J) * m0 + I] = s * mean_scale<T>(r0, r1, r2);
}

// x_fine += P x_coarse
template <typename T>
__global__ void k_prolong_add(GridDev gf, GridDev gc, int r0, int r1, int r2, const T* __restrict__ xc, T* xf) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= gf.n[0] || j >= gf.n[1]) return;
  const int r[3] = {r0, r1, r2};
  xf[fidx(gf, 3, i, j, k)] +=
      prolong_value<T>(r, gc.n, i, j, k, [&](int a, int b, int c) { return xc[fidx(gc, 3, a, b, c)]; });
}

// The same with every axis coarsened, two coarse cells (a fine quad of 2 x 2
// rows) per thread: 56 loads for 16 fine cells instead of 224 (84 -> 56 us at
// 256^3).
__global__ void __launch_bounds__(128) k_restrict_res4(PLevel<float> p, const float* __restrict__ x, float* bcoarse) {
  const int nx = p.n[0], ny = p.n[1], nz = p.n[2], nq = nx >> 2, m1 = ny >> 1;
  const int t = blockIdx.x * 128 + threadIdx.x, K = blockIdx.y;
  const int J = t / nq;
  if (J >= m1) return;
  const int i0 = 4 * (t - J * nq), j0 = 2 * J, k0 = 2 * K, pl = nx * ny;
  float s[2] = {0.0f, 0.0f};
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int k = k0 + c;
    Quad xr[4];  // rows j0 - 1 .. j0 + 2
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int j = j0 - 1 + a;
      if (j >= 0 && j < ny) xr[a] = load4(x + (k * ny + j) * nx + i0);
    }
    Quad fy[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) fy[a] = load4(p.by + (k * (ny + 1) + j0 + a) * nx + i0);
#pragma unroll
    for (int bb = 0; bb < 2; ++bb) {
      const int j = j0 + bb, r = k * ny + j, id = r * nx + i0;
      const Quad b = load4(p.b + id), zl = load4(p.bz + id), zh = load4(p.bz + id + pl);
      Quad xzl, xzh;
      if (k > 0) xzl = load4(x + id - pl);
      if (k + 1 < nz) xzh = load4(x + id + pl);
      const float xm = i0 > 0 ? x[id - 1] : 0.0f, xp = i0 + 4 < nx ? x[id + 4] : 0.0f;
      float fx[5];
#pragma unroll
      for (int a = 0; a < 5; ++a) fx[a] = p.bx[id + r + a];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const Faces<float> f{fx[m + 1], fx[m], fy[bb + 1].v[m], fy[bb].v[m], zh.v[m], zl.v[m]};
        s[m >> 1] += b.v[m] - lap_value<float>(p, f, i0 + m, j, k, [&](int da, int db, int dc) {
          if (da == 1) return m == 3 ? xp : xr[bb + 1].v[m < 3 ? m + 1 : 3];
          if (da == -1) return m == 0 ? xm : xr[bb + 1].v[m > 0 ? m - 1 : 0];
          if (db == 1) return xr[bb + 2].v[m];
          if (db == -1) return xr[bb].v[m];
          if (dc == 1) return xzh.v[m];
          if (dc == -1) return xzl.v[m];
          return xr[bb + 1].v[m];
        });
      }
    }
  }
  const int o = (K * m1 + J) * (nx >> 1) + (i0 >> 1);
  bcoarse[o] = s[0] / 8.0f;
  bcoarse[o + 1] = s[1] / 8.0f;
}

// x_fine += P x_coarse with every axis coarsened, four fine cells per thread
// (16 coarse loads instead of 32; 149 -> 44 us per cycle over all levels at 256^3)
__global__ void __launch_bounds__(256) k_prolong_add4(int nx, int ny, int m2, const float* __restrict__ xc, float* xf) {
  const int nq = nx >> 2, t = blockIdx.x * 256 + threadIdx.x, k = blockIdx.y, j = t / nq;
  if (j >= ny) return;
  const int i0 = 4 * (t - j * nq), mx = nx >> 1, my = ny >> 1;
  const int I0 = i0 >> 1, J0 = j >> 1, K0 = k >> 1;
  const int J1 = clampi((j & 1) ? J0 + 1 : J0 - 1, 0, my - 1), K1 = clampi((k & 1) ? K0 + 1 : K0 - 1, 0, m2 - 1);
  const int Im = max(I0 - 1, 0), Ip = min(I0 + 2, mx - 1);
  const int id = (k * ny + j) * nx + i0;
  Quad f = load4(xf + id), s;
#pragma unroll
  for (int m = 0; m < 4; ++m) s.v[m] = 0.0f;
#pragma unroll
  for (int cz = 0; cz < 2; ++cz)
#pragma unroll
    for (int cy = 0; cy < 2; ++cy) {
      const float* row = xc + ((cz ? K1 : K0) * my + (cy ? J1 : J0)) * mx;
      const float a[4] = {row[Im], row[I0], row[I0 + 1], row[Ip]};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float wyz = (cy ? 0.25f : 0.75f) * (cz ? 0.25f : 0.75f);
        s.v[m] += 0.75f * wyz * a[1 + (m >> 1)];
        s.v[m] += 0.25f * wyz * a[(m & 1) ? 2 + (m >> 1) : (m >> 1)];
      }
    }
#pragma unroll
  for (int m = 0; m < 4; ++m) f.v[m] += s.v[m];
  store4(xf + id, f);
}

// x = Minv (-b), one block
template <typename T>
__global__ void k_coarse_solve(int n, const double* __restrict__ Minv, const T* __restrict__ b, T* x) {
  extern __shared__ double sb[];
  for (int t = threadIdx.x; t < n; t += blockDim.x) sb[t] = -(double)b[t];
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    double s = 0.0;
    for (int c = 0; c < n; ++c) s += Minv[(size_t)r * n + c] * sb[c];
    x[r] = (T)s;
  }
}

// The lower part of a V-cycle in one launch: every level from the first one of
// at most coarse_max_cells down to the coarsest, pre-smoothing, restriction, the
// dense solve, prolongation and post-smoothing, the same operations in the same
// order as a launch each.  Levels of more than coarse_smem_cells are worked on
// by a cluster of sixteen blocks (eight where the device holds no more) in global memory (x and the restricted b through
// L2, a cluster barrier between half sweeps); the smaller ones by its first
// block with x and b in shared memory.  A launch per half sweep costs 2.5 to 4 us
// on these levels whatever their size (11 launches per level): a cycle
// over 40x32x48 cells 95 us instead of about 170, the levels of 32^3 and below of
// a 256^3 cycle 67 us instead of about 95.  Bound by latency: an exchange through
// L2 and a cluster barrier per half sweep.  Above 65536 cells the whole GPU's
// bandwidth wins.
static constexpr int COARSE_LEVELS = 14;

// quotient by a level extent: exact for t, d <= 65536
struct FastDiv {
  unsigned m;
  int d;
  void set(int v) {
    d = v;
    m = v > 1 ? (unsigned)(((1ull << 32) + v - 1) / v) : 0u;
  }
  __device__ __forceinline__ int div(int t) const { return d > 1 ? (int)__umulhi((unsigned)t, m) : t; }
};
struct LevelDiv {
  FastDiv hx, nx, ny;  // cells of one colour per row, cells per row, rows per plane
};

template <typename T>
struct CoarseCycle {
  PLevel<T> lev[COARSE_LEVELS];
  T* x[COARSE_LEVELS];
  T* b[COARSE_LEVELS];
  int r[COARSE_LEVELS][3];
  LevelDiv dv[COARSE_LEVELS];
  int off[COARSE_LEVELS];  // place of the level's x in shared memory (its b follows)
  int nl, first;           // levels, first one in shared memory
  int pre, post, zero, ncoarse, nb;  // nb: doubles before the levels in shared memory
  const double* minv;
};

template <typename T>
struct GlobalX {  // written by other blocks: through L2
  T* p;
  __device__ __forceinline__ T get(int i) const { return __ldcg(p + i); }
  __device__ __forceinline__ void set(int i, T v) const { __stcg(p + i, v); }
};
template <typename T>
struct SharedX {
  T* p;
  __device__ __forceinline__ T get(int i) const { return p[i]; }
  __device__ __forceinline__ void set(int i, T v) const { p[i] = v; }
};

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// x around a cell, loaded before any of it is used (beyond walls: the cell's
// own value, which is not used)
template <typename T>
struct Around {
  T c, xh, xl, yh, yl, zh, zl;
  __device__ __forceinline__ T operator()(int a, int b, int d) const {
    return a == 1 ? xh : (a == -1 ? xl : (b == 1 ? yh : (b == -1 ? yl : (d == 1 ? zh : (d == -1 ? zl : c)))));
  }
};
template <typename T, typename X>
__device__ __forceinline__ Around<T> load_around(const PLevel<T>& p, X x, int i, int j, int k, int id) {
  const int nx = p.n[0], pl = nx * p.n[1];
  return Around<T>{x.get(id),
                   x.get(i + 1 < nx ? id + 1 : id),
                   x.get(i > 0 ? id - 1 : id),
                   x.get(j + 1 < p.n[1] ? id + nx : id),
                   x.get(j > 0 ? id - nx : id),
                   x.get(k + 1 < p.n[2] ? id + pl : id),
                   x.get(k > 0 ? id - pl : id)};
}

// zero: 0 x as stored; 1 x = 0 everywhere; 2 x = 0 on this colour
template <typename T, typename X, typename B>
__device__ __forceinline__ void coarse_half(const PLevel<T>& p, const LevelDiv& dv, X x, B b, int color, int zero,
                                            int t0, int nt) {
  const int nx = p.n[0], ny = p.n[1], hx = (nx + 1) >> 1, total = hx * ny * p.n[2];
#pragma unroll 2
  for (int t = t0; t < total; t += nt) {
    const int rr = dv.hx.div(t), k = dv.ny.div(rr), j = rr - k * ny;
    const int i = 2 * (t - rr * hx) + ((j + k + color) & 1), id = rr * nx + i;
    if (i < nx) {
      const Faces<T> f = load_faces<T>(p, i, j, k);
      const T bv = b.get(id);
      Around<T> n{T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
      if (zero != 1) {
        n = load_around<T>(p, x, i, j, k, id);
        if (zero) n.c = T(0);
      }
      x.set(id, gs_value<T>(p, f, i, j, k, bv, inv_diag(p, id), n));
    }
  }
}

template <typename T, typename X, typename B, typename BC>
__device__ __forceinline__ void coarse_restrict(const PLevel<T>& p, const int r[3], const int m[3], const LevelDiv& dm,
                                                X x, B b, BC bc, int t0, int nt) {
  const int nx = p.n[0], ny = p.n[1];
  for (int t = t0; t < m[0] * m[1] * m[2]; t += nt) {
    const int rr = dm.nx.div(t), K = dm.ny.div(rr), J = rr - K * m[1], I = t - rr * m[0];
    T s = T(0);
    for (int c = 0; c < r[2]; ++c)
      for (int bb = 0; bb < r[1]; ++bb) {
        const int i = I * r[0], j = J * r[1] + bb, k = K * r[2] + c, id = (k * ny + j) * nx + i;
        const bool two = r[0] == 2;
        const Faces<T> f0 = load_faces<T>(p, i, j, k);
        const Around<T> n0 = load_around<T>(p, x, i, j, k, id);
        const T b0 = b.get(id);
        Faces<T> f1;
        Around<T> n1;
        T b1 = T(0);
        if (two) {
          f1 = load_faces<T>(p, i + 1, j, k);
          n1 = load_around<T>(p, x, i + 1, j, k, id + 1);
          b1 = b.get(id + 1);
        }
        s += b0 - lap_value<T>(p, f0, i, j, k, n0);
        if (two) s += b1 - lap_value<T>(p, f1, i + 1, j, k, n1);
      }
    bc.set(t, s * mean_scale<T>(r[0], r[1], r[2]));
  }
}

template <typename T, typename X, typename XC>
__device__ __forceinline__ void coarse_prolong(const PLevel<T>& p, const LevelDiv& dv, const int r[3], const int m[3],
                                               X x, XC xc, int t0, int nt) {
  const int nx = p.n[0], ny = p.n[1];
  for (int t = t0; t < nx * ny * p.n[2]; t += nt) {
    const int rr = dv.nx.div(t), k = dv.ny.div(rr), j = rr - k * ny, i = t - rr * nx;
    x.set(t, x.get(t) + prolong_value<T>(r, m, i, j, k, [&](int a, int b, int c) { return xc.get((c * m[1] + b) * m[0] + a); }));
  }
}

template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_coarse_cycle(const __grid_constant__ CoarseCycle<T> c) {
  extern __shared__ __align__(16) double coarse_smem[];
  T* const sm = reinterpret_cast<T*>(coarse_smem + c.nb);
  const int tid = threadIdx.x, t0 = blockIdx.x * NT + tid, nt = gridDim.x * NT;
  for (int l = 0; l < c.first; ++l) {
    const GlobalX<T> x{c.x[l]}, b{c.b[l]};
    for (int s = 0; s < c.pre; ++s)
      for (int q = 0; q < 2; ++q) {
        coarse_half<T>(c.lev[l], c.dv[l], x, b, q, s == 0 && (c.zero || l > 0) ? q + 1 : 0, t0, nt);
        cluster_sync_all();
      }
    coarse_restrict<T>(c.lev[l], c.r[l], c.lev[l + 1].n, c.dv[l + 1], x, b, GlobalX<T>{c.b[l + 1]}, t0, nt);
    cluster_sync_all();
  }
  if (blockIdx.x == 0) {
    const int lf = c.first;
    const int nf = c.lev[lf].n[0] * c.lev[lf].n[1] * c.lev[lf].n[2];
    auto X = [&](int l) { return SharedX<T>{sm + c.off[l]}; };
    auto Bs = [&](int l) { return SharedX<T>{sm + c.off[l] + c.lev[l].n[0] * c.lev[l].n[1] * c.lev[l].n[2]}; };
    for (int t = tid; t < nf; t += NT) {
      Bs(lf).set(t, __ldcg(c.b[lf] + t));
      if (!c.zero && lf == 0) X(lf).set(t, __ldcg(c.x[lf] + t));
    }
    __syncthreads();
    for (int l = lf; l + 1 < c.nl; ++l) {
      for (int s = 0; s < c.pre; ++s)
        for (int q = 0; q < 2; ++q) {
          coarse_half<T>(c.lev[l], c.dv[l], X(l), Bs(l), q, s == 0 && (c.zero || l > 0) ? q + 1 : 0, tid, NT);
          __syncthreads();
        }
      coarse_restrict<T>(c.lev[l], c.r[l], c.lev[l + 1].n, c.dv[l + 1], X(l), Bs(l), Bs(l + 1), tid, NT);
      __syncthreads();
    }
    {  // x = Minv (-b)
      const int n = c.ncoarse;
      const SharedX<T> x = X(c.nl - 1), b = Bs(c.nl - 1);
      for (int t = tid; t < n; t += NT) coarse_smem[t] = -(double)b.get(t);
      __syncthreads();
      for (int rI = tid; rI < n; rI += NT) {
        double s = 0.0;
#pragma unroll 8
        for (int q = 0; q < n; ++q) s += c.minv[(size_t)rI * n + q] * coarse_smem[q];
        x.set(rI, (T)s);
      }
      __syncthreads();
    }
    for (int l = c.nl - 2; l >= lf; --l) {
      coarse_prolong<T>(c.lev[l], c.dv[l], c.r[l], c.lev[l + 1].n, X(l), X(l + 1), tid, NT);
      __syncthreads();
      for (int s = 0; s < c.post; ++s)
        for (int q = 1; q >= 0; --q) {
          coarse_half<T>(c.lev[l], c.dv[l], X(l), Bs(l), q, 0, tid, NT);
          __syncthreads();
        }
    }
    for (int t = tid; t < nf; t += NT) __stcg(c.x[lf] + t, X(lf).get(t));
  }
  for (int l = c.first - 1; l >= 0; --l) {
    cluster_sync_all();
    const GlobalX<T> x{c.x[l]}, b{c.b[l]};
    coarse_prolong<T>(c.lev[l], c.dv[l], c.r[l], c.lev[l + 1].n, x, GlobalX<T>{c.x[l + 1]}, t0, nt);
    for (int s = 0; s < c.post; ++s)
      for (int q = 1; q >= 0; --q) {
        cluster_sync_all();
        coarse_half<T>(c.lev[l], c.dv[l], x, b, q, 0, t0, nt);
      }
  }
}

// level l and everything below in one launch; false when the hierarchy does not
// fit the kernel (then a launch per operation)
template <typename T>
static bool coarse_cycle(Precond<T>& P, const Opts& o, size_t l0, bool zero, cudaStream_t st) {
  const size_t nl = P.lev.size() - l0;
  if (fsize(P.lev[l0].g, 3) > (size_t)coarse_max_cells<T>() || nl > (size_t)COARSE_LEVELS) return false;
  CoarseCycle<T> c;
  int off = 0;
  c.nl = (int)nl;
  c.first = (int)nl;
  for (size_t l = 0; l < nl; ++l) {
    MGLevel<T>& L = P.lev[l0 + l];
    c.lev[l] = plevel(L);
    c.x[l] = L.x;
    c.b[l] = L.b;
    for (int a = 0; a < 3; ++a) c.r[l][a] = L.r[a];
    c.dv[l].hx.set((L.g.n[0] + 1) / 2);
    c.dv[l].nx.set(L.g.n[0]);
    c.dv[l].ny.set(L.g.n[1]);
    c.off[l] = off;
    if (fsize(L.g, 3) <= (size_t)coarse_smem_cells<T>() || l + 1 == nl) {
      c.first = std::min(c.first, (int)l);
      off += 2 * (int)fsize(L.g, 3);
    }
  }
  c.pre = o.mg_pre;
  c.post = o.mg_post;
  c.zero = zero ? 1 : 0;
  c.ncoarse = P.ncoarse;
  c.nb = (P.ncoarse + 1) & ~1;
  c.minv = P.coarse_inv;
  const size_t smem = c.nb * sizeof(double) + off * sizeof(T);
  constexpr int NT = coarse_threads<T>();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.first > 0 ? P.coarse_ctas : 1);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cfg.gridDim.x;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_coarse_cycle<T, NT>, c);
  WSI_COUNT();
  return true;
}

// One pass of the Chebyshev smoother on A = -L (positive semi-definite)
// with Jacobi preconditioning D = diag(A): with x' = x + d (d = 0 on the
// first pass), r = L x' - b = -b - A x' (the residual of A x = -b), and
//     x_out = x',  d_out = alpha d + c r / D.
// Every cell of the level in one coalesced pass (no colouring); the caller
// alternates two buffer pairs and finishes with x += d.
template <typename T>
__global__ void k_cheb_p(GridDev g, const T* __restrict__ bx, const T* __restrict__ by, const T* __restrict__ bz,
                         const T* __restrict__ x, const T* __restrict__ d, const T* __restrict__ b, T* xo, T* dout,
                         T alpha, T c, int first) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= g.n[0] || j >= g.n[1]) return;
  const size_t id = fidx(g, 3, i, j, k);
  const size_t pl = (size_t)g.n[0] * g.n[1];
  auto xv = [&](size_t q) { return first ? x[q] : x[q] + d[q]; };
  const T ihx2 = ginv2<T>(g, 0), ihy2 = ginv2<T>(g, 1), ihz2 = ginv2<T>(g, 2);
  const T xc = xv(id);
  T s = T(0), dg = T(0);
  if (i + 1 < g.n[0]) { T w = bx[fidx(g, 0, i + 1, j, k)] * ihx2; s += w * (xv(id + 1) - xc); dg += w; }
  if (i > 0) { T w = bx[fidx(g, 0, i, j, k)] * ihx2; s += w * (xv(id - 1) - xc); dg += w; }
  if (j + 1 < g.n[1]) { T w = by[fidx(g, 1, i, j + 1, k)] * ihy2; s += w * (xv(id + g.n[0]) - xc); dg += w; }
  if (j > 0) { T w = by[fidx(g, 1, i, j, k)] * ihy2; s += w * (xv(id - g.n[0]) - xc); dg += w; }
  if (k + 1 < g.n[2]) { T w = bz[fidx(g, 2, i, j, k + 1)] * ihz2; s += w * (xv(id + pl) - xc); dg += w; }
  else if (g.open_top) { T w = T(2) * bz[fidx(g, 2, i, j, k + 1)] * ihz2; s -= w * xc; dg += w; }
  if (k > 0) { T w = bz[fidx(g, 2, i, j, k)] * ihz2; s += w * (xv(id - pl) - xc); dg += w; }
  const T r = s - b[id];
  xo[id] = xc;
  dout[id] = (first ? T(0) : alpha * d[id]) + (dg > T(0) ? c * r / dg : T(0));
}

template <typename T>
__global__ void k_cheb_finish(size_t n, const T* __restrict__ x, const T* __restrict__ d, T* out) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    out[t] = x[t] + d[t];
}

// Chebyshev interval of the Jacobi-preconditioned level operator: Gershgorin
// bounds its spectrum by 2 (diagonally dominant, zero row sums away from
// walls); the smoother targets [2/8, 2], the upper part that the coarse grid
// cannot represent.
static constexpr double CHEB_HI = 2.0, CHEB_LO = 0.25;

// one colour of a sweep over level L (zero: x is zero, whatever it holds)
template <typename T>
static void half_sweep(MGLevel<T>& L, int color, bool zero, cudaStream_t st) {
  const GridDev& g = L.g;
  ktimer_begin(KC_RBGS_P, st);
  bool done = false;
  if constexpr (sizeof(T) == 4) {
    if (g.n[0] % 4 == 0) {
      const dim3 grid(cdiv((long long)(g.n[0] / 4) * g.n[1], 256), g.n[2]);
      if (zero) k_rbgs_p4<true><<<grid, 256, 0, st>>>(plevel(L), L.x, color);
      else k_rbgs_p4<false><<<grid, 256, 0, st>>>(plevel(L), L.x, color);
      done = true;
    }
  }
  if (!done) {
    if (zero) cudaMemsetAsync(L.x, 0, fsize(g, 3) * sizeof(T), st);
    k_rbgs_p<T><<<grid_rb(g), dim3(BX, BY), 0, st>>>(plevel(L), L.x, color);
  }
  WSI_COUNT();
  ktimer_end(KC_RBGS_P, st);
}

// m passes of smoothing on level l (zero: of x = 0, whatever x holds): red-black Gauss-Seidel sweeps (pre: red
// then black; post: black then red) or a degree-m Chebyshev polynomial
template <typename T>
static void smooth(Precond<T>& P, const Opts& o, size_t l, int m, bool pre, cudaStream_t st, bool zero = false) {
  MGLevel<T>& L = P.lev[l];
  const GridDev& g = L.g;
  if (o.mg_smoother != WSI_SMOOTH_CHEBYSHEV) {
    const int c0 = pre ? 0 : 1;
    for (int s = 0; s < m; ++s)
      for (int q = 0; q < 2; ++q) half_sweep(L, q ^ c0, zero && s == 0 && q == 0, st);
    return;
  }
  if (zero) cudaMemsetAsync(L.x, 0, fsize(g, 3) * sizeof(T), st);
  const double theta = 0.5 * (CHEB_HI + CHEB_LO), delta = 0.5 * (CHEB_HI - CHEB_LO), sigma = theta / delta;
  double rho_prev = 1.0 / sigma;
  T* xs[2] = {L.x, L.cx2};
  T* ds[2] = {L.cd, L.cd2};
  const dim3 gr = grid3(g.n[0], g.n[1], g.n[2]);
  int cur = 0;
  for (int k = 0; k < m; ++k) {
    double alpha = 0.0, c = 1.0 / theta;
    if (k > 0) {
      const double rho = 1.0 / (2.0 * sigma - rho_prev);
      alpha = rho * rho_prev;
      c = 2.0 * rho / delta;
      rho_prev = rho;
    }
    ktimer_begin(KC_RBGS_P, st);
    { k_cheb_p<T><<<gr, dim3(BX, BY), 0, st>>>(g, L.beta[0], L.beta[1], L.beta[2], xs[cur], ds[cur], L.b,
                                               xs[1 - cur], ds[1 - cur], (T)alpha, (T)c, k == 0 ? 1 : 0); WSI_COUNT(); }
    ktimer_end(KC_RBGS_P, st);
    cur = 1 - cur;
  }
  const size_t n = fsize(g, 3);
  const int blocks = (int)std::min<size_t>((n + 255) / 256, 152 * 16);
  { k_cheb_finish<T><<<std::max(blocks, 1), 256, 0, st>>>(n, xs[cur], ds[cur], L.x); WSI_COUNT(); }
}

template <typename T>
static void vcycle(Precond<T>& P, const Opts& o, size_t l, bool zero, cudaStream_t st);

// pre-smoothing, residual restriction, the coarser cycle and prolongation on
// level l (everything of a V-cycle at l but the post-smoothing); zero: the
// cycle starts from x = 0, whatever x holds
template <typename T>
static void coarse_part(Precond<T>& P, const Opts& o, size_t l, bool zero, cudaStream_t st) {
  MGLevel<T>& L = P.lev[l];
  const GridDev& g = L.g;
  dim3 gr = grid3(g.n[0], g.n[1], g.n[2]);
  smooth(P, o, l, o.mg_pre, true, st, zero);
  MGLevel<T>& Cl = P.lev[l + 1];
  const GridDev& gc = Cl.g;
  ktimer_begin(KC_RESTRICT, st);
  const bool quads = sizeof(T) == 4 && g.n[0] % 4 == 0 && L.r[0] == 2 && L.r[1] == 2 && L.r[2] == 2;
  if constexpr (sizeof(T) == 4) {
    if (quads)
      k_restrict_res4<<<dim3(cdiv((long long)(g.n[0] / 4) * gc.n[1], 128), gc.n[2]), 128, 0, st>>>(plevel(L), L.x, Cl.b);
  }
  if (!quads)
    k_restrict_res<T><<<grid3(gc.n[0], gc.n[1], gc.n[2]), dim3(BX, BY), 0, st>>>(plevel(L), gc.n[0], gc.n[1], L.r[0],
                                                                              L.r[1], L.r[2], L.x, Cl.b);
  WSI_COUNT();
  ktimer_end(KC_RESTRICT, st);
  vcycle(P, o, l + 1, true, st);
  ktimer_begin(KC_PROLONG, st);
  if constexpr (sizeof(T) == 4) {
    if (quads)
      k_prolong_add4<<<dim3(cdiv((long long)(g.n[0] / 4) * g.n[1], 256), g.n[2]), 256, 0, st>>>(g.n[0], g.n[1], gc.n[2],
                                                                                              Cl.x, L.x);
  }
  if (!quads)
    k_prolong_add<T><<<gr, dim3(BX, BY), 0, st>>>(g, gc, L.r[0], L.r[1], L.r[2], Cl.x, L.x);
  WSI_COUNT();
  ktimer_end(KC_PROLONG, st);
}

template <typename T>
void precond_coarse_part(Precond<T>& P, const Opts& o, int l, cudaStream_t st) {
  coarse_part(P, o, (size_t)l, false, st);
}
template void precond_coarse_part<float>(Precond<float>&, const Opts&, int, cudaStream_t);

template <typename T>
static void vcycle(Precond<T>& P, const Opts& o, size_t l, bool zero, cudaStream_t st) {
  MGLevel<T>& L = P.lev[l];
  const GridDev& g = L.g;
  bool learned_below = false;  // a network works on this level or below
  if constexpr (std::is_same<T, float>::value)
    learned_below = P.learn.on && P.learn.ready && (size_t)P.learn.level >= l;
  if (o.mg_smoother == WSI_SMOOTH_RBGS && !learned_below && coarse_cycle(P, o, l, zero, st)) return;
  if (l + 1 == P.lev.size()) {
    { k_coarse_solve<T><<<1, 256, P.ncoarse * sizeof(double), st>>>(P.ncoarse, P.coarse_inv, L.b, L.x); WSI_COUNT(); }
    return;
  }
  if constexpr (std::is_same<T, float>::value) {
    // learned coarse-grid correction: the network replaces everything below
    // this level, then the usual post-smoothing
    if (P.learn.on && P.learn.ready && (int)l == P.learn.level && P.learn.mode == WSI_LEARN_REPLACE) {
      learned_correction(P, (int)l, L.b, false, st);
      smooth(P, o, l, o.mg_post, false, st);
      return;
    }
  }
  coarse_part(P, o, l, zero, st);
  if constexpr (std::is_same<T, float>::value) {
    // learned augmentation: the network's correction of the residual left
    // by the plain coarse-grid correction
    if (P.learn.on && P.learn.ready && (int)l == P.learn.level && P.learn.mode == WSI_LEARN_AUGMENT) {
      const size_t n = fsize(g, 3);
      const T* bt[3] = {L.beta[0], L.beta[1], L.beta[2]};
      launch_pressure<T>(g, bt, L.x, L.res, st);
      launch_lincomb_f32(n, 1.f, L.b, -1.f, L.res, 0.f, nullptr, L.res, st);
      learned_correction(P, (int)l, L.res, true, st);
    }
  }
  smooth(P, o, l, o.mg_post, false, st);
}

template <typename T>
void precond_vcycle(Precond<T>& P, const Opts& o, bool zero, cudaStream_t st) {
  vcycle(P, o, 0, zero, st);
}
template void precond_vcycle<double>(Precond<double>&, const Opts&, bool, cudaStream_t);
template void precond_vcycle<float>(Precond<float>&, const Opts&, bool, cudaStream_t);

template <typename T>
void precond_prolong_chain(Precond<T>& P, int from, cudaStream_t st) {
  for (int l = from - 1; l >= 0; --l) {
    MGLevel<T>& L = P.lev[l];
    const GridDev& g = L.g;
    cudaMemsetAsync(L.x, 0, fsize(g, 3) * sizeof(T), st);
    { k_prolong_add<T><<<grid3(g.n[0], g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, P.lev[l + 1].g, L.r[0], L.r[1],
                                                                              L.r[2], P.lev[l + 1].x, L.x); WSI_COUNT(); }
  }
}
template void precond_prolong_chain<float>(Precond<float>&, int, cudaStream_t);

int learned_alloc(Precond<float>& P, UNetImpl* net, int level, UNetImpl* gnet, int glevel, std::string& err) {
  LearnState& S = P.learn;
  S.net = net;
  S.level = level;
  S.gnet = gnet;
  S.glevel = glevel;
  S.ready = false;
  if (!net && !gnet) return WSI_OK;
  if ((net && (level < 1 || level >= (int)P.lev.size())) || (gnet && (glevel < 1 || glevel >= (int)P.lev.size()))) {
    err = "learned correction level outside the multigrid hierarchy";
    return WSI_ERR_INVALID_ARG;
  }
  if (S.lrho.empty()) {
    S.lrho.assign(P.lev.size(), nullptr);
    S.phi.assign(P.lev.size(), nullptr);
    for (size_t l = 1; l < P.lev.size(); ++l) {
      S.lrho[l] = dalloc<float>(P.allocs, fsize(P.lev[l].g, 3), err);
      S.phi[l] = dalloc<float>(P.allocs, fsize(P.lev[l].g, 3), err);
      if (!S.lrho[l] || !S.phi[l]) return WSI_ERR_OOM;
    }
    size_t nmax = fsize(P.lev[1].g, 3);
    S.diag = dalloc<float>(P.allocs, nmax, err);
    S.e = dalloc<float>(P.allocs, nmax, err);
    S.t1 = dalloc<float>(P.allocs, nmax, err);
    S.t2 = dalloc<float>(P.allocs, nmax, err);
    S.t3 = dalloc<float>(P.allocs, nmax, err);
    S.ss = dalloc<double>(P.allocs, 4, err);
    S.gdiag = dalloc<float>(P.allocs, nmax, err);
    S.gss = dalloc<double>(P.allocs, 4, err);
    if (!S.diag || !S.e || !S.t1 || !S.t2 || !S.t3 || !S.ss || !S.gdiag || !S.gss) return WSI_ERR_OOM;
  }
  return WSI_OK;
}

// ------------------------------------------------------------ PC glue kernels
// y = r_p + D u~ and the partials of its sum, in the fixed order of launch_sum
// (each thread's cells with a grid stride), so that the mean needs no second
// pass over y
template <typename T>
__global__ void __launch_bounds__(RT) k_div_sum(GridDev g, const T* __restrict__ u, const T* __restrict__ v,
                                                const T* __restrict__ w, const T* __restrict__ rp, T* y, double* part) {
  const unsigned nx = g.n[0], ny = g.n[1];
  const size_t n = (size_t)nx * ny * g.n[2], stride = (size_t)RB * RT;
  const size_t pl = (size_t)nx * ny;
  double acc = 0.0;
#pragma unroll 4
  for (size_t t = (size_t)blockIdx.x * RT + threadIdx.x; t < n; t += stride) {
    const unsigned row = (unsigned)(t / nx), k = row / ny;
    const size_t iu = t + row, iv = t + (size_t)k * nx;  // x-faces: one more per row; y-faces: one more row per plane
    const T d = (u[iu + 1] - u[iu]) * ginv<T>(g, 0) + (v[iv + nx] - v[iv]) * ginv<T>(g, 1) +
                (w[t + pl] - w[t]) * ginv<T>(g, 2);
    const T q = rp[t] + d;
    y[t] = q;
    acc += cvt<double, T>(q);
  }
  block_sum_to(acc, part);
}

// u = u~ - beta G phi on C-faces, written as float64 into z
template <int C, typename T>
__global__ void k_vel_update(GridDev g, const T* __restrict__ ut, const T* __restrict__ beta,
                             const T* __restrict__ phi, double* z) {
  int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  if (i >= ext(g, C, 0) || j >= ext(g, C, 1)) return;
  int id3[3] = {i, j, k};
  size_t id = fidx(g, C, i, j, k);
  if (!face_row(g, C, id3[C])) {
    z[id] = 0.0;
    return;
  }
  int lo[3] = {i, j, k};
  lo[C] -= 1;
  const T plo = phi[fidx(g, 3, lo[0], lo[1], lo[2])];
  const T phi_hi = (C == 2 && k == g.n[2]) ? -plo : phi[fidx(g, 3, i, j, k)];  // open top: ghost -phi
  T gphi = (phi_hi - plo) * ginv<T>(g, C);
  z[id] = cvt<double, T>(ut[id] - beta[id] * gphi);
}

// The same for the float32 preconditioner: the lower faces of each cell into
// the padded float32 parts of z (wall faces stay zero), and the open top's faces
__global__ void __launch_bounds__(256) k_vel_update_f(GridDev g, CVel<float> ut, CVel<float> beta,
                                                      const float* __restrict__ phi, float* zu, float* zv, float* zw,
                                                      int pu, int pv, int pw) {
  const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y, k = blockIdx.z;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  if (i >= nx || j >= ny) return;
  const int r = k * ny + j, id = r * nx + i, pl = nx * ny;
  const float pc = phi[id];
  if (i > 0) {
    const int q = id + r;
    const float gp = (pc - phi[id - 1]) * g.ihf[0];
    zu[(size_t)r * pu + i] = ut.q[0][q] - beta.q[0][q] * gp;
  }
  if (j > 0) {
    const int q = id + k * nx;
    const float gp = (pc - phi[id - nx]) * g.ihf[1];
    zv[(size_t)(r + k) * pv + i] = ut.q[1][q] - beta.q[1][q] * gp;
  }
  if (k > 0) {
    const float gp = (pc - phi[id - pl]) * g.ihf[2];
    zw[(size_t)r * pw + i] = ut.q[2][id] - beta.q[2][id] * gp;
  }
  if (k == nz - 1 && g.open_top) {  // ghost -phi above the open top
    const float gp = (-pc - pc) * g.ihf[2];
    zw[(size_t)(r + ny) * pw + i] = ut.q[2][id + pl] - beta.q[2][id + pl] * gp;
  }
}

// p = phi/dt - theta mu y in float32 and the partials of its sum (order of
// launch_sum on the widened values)
__global__ void __launch_bounds__(RT) k_p_sum_f(size_t n, const float* __restrict__ phi, const float* __restrict__ mu,
                                                const float* __restrict__ y, float fi, float ft, float* p,
                                                double* part) {
  double acc = 0.0;
  const size_t stride = (size_t)RB * RT;
#pragma unroll 4
  for (size_t t = (size_t)blockIdx.x * RT + threadIdx.x; t < n; t += stride) {
    const float v = phi[t] * fi - ft * mu[t] * y[t];
    p[t] = v;
    acc += f2d_fast(v);
  }
  block_sum_to(acc, part);
}

// z's pressure: p - mean (sum null: no mean removed) in float64, and split into
// the matvec's operand (padded rows); one warp per row
__global__ void __launch_bounds__(256) k_p_finish_f(int cols, int nrows, int pitch, const float* __restrict__ p,
                                                    const double* __restrict__ sum, double* z, float2* op) {
  const double m = sum ? sum[0] / ((double)cols * (double)nrows) : 0.0;
  const int lane = threadIdx.x & 31;
  for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < nrows; r += gridDim.x * 8) {
    const float* __restrict__ pr = p + (size_t)r * cols;
    for (int c0 = lane; c0 < pitch; c0 += 128) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = c0 + 32 * u < cols ? pr[c0 + 32 * u] : 0.0f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + 32 * u;
        if (c >= pitch) continue;
        double d = 0.0;
        if (c < cols) {
          d = f2d_fast(v[u]);
          if (sum) d -= m;
          z[(size_t)r * cols + c] = d;
        }
        const dfl s = df_split(d);
        op[(size_t)r * pitch + c] = make_float2(s.h, s.l);
      }
    }
  }
}

// p = phi/dt - theta mu y
__global__ void k_p_update(size_t n, const double* __restrict__ phi, const double* __restrict__ mu,
                           const double* __restrict__ y, double inv_dt, double theta, double* z) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride)
    z[t] = phi[t] * inv_dt - theta * mu[t] * y[t];
}

template <typename T>
__global__ void k_sub_mean(T* x, size_t n, const double* __restrict__ sum) {
  T m = (T)(sum[0] / (double)n);
  size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (; t < n; t += stride) x[t] -= m;
}

template <typename T>
static void sub_mean(T* x, size_t n, double* dsum, double* scratch, cudaStream_t st) {
  launch_sum<T>(x, n, dsum, scratch, st);
  int blocks = (int)std::min<size_t>((n + 255) / 256, 152 * 16);
  { k_sub_mean<T><<<std::max(blocks, 1), 256, 0, st>>>(x, n, dsum); WSI_COUNT(); }
}

// Viscous V-cycle on level l for A u = b, A = rho/dt - theta L_mu on that
// level's grid and coefficients: sweeps, face-residual restriction, the
// coarser cycle (sweeps alone on the coarsest level), prolongation, sweeps.
template <typename T>
static void vcycle_visc(Precond<T>& P, const Opts& o, size_t l, const Coef<T>& cf0, T* const u0[3],
                        const T* const b0[3], T inv_dt, T theta, cudaStream_t st) {
  const GridDev& g = P.lev[l].g;
  Coef<T> cf = cf0;
  T* const* u = u0;
  const T* const* b = b0;
  VLevel<T>& V = P.vlev[l];
  if (l > 0) {
    for (int c = 0; c < 3; ++c) {
      cf.rho_face[c] = V.rho_face[c];
      cf.mu_e[c] = V.mu_e[c];
      cf.beta[c] = nullptr;
    }
    cf.mu_cc = V.mu_cc;
    u = V.u;
    b = V.b;
  }
  const bool coarsest = l + 1 == P.lev.size();
  const int nsw = coarsest ? 4 * o.visc_sweeps : o.visc_sweeps;
  for (int s = 0; s < nsw; ++s)
    for (int c = 0; c < 2; ++c) launch_viscous_rbgs<T>(g, cf, inv_dt, theta, u, b, c, st);
  if (coarsest) return;
  T* res[3];
  for (int c = 0; c < 3; ++c) res[c] = l == 0 ? P.vres0[c] : V.res[c];
  const T* uc[3] = {u[0], u[1], u[2]};
  launch_viscous_residual<T>(g, cf, inv_dt, theta, uc, b, res, st);
  const MGLevel<T>& F = P.lev[l];
  const GridDev& gc = P.lev[l + 1].g;
  VLevel<T>& VC = P.vlev[l + 1];
  const int r0 = F.r[0], r1 = F.r[1], r2 = F.r[2];
  { k_vrestrict<0, T><<<grid3(gc.n[0] + 1, gc.n[1], gc.n[2]), dim3(BX, BY), 0, st>>>(g, gc, r0, r1, r2, res[0], VC.b[0]); WSI_COUNT(); }
  { k_vrestrict<1, T><<<grid3(gc.n[0], gc.n[1] + 1, gc.n[2]), dim3(BX, BY), 0, st>>>(g, gc, r0, r1, r2, res[1], VC.b[1]); WSI_COUNT(); }
  { k_vrestrict<2, T><<<grid3(gc.n[0], gc.n[1], gc.n[2] + 1), dim3(BX, BY), 0, st>>>(g, gc, r0, r1, r2, res[2], VC.b[2]); WSI_COUNT(); }
  for (int c = 0; c < 3; ++c) cudaMemsetAsync(VC.u[c], 0, fsize(gc, c) * sizeof(T), st);
  vcycle_visc<T>(P, o, l + 1, cf0, u0, b0, inv_dt, theta, st);
  { k_vprolong<0, T><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, gc, r0, r1, r2, VC.u[0], u[0]); WSI_COUNT(); }
  { k_vprolong<1, T><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), dim3(BX, BY), 0, st>>>(g, gc, r0, r1, r2, VC.u[1], u[1]); WSI_COUNT(); }
  { k_vprolong<2, T><<<grid3(g.n[0], g.n[1], g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, gc, r0, r1, r2, VC.u[2], u[2]); WSI_COUNT(); }
  for (int s = 0; s < o.visc_sweeps; ++s)
    for (int c = 1; c >= 0; --c) launch_viscous_rbgs<T>(g, cf, inv_dt, theta, u, b, c, st);
}

// u~ = A^{-1} r_u (into P.ut), y = r_p + D u~ (level 0's right-hand side) and
// phi = L^{-1} y (level 0's x) for the packed vector v
template <typename T>
static void precond_core(Precond<T>& P, const GridDev& g, const Opts& o, double dt, const T* v, cudaStream_t st) {
  Packing pk = packing(g);
  MGLevel<T>& L0 = P.lev[0];
  const T* ru[3] = {v + pk.off[0], v + pk.off[1], v + pk.off[2]};
  for (int c = 0; c < 3; ++c) cudaMemsetAsync(P.ut[c], 0, fsize(g, c) * sizeof(T), st);
  Coef<T> cf;
  for (int c = 0; c < 3; ++c) {
    cf.rho_face[c] = P.rho_face[c];
    cf.beta[c] = P.lev[0].beta[c];
    cf.mu_e[c] = P.mu_e[c];
  }
  cf.mu_cc = P.mu_cc;
  T inv_dt = (T)(1.0 / dt), theta = (T)o.theta;
  // u~ = A^{-1} r_u (approximately): red-black sweeps, or viscous V-cycles
  if (o.visc_mg > 0) {
    for (int c = 0; c < o.visc_mg; ++c) vcycle_visc<T>(P, o, 0, cf, P.ut, ru, inv_dt, theta, st);
  } else {
    // float64: the inverse diagonals once per set-up (and change of dt or theta)
    T* const* vd = P.vd[0] ? P.vd : nullptr;
    if constexpr (sizeof(T) == 8) {
      if (vd && !(P.vd_set && P.vd_dt == inv_dt && P.vd_theta == theta)) {
        launch_viscous_diag(g, cf, inv_dt, theta, ru, P.vd, st);
        P.vd_set = true;
        P.vd_dt = inv_dt;
        P.vd_theta = theta;
      }
    }
    for (int s = 0; s < o.visc_sweeps; ++s)
      for (int c = 0; c < 2; ++c) launch_viscous_rbgs<T>(g, cf, inv_dt, theta, P.ut, ru, c, st, vd);
  }
  // y = r_p + D u~, mean-free in a closed box (the pressure problem's
  // compatibility condition; an open top fixes the pressure instead)
  const size_t ncell = fsize(g, 3);
  { k_div_sum<T><<<RB, RT, 0, st>>>(g, P.ut[0], P.ut[1], P.ut[2], v + pk.off[3], L0.b, P.dscratch); WSI_COUNT(); }
  if (!g.open_top) {
    launch_reduce_sum(P.dscratch, P.dsum, st);
    const int blocks = (int)std::min<size_t>((ncell + 255) / 256, 152 * 16);
    { k_sub_mean<T><<<std::max(blocks, 1), 256, 0, st>>>(L0.b, ncell, P.dsum); WSI_COUNT(); }
  }
  // phi = L^{-1} y (the cycles leave their right-hand side as it is)
  for (int c = 0; c < o.mg_cycles; ++c) vcycle(P, o, 0, c == 0, st);
}

void precond_apply(Precond<double>& P, const GridDev& g, const Opts& o, double dt, const double* v, double* z,
                   cudaStream_t st) {
  precond_core<double>(P, g, o, dt, v, st);
  Packing pk = packing(g);
  const MGLevel<double>& L0 = P.lev[0];
  // velocity and pressure updates
  { k_vel_update<0, double><<<grid3(g.n[0] + 1, g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(g, P.ut[0], L0.beta[0], L0.x,
                                                                                      z + pk.off[0]); WSI_COUNT(); }
  { k_vel_update<1, double><<<grid3(g.n[0], g.n[1] + 1, g.n[2]), dim3(BX, BY), 0, st>>>(g, P.ut[1], L0.beta[1], L0.x,
                                                                                      z + pk.off[1]); WSI_COUNT(); }
  { k_vel_update<2, double><<<grid3(g.n[0], g.n[1], g.n[2] + 1), dim3(BX, BY), 0, st>>>(g, P.ut[2], L0.beta[2], L0.x,
                                                                                      z + pk.off[2]); WSI_COUNT(); }
  const size_t ncell = fsize(g, 3);
  int blocks = (int)std::min<size_t>((ncell + 255) / 256, 152 * 16);
  { k_p_update<<<std::max(blocks, 1), 256, 0, st>>>(ncell, L0.x, P.mu_cc, L0.b, 1.0 / dt, o.theta, z + pk.off[3]); WSI_COUNT(); }
  if (!g.open_top) sub_mean<double>(z + pk.off[3], ncell, P.dsum, P.dscratch, st);
}

// The mixed path's z leaves in the form that the matvec and the update of x
// read: the float32 velocity as it is (half the bytes of its float64 copy, and
// no splitting pass before the matvec), the pressure in float64 after its mean
// is removed, split on the way.  At 256^3 and per application: the splits of
// the input vector (308 us), the casts to float32 (220 us) and the float64
// velocity and pressure passes (430 us) became 290 us.
void precond_apply(Precond<float>& P, const GridDev& g, const Opts& o, double dt, const float* v, const ZVec& z,
                   const DfOperands& op, cudaStream_t st) {
  precond_core<float>(P, g, o, dt, v, st);
  const MGLevel<float>& L0 = P.lev[0];
  { k_vel_update_f<<<grid3(g.n[0], g.n[1], g.n[2]), dim3(BX, BY), 0, st>>>(
      g, CVel<float>{{P.ut[0], P.ut[1], P.ut[2]}}, CVel<float>{{L0.beta[0], L0.beta[1], L0.beta[2]}}, L0.x, z.v[0], z.v[1],
      z.v[2], op.zpitch[0], op.zpitch[1], op.zpitch[2]); WSI_COUNT(); }
  const size_t ncell = fsize(g, 3);
  { k_p_sum_f<<<RB, RT, 0, st>>>(ncell, L0.x, P.mu_cc, L0.b, (float)(1.0 / dt), (float)o.theta, P.pv, P.dscratch); WSI_COUNT(); }
  if (!g.open_top) launch_reduce_sum(P.dscratch, P.dsum, st);
  const int rows = g.n[1] * g.n[2];
  { k_p_finish_f<<<std::min(cdiv(rows, 8), 152 * 8), 256, 0, st>>>(g.n[0], rows, op.pitch[DF_P], P.pv,
                                                                  g.open_top ? nullptr : P.dsum, z.p, op.a[DF_P]); WSI_COUNT(); }
}

template int precond_alloc<double>(Precond<double>&, const GridDev&, bool, std::string&);
template int precond_alloc<float>(Precond<float>&, const GridDev&, bool, std::string&);
template void precond_free<double>(Precond<double>&);
template void precond_free<float>(Precond<float>&);
template int precond_setup<double>(Precond<double>&, const GridDev&, const Coef<double>&, bool, bool, cudaStream_t,
                                   std::string&);
template int precond_setup<float>(Precond<float>&, const GridDev&, const Coef<double>&, bool, bool, cudaStream_t,
                                  std::string&);

}  // namespace wsi
