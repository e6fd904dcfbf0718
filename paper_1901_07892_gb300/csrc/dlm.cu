// DLM rigidity step (Sec. 4.2.5) and the IB4 Lagrangian-Eulerian transfers
// (Sec. 3.3) with the wall-adjoint forms J_BC / S_BC (Sec. 3.3.2).
//
// Both transfers work cell by cell.  The markers are binned by the cell that
// holds them (counting sort), and one warp serves up to 64 markers of a cell: their
// taps cover the same 4 x 5 x 5 faces of each component, so interpolation loads
// and splits these 300 values once for all of them, and spreading sums their
// contributions in shared memory and issues one atomic per face instead of one per
// marker and tap.  Markers outside the grid or not finite, and many markers far
// apart, get a thread each.  Weights and sums are double-float (float64 accuracy on the
// float32 pipes; GB300's float64 rate is 1/64 of its float32 rate).  Taps that
// fall beyond a wall are folded onto their mirror image with the ghost sign
// (tangential: the wall's sign; normal: odd about the wall face, whose own
// value is zero so taps landing on it drop out), which makes S_BC the exact
// adjoint of J_BC.  Rigid-body sums are deterministic two-stage reductions.
#include <math.h>

#include <algorithm>

#include "df.cuh"
#include "internal.h"

namespace wsi {

// Peskin's four-point kernel (the published formula; Sec. 3.3.1 cites it),
// evaluated in double-float arithmetic (float64 accuracy on the float32
// pipes): r = |r|; (3 - 2r + sqrt(1 + 4r - 4r^2))/8 for r <= 1,
// (5 - 2r - sqrt(-7 + 12r - 4r^2))/8 for 1 < r <= 2, 0 beyond.  The branch
// is chosen on the leading part of r; the branches agree in value and slope
// at r = 1 and r = 2, so the choice at a tie costs O(lo^2).
__device__ __forceinline__ dfl phi4_df(dfl r) {
  if (r.h < 0.0f) r = df_neg(r);
  if (r.h > 2.0f) return df_from_float(0.0f);
  const dfl r2 = df_mul(r, r);
  const dfl two_r = df_scale(r, 2.0f);
  if (r.h <= 1.0f) {
    // 1 + 4r - 4r^2
    const dfl u = df_add(df_from_float(1.0f), df_scale(df_sub(r, r2), 4.0f));
    return df_scale(df_add(df_sub(df_from_float(3.0f), two_r), df_sqrt(u)), 0.125f);
  }
  // -7 + 12r - 4r^2
  const dfl u = df_sub(df_sub(df_mul(r, df_from_float(12.0f)), df_scale(r2, 4.0f)), df_from_float(7.0f));
  return df_scale(df_sub(df_sub(df_from_float(5.0f), two_r), df_sqrt(u)), 0.125f);
}

struct Tap {
  int idx[4];
  dfl w[4];  // kernel weight times ghost sign; 0 for dropped taps
};

// the four taps along axis d of a marker at coordinate Xd, for a component
// normal to d (normal = true: faces at integer positions) or tangential
// (cell centres, offset by half a cell); positions in double-float
__device__ __forceinline__ void taps_axis(const GridDev& g, bool normal, int d, dfl Xd, dfl ih, Tap& t) {
  const int n = g.n[d];
  dfl xs = df_mul(Xd, ih);
  if (!normal) xs = df_sub(xs, df_from_float(0.5f));
  const int base = df_floor(xs) - 1;
  const float s_lo = g.bcf[2 * d], s_hi = g.bcf[2 * d + 1];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int i = base + q;
    const dfl r = df_sub(df_from_float((float)i), xs);
    float sg = 1.0f;
    for (int it = 0; it < 8; ++it) {
      if (normal) {
        if (i < 0) { i = -i; sg = -sg; }
        if (i > n) { i = 2 * n - i; sg = -sg; }
      } else {
        if (i < 0) { i = -1 - i; sg *= s_lo; }
        if (i >= n) { i = 2 * n - 1 - i; sg *= s_hi; }
      }
    }
    const bool valid = normal ? (i > 0 && i < n) : (i >= 0 && i < n);
    t.idx[q] = valid ? i : 0;
    const dfl w = phi4_df(r);
    t.w[q] = valid ? (sg < 0.0f ? df_neg(w) : w) : df_from_float(0.0f);
  }
}

// per marker: the normal and tangential taps of each axis (components share
// them: component c uses the normal taps on axis c, tangential elsewhere)
struct MarkerTaps {
  Tap tn[3], tt[3];
};

__device__ __forceinline__ void marker_taps(const GridDev& g, const double* __restrict__ X, int m, MarkerTaps& T) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const dfl xd = df_split(X[3 * m + d]);
    const dfl ih = df_split(g.ih[d]);
    taps_axis(g, true, d, xd, ih, T.tn[d]);
    taps_axis(g, false, d, xd, ih, T.tt[d]);
  }
}

// Markers of sparse cells get a warp per cell or, where there are at least this many
// of them, a thread each: the warp has the lower latency, the thread does less work.
// From markers at random over 96^3, the kernels of a call with a warp per cell and
// with a thread per marker: interpolation 10000 53 and 100 us, 16500 71 and 91, 30000
// 116 and 86, 300000 766 and 328; spreading 30000 125 and 171, 100000 251 and 254,
// 300000 561 and 463.  (Cells of four or more: a million markers with a thread each
// up to one, two and three to a cell 1281, 1038 and 1014 us, a warp each 1759.)
static constexpr int INTERP_LIST_MIN = 24576, SPREAD_LIST_MIN = 131072;

// The t-th marker of those that get a thread each: the irregular ones and, where
// there are list_min or more of them, those of sparse cells (total: how many)
__device__ __forceinline__ int list_total(const int* __restrict__ ctr, int list_min) {
  return ctr[BIN_IRR] + (ctr[BIN_SPARSE] >= list_min ? ctr[BIN_SPARSE] : 0);
}
__device__ __forceinline__ int list_marker(int t, int n, const int* __restrict__ irr, const int* __restrict__ perm,
                                           const int* __restrict__ ctr) {
  return t < ctr[BIN_IRR] ? irr[t] : perm[n - 1 - (t - ctr[BIN_IRR])];
}

// One thread per marker, all three components; separable sums
// sum_z w_z sum_y w_y sum_x w_x q in double-float, one float64 addition per
// component at the end
__global__ void __launch_bounds__(128) k_interp_list(GridDev g, CVel<double> vel, const double* __restrict__ X, int n,
                                                     const int* __restrict__ irr, const int* __restrict__ perm,
                                                     const int* __restrict__ ctr, double* U) {
  const int total = list_total(ctr, INTERP_LIST_MIN);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int m = list_marker(t, n, irr, perm, ctr);
    MarkerTaps T;
    marker_taps(g, X, m, T);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const Tap& tx = c == 0 ? T.tn[0] : T.tt[0];
      const Tap& ty = c == 1 ? T.tn[1] : T.tt[1];
      const Tap& tz = c == 2 ? T.tn[2] : T.tt[2];
      const double* __restrict__ q = vel.q[c];
      const size_t sx = (size_t)(g.n[0] + (c == 0)), sy = sx * (size_t)(g.n[1] + (c == 1));
      dfl s = df_from_float(0.0f);
#pragma unroll
      for (int kz = 0; kz < 4; ++kz) {
        if (tz.w[kz].h == 0.0f) continue;
        dfl sz = df_from_float(0.0f);
#pragma unroll
        for (int ky = 0; ky < 4; ++ky) {
          if (ty.w[ky].h == 0.0f) continue;
          const double* row = q + (size_t)tz.idx[kz] * sy + (size_t)ty.idx[ky] * sx;
          dfl sr = df_from_float(0.0f);
#pragma unroll
          for (int kx = 0; kx < 4; ++kx) sr = df_add(sr, df_mul(tx.w[kx], df_split(row[tx.idx[kx]])));
          sz = df_add(sz, df_mul(ty.w[ky], sr));
        }
        s = df_add(s, df_mul(tz.w[kz], sz));
      }
      U[3 * m + c] = df_to_double(s);
    }
  }
}

// Deterministic spreading.  Float64 atomics would sum each face's
// contributions in a varying order; instead every contribution is rounded to
// a multiple of a power-of-two quantum 2^-E and added as a 64-bit integer,
// whose sum does not depend on the order.  E is chosen on the device per call
// from a bound on any face's sum: at most 5 cells per axis hold markers whose
// taps reach a face (twice that count where taps fold at a wall), each tap
// weight is at most phi4(0)^3 = 1/8, so |sum| <= 128 c_max max|F| scale with
// c_max the most markers in one cell; E puts that bound below 2^61.  The
// quantum is then ~2^-50 of the largest contribution.

// integer nearest to f 2^E for a float f with |f 2^E| < 2^62 (integer
// operations on the bit pattern, no branch; ties away from zero): the 24-bit
// significand shifted right with rounding, or left in 64 bits
__device__ __forceinline__ long long fixed_of(float f, int E) {
  const unsigned u = __float_as_uint(f);
  const int ex = (int)((u >> 23) & 0xFFu), sh = ex - 150 + E;
  const unsigned m = ex ? ((u & 0x7FFFFFu) | 0x800000u) : 0u;  // zero (and subnormals, < 2^-126)
  const int n = min(max(-sh, 0), 25);
  const int r = (int)((m + ((1u << n) >> 1)) >> n);
  return (long long)((unsigned long long)(long long)((int)u < 0 ? -r : r) << max(sh, 0));
}

// E of the current call from the largest cell count and the bits of max|F|
__device__ __forceinline__ int spread_exponent(const int* __restrict__ ctr, const unsigned long long* __restrict__ fmx,
                                               double scale) {
  const double c = (double)ctr[BIN_CMAX], f = __longlong_as_double((long long)fmx[0]);
  const double B = 128.0 * c * f * scale;
  int e = 0;
  const bool pos = B > 0.0 && B < 1e300;
  if (pos) frexp(B, &e);  // B < 2^e
  return pos ? 61 - e : 0;
}

__global__ void __launch_bounds__(128) k_spread_list(GridDev g, const double* __restrict__ F,
                                                     const double* __restrict__ X, int n, const int* __restrict__ irr,
                                                     const int* __restrict__ perm, const int* __restrict__ ctr,
                                                     const unsigned long long* __restrict__ fmx, double scale,
                                                     Vel<unsigned long long> acc) {
  const int total = list_total(ctr, SPREAD_LIST_MIN);
  if (total == 0) return;
  const int E = spread_exponent(ctr, fmx, scale);
  const dfl sc = df_split(scale);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int m = list_marker(t, n, irr, perm, ctr);
    MarkerTaps T;
    marker_taps(g, X, m, T);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const Tap& tx = c == 0 ? T.tn[0] : T.tt[0];
      const Tap& ty = c == 1 ? T.tn[1] : T.tt[1];
      const Tap& tz = c == 2 ? T.tn[2] : T.tt[2];
      unsigned long long* q = acc.q[c];
      const size_t sx = (size_t)(g.n[0] + (c == 0)), sy = sx * (size_t)(g.n[1] + (c == 1));
      const dfl f = df_mul(df_split(F[3 * m + c]), sc);
#pragma unroll
      for (int kz = 0; kz < 4; ++kz) {
        if (tz.w[kz].h == 0.0f) continue;
#pragma unroll
        for (int ky = 0; ky < 4; ++ky) {
          if (ty.w[ky].h == 0.0f) continue;
          const dfl wyz = df_mul(tz.w[kz], ty.w[ky]);
          unsigned long long* row = q + (size_t)tz.idx[kz] * sy + (size_t)ty.idx[ky] * sx;
#pragma unroll
          for (int kx = 0; kx < 4; ++kx)
            if (tx.w[kx].h != 0.0f) {
              const dfl v = df_mul(wyz, df_mul(f, tx.w[kx]));
              atomicAdd(&row[tx.idx[kx]], (unsigned long long)(fixed_of(v.h, E) + fixed_of(v.l, E)));
            }
        }
      }
    }
  }
}

// ------------------------------------------------------------- binning by cell
// the cell of a marker for the quantum's bound: float64, clamped into the grid
__device__ __forceinline__ int bound_cell(const GridDev& g, const double* __restrict__ X, int m) {
  int c[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) c[d] = clampi((int)floor(X[3 * m + d] * g.ih[d]), 0, g.n[d] - 1);
  return (int)fidx(g, 3, c[0], c[1], c[2]);
}

// Pass 1: cell of each marker and its rank in that cell (the arrival order of
// an atomic; results don't depend on it: interpolation treats each marker by
// itself, spreading adds integers).  The cell follows the taps' double-float
// positions; bcnt counts by the float64 ones, which may differ on a cell face.
__global__ void __launch_bounds__(256) k_bin_count(GridDev g, const double* __restrict__ X, int n, int* cnt, int* bcnt,
                                                   int* cellof, int* rank, int* irr, int* ctr) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const bool valid = m < n;
  int c[3] = {0, 0, 0};
  bool in = valid;
  if (valid) {
    if (bcnt) atomicAdd(&bcnt[bound_cell(g, X, m)], 1);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const dfl x = df_split(X[3 * m + d]);
      c[d] = df_floor(df_mul(x, df_split(g.ih[d])));
      in = in && fabsf(x.h) < 1e30f && c[d] >= 0 && c[d] < g.n[d];
    }
  }
  const unsigned out = __ballot_sync(0xffffffffu, valid && !in);
  if (out) {  // places in the irregular list, one atomic per warp
    int first = 0;
    if (lane == 0) first = atomicAdd(&ctr[BIN_IRR], __popc(out));
    first = __shfl_sync(0xffffffffu, first, 0);
    if (valid && !in) {
      irr[first + __popc(out & ((1u << lane) - 1u))] = m;
      cellof[m] = -1;
      rank[m] = 0;
    }
  }
  if (!in) return;
  const int cell = (int)fidx(g, 3, c[0], c[1], c[2]);
  cellof[m] = cell;
  rank[m] = atomicAdd(&cnt[cell], 1);
}

// Pass 2: the first marker of each cell takes a range of the sorted order and
// places in the cell list, one for each CELL_MAX of its markers: what one warp works
// on (3000 markers in one cell by one warp: interpolation 1600 us, spreading 3340;
// shared out 50 and 107.  With 32 instead of 64 a lattice of 64 to a cell, a million
// markers, is 5 % slower).  Sparse cells, of at most CELL_FEW markers, take their
// ranges and places from the other end of the same arrays.  Five atomics per block;
// cnt then holds the range's start.  Also the largest of the bound's counts (bcnt not
// null).
static constexpr int CELL_MAX = 64, CELL_FEW = 3;
__global__ void __launch_bounds__(256) k_bin_alloc(GridDev g, const double* __restrict__ X, int n,
                                                   const int* __restrict__ bcnt, const int* __restrict__ cellof,
                                                   const int* __restrict__ rank, int* cnt, int* lcell, int* lstart, int* lcnt, int* ctr) {
  __shared__ int sm[8], sc[8], sf[8], sx[8], base[4];
  const int m = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int cell = m < n ? cellof[m] : -1;
  const bool first = cell >= 0 && rank[m] == 0;
  const int k = first ? cnt[cell] : 0;
  const bool few = first && k <= CELL_FEW;
  const int ka = few ? 0 : k, nb = (ka + CELL_MAX - 1) / CELL_MAX;
  // inclusive scans: markers and places of the others, markers and cells (in the
  // upper half) of the sparse ones
  int a = ka, b = nb, f = few ? k + (1 << 16) : 0, x = bcnt && m < n ? bcnt[bound_cell(g, X, m)] : 0;
  for (int o = 1; o < 32; o <<= 1) {
    const int ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o),
              uf = __shfl_up_sync(0xffffffffu, f, o);
    if (lane >= o) {
      a += ua;
      b += ub;
      f += uf;
    }
    x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
  }
  if (lane == 31) {
    sm[wid] = a;
    sc[wid] = b;
    sf[wid] = f;
    sx[wid] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int ta = 0, tb = 0, tf = 0, tx = 0;
    for (int w = 0; w < 8; ++w) {
      const int va = sm[w], vb = sc[w], vf = sf[w];
      sm[w] = ta;
      sc[w] = tb;
      sf[w] = tf;
      ta += va;
      tb += vb;
      tf += vf;
      tx = max(tx, sx[w]);
    }
    base[0] = atomicAdd(&ctr[BIN_TOTAL], ta);
    base[1] = atomicAdd(&ctr[BIN_CELLS], tb);
    base[2] = atomicAdd(&ctr[BIN_SPARSE], tf & 0xffff);
    base[3] = atomicAdd(&ctr[BIN_SPARSE_CELLS], tf >> 16);
    atomicMax(&ctr[BIN_CMAX], tx);
  }
  __syncthreads();
  if (few) {
    const int v = sf[wid] + f, start = n - base[2] - (v & 0xffff), slot = n - base[3] - (v >> 16);
    lcell[slot] = cell;
    lstart[slot] = start;
    lcnt[slot] = k;
    cnt[cell] = start;
  } else if (first) {
    const int start = base[0] + sm[wid] + a - k, slot = base[1] + sc[wid] + b - nb;
    for (int q = 0; q < nb; ++q) {
      lcell[slot + q] = cell;
      lstart[slot + q] = start + q * CELL_MAX;
      lcnt[slot + q] = min(k - q * CELL_MAX, CELL_MAX);
    }
    cnt[cell] = start;
  }
}

// Pass 3: markers in cell order; the bound's counts (bcnt not null) back to zero
__global__ void __launch_bounds__(256) k_bin_fill(GridDev g, const double* __restrict__ X, int n,
                                                  const int* __restrict__ cellof, const int* __restrict__ rank,
                                                  const int* __restrict__ cnt, int* bcnt, int* perm) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n) return;
  if (bcnt) bcnt[bound_cell(g, X, m)] = 0;
  const int cell = cellof[m];
  if (cell >= 0) perm[cnt[cell] + rank[m]] = m;
}

void launch_marker_bins(const GridDev& g, const double* X, int n, const MarkerBins& b, bool spread, cudaStream_t st) {
  if (n <= 0) return;
  cudaMemsetAsync(b.ctr, 0, BIN_CTR_BYTES, st);
  const int blocks = cdiv(n, 256);
  int* const bcnt = spread ? b.bcnt : nullptr;  // (only spreading has a quantum)
  { k_bin_count<<<blocks, 256, 0, st>>>(g, X, n, b.cnt, bcnt, b.cellof, b.rank, b.irr, b.ctr); WSI_COUNT(); }
  { k_bin_alloc<<<blocks, 256, 0, st>>>(g, X, n, bcnt, b.cellof, b.rank, b.cnt, b.lcell, b.lstart, b.lcnt,
                                           b.ctr); WSI_COUNT(); }
  { k_bin_fill<<<blocks, 256, 0, st>>>(g, X, n, b.cellof, b.rank, b.cnt, bcnt, b.perm); WSI_COUNT(); }
}

// counts of the cells back to zero for the next binning
__global__ void k_bin_clear(int n, const int* __restrict__ lcell, const int* __restrict__ ctr, int* cnt) {
  const int nc = ctr[BIN_CELLS], total = nc + ctr[BIN_SPARSE_CELLS];
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x)
    cnt[lcell[t < nc ? t : n - 1 - (t - nc)]] = 0;
}

void launch_marker_bins_clear(int n, const MarkerBins& b, cudaStream_t st) {
  if (n <= 0) return;
  { k_bin_clear<<<std::min(cdiv(n, 256), 152 * 4), 256, 0, st>>>(n, b.lcell, b.ctr, b.cnt); WSI_COUNT(); }
}

// ------------------------------------------------------------- cell transfers
// The faces that the taps of a cell's markers reach: along the component's own
// axis the four faces cell - 1 .. cell + 2, along the others the five centres
// cell - 2 .. cell + 2 (each marker uses four of them, from offset 0 or 1): 300
// slots, s = 100 c + (iz ny + iy) nx + ix.  Both kernels are bound by
// instruction issue (square roots and double-float sums).
static constexpr int CW = 4;  // warps per block
static constexpr int MB = 8;  // markers per batch

struct Slot {
  int c, ix, iy, iz;
};
__device__ __forceinline__ Slot slot_of(int s) {
  Slot q;
  q.c = s / 100;
  const int r = s - 100 * q.c, nx = q.c == 0 ? 4 : 5, ny = q.c == 1 ? 4 : 5;
  const int yz = r / nx;
  q.ix = r - yz * nx;
  q.iz = yz / ny;
  q.iy = yz - q.iz * ny;
  return q;
}

// index of unfolded position i along axis d: the face or cell it maps to and
// the ghost sign (0: dropped)
__device__ __forceinline__ int fold_index(const GridDev& g, int d, bool normal, int i, float& sg) {
  const int n = g.n[d];
  sg = 1.0f;
  if (normal) {
    for (int it = 0; it < 8 && (i < 0 || i > n); ++it) {
      if (i < 0) { i = -i; sg = -sg; }
      if (i > n) { i = 2 * n - i; sg = -sg; }
    }
    if (i <= 0 || i >= n) sg = 0.0f;
  } else {
    for (int it = 0; it < 8 && (i < 0 || i >= n); ++it) {
      if (i < 0) { i = -1 - i; sg *= g.bcf[2 * d]; }
      if (i >= n) { i = 2 * n - 1 - i; sg *= g.bcf[2 * d + 1]; }
    }
    if (i < 0 || i >= n) sg = 0.0f;
  }
  return sg != 0.0f ? i : 0;
}

// the lane's ten slots of a cell as offsets into the packed velocity layout
struct CellFaces {
  int off[10];     // from face (i, j, k) of the slot's component
  size_t base[3];  // face (i, j, k) of the current cell per component
  int ci, cj, ck;
  bool inner;      // no tap of the cell reaches a wall
  __device__ __forceinline__ void init(const GridDev& g, int lane) {
#pragma unroll
    for (int t = 0; t < 10; ++t) {
      const Slot q = slot_of(min(lane + 32 * t, 299));
      const int sx = g.n[0] + (q.c == 0), sy = sx * (g.n[1] + (q.c == 1));
      off[t] = (q.iz - (q.c == 2 ? 1 : 2)) * sy + (q.iy - (q.c == 1 ? 1 : 2)) * sx + q.ix - (q.c == 0 ? 1 : 2);
    }
  }
  __device__ __forceinline__ void move(const GridDev& g, int cid) {
    const int row = cid / g.n[0];
    ci = cid - row * g.n[0];
    ck = row / g.n[1];
    cj = row - ck * g.n[1];
    base[0] = fidx(g, 0, ci, cj, ck);
    base[1] = fsize(g, 0) + fidx(g, 1, ci, cj, ck);
    base[2] = fsize(g, 0) + fsize(g, 1) + fidx(g, 2, ci, cj, ck);
    inner = ci >= 2 && ci + 2 < g.n[0] && cj >= 2 && cj + 2 < g.n[1] && ck >= 2 && ck + 2 < g.n[2];
  }
  // packed face of slot t of this lane (cells without taps beyond a wall)
  __device__ __forceinline__ size_t face(int lane, int t) const {
    const int s = lane + 32 * t;
    return (s < 100 ? base[0] : (s < 200 ? base[1] : base[2])) + (ptrdiff_t)off[t];
  }
  // packed face of slot s and its sign, folded at walls
  __device__ __forceinline__ size_t folded_face(const GridDev& g, int s, float& sg) const {
    const Slot q = slot_of(s);
    float s0, s1, s2;
    const int i = fold_index(g, 0, q.c == 0, ci - (q.c == 0 ? 1 : 2) + q.ix, s0);
    const int j = fold_index(g, 1, q.c == 1, cj - (q.c == 1 ? 1 : 2) + q.iy, s1);
    const int k = fold_index(g, 2, q.c == 2, ck - (q.c == 2 ? 1 : 2) + q.iz, s2);
    sg = s0 * s1 * s2;
    return (q.c == 0 ? 0 : (q.c == 1 ? fsize(g, 0) : fsize(g, 0) + fsize(g, 1))) + fidx(g, q.c, i, j, k);
  }
};

// Weights of a batch of markers, shared by the warp: sets 0 .. 2 the faces
// normal to axis t, 3 .. 5 the centres along axis t - 3, four taps each, and
// per component the offset of the marker's first tap among the cell's slots
struct BatchWeights {
  float2 w[MB][24];
  float2 xs[MB][6];
  int base[MB][6];
  int off[MB][3];
};
__device__ __forceinline__ void batch_weights(const GridDev& g, const double* __restrict__ X,
                                              const int* __restrict__ perm, int nm, int lane, int ci, int cj, int ck,
                                              BatchWeights& B) {
  for (int e = lane; e < nm * 6; e += 32) {
    const int mk = e / 6, t = e - 6 * mk, d = t < 3 ? t : t - 3;
    dfl xs = df_mul(df_split(X[3 * perm[mk] + d]), df_split(g.ih[d]));
    if (t >= 3) xs = df_sub(xs, df_from_float(0.5f));
    B.xs[mk][t] = make_float2(xs.h, xs.l);
    B.base[mk][t] = df_floor(xs) - 1;
  }
  __syncwarp();
  if (lane < nm) {
    const int ox = min(max(B.base[lane][3] - (ci - 2), 0), 1), oy = min(max(B.base[lane][4] - (cj - 2), 0), 1),
              oz = min(max(B.base[lane][5] - (ck - 2), 0), 1);
    B.off[lane][0] = (oz * 5 + oy) * 4;
    B.off[lane][1] = oz * 4 * 5 + ox;
    B.off[lane][2] = oy * 5 + ox;
  }
  // the two inner taps of every set first, then the two outer ones: the lanes
  // of a pass take the same branch of the kernel function
#pragma unroll 1
  for (int half = 0; half < 2; ++half)
    for (int e = lane; e < nm * 12; e += 32) {
      const int mk = e / 12, t = (e - 12 * mk) >> 1, q = half ? 3 * (e & 1) : 1 + (e & 1);
      const float2 x = B.xs[mk][t];
      const dfl wt = phi4_df(df_sub(df_from_float((float)(B.base[mk][t] + q)), dfl{x.x, x.y}));
      B.w[mk][t * 4 + q] = make_float2(wt.h, wt.l);
    }
  __syncwarp();
}

// Interpolation: the cell's 300 values split once into shared memory; four
// lanes per marker (one per z tap), eight markers at a time, double-float
// separable sums.  1.49 million markers (eight to a cell) at 256 x 128 x 128:
// 661 us (one thread per marker, 192 loads and splits each: 1153 us).
__global__ void __launch_bounds__(32 * CW, 8) k_interp_cells(GridDev g, const double* __restrict__ vel,
                                                          const double* __restrict__ X, int n, const int* __restrict__ perm,
                                                          const int* __restrict__ lcell,
                                                          const int* __restrict__ lstart,
                                                          const int* __restrict__ lcnt, const int* __restrict__ ctr,
                                                          double* U) {
  __shared__ float2 sv[CW][300];
  __shared__ BatchWeights sb[CW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nlist = ctr[BIN_CELLS], ncells = nlist + (ctr[BIN_SPARSE] < INTERP_LIST_MIN ? ctr[BIN_SPARSE_CELLS] : 0);
  CellFaces cf;
  cf.init(g, lane);
  for (int e = blockIdx.x * CW + w; e < ncells; e += gridDim.x * CW) {
    const int l = e < nlist ? e : n - 1 - (e - nlist), cnt = lcnt[l];
    const int* pm = perm + lstart[l];
    cf.move(g, lcell[l]);
    __syncwarp();
    if (cf.inner) {
      double v[10];
#pragma unroll
      for (int t = 0; t < 10; ++t)
        if (lane + 32 * t < 300) v[t] = vel[cf.face(lane, t)];
#pragma unroll
      for (int t = 0; t < 10; ++t)
        if (lane + 32 * t < 300) {
          const dfl a = df_split(v[t]);
          sv[w][lane + 32 * t] = make_float2(a.h, a.l);
        }
    } else {
#pragma unroll 1
      for (int s = lane; s < 300; s += 32) {
        float sg;
        const dfl a = df_split(vel[cf.folded_face(g, s, sg)]);
        sv[w][s] = sg == 0.0f ? make_float2(0.f, 0.f) : make_float2(sg * a.h, sg * a.l);
      }
    }
    for (int b0 = 0; b0 < cnt; b0 += MB) {
      const int nm = min(MB, cnt - b0);
      __syncwarp();
      batch_weights(g, X, pm + b0, nm, lane, cf.ci, cf.cj, cf.ck, sb[w]);
      const int mk = lane >> 2, kz = lane & 3;
      const bool on = mk < nm;
      // rolled: the unrolled body is larger than the instruction cache likes
      // (3.9 stalled cycles per issue waiting for instructions)
#pragma unroll 1
      for (int c = 0; c < 3; ++c) {
        dfl s = df_from_float(0.0f);
        if (on) {
          const float2* W = sb[w].w[mk];
          const int tx = c == 0 ? 0 : 3, ty = c == 1 ? 1 : 4, tz = c == 2 ? 2 : 5;
          const int nx = c == 0 ? 4 : 5, ny = c == 1 ? 4 : 5;
          const float2* V = &sv[w][100 * c + kz * ny * nx + sb[w].off[mk][c]];
          dfl wx[4];
#pragma unroll
          for (int kx = 0; kx < 4; ++kx) wx[kx] = dfl{W[tx * 4 + kx].x, W[tx * 4 + kx].y};
          dfl sz = df_from_float(0.0f);
#pragma unroll
          for (int ky = 0; ky < 4; ++ky) {
            dfl sr = df_from_float(0.0f);
#pragma unroll
            for (int kx = 0; kx < 4; ++kx) {
              const float2 a = V[ky * nx + kx];
              sr = df_add(sr, df_mul(wx[kx], dfl{a.x, a.y}));
            }
            // (a row or plane of weight zero is left out, as in k_interp_list:
            // what it holds need not be finite)
            const float2 a = W[ty * 4 + ky];
            const dfl t = df_add(sz, df_mul(dfl{a.x, a.y}, sr));
            if (a.x != 0.0f) sz = t;
          }
          const float2 a = W[tz * 4 + kz];
          if (a.x != 0.0f) s = df_mul(dfl{a.x, a.y}, sz);
        }
        // z taps in order: lane kz = 0 adds its three neighbours'
        dfl tot = s;
#pragma unroll
        for (int o = 1; o < 4; ++o) {
          const dfl r{__shfl_down_sync(0xffffffffu, s.h, o), __shfl_down_sync(0xffffffffu, s.l, o)};
          tot = df_add(tot, r);
        }
        if (on && kz == 0) U[3 * pm[b0 + mk] + c] = df_to_double(tot);
      }
    }
  }
}

// Spreading: the contributions of a cell's markers are added, as integers, to
// the cell's 300 slots in shared memory (a lane per tap: two taps of each
// component, the markers one after another), then one atomic per face.  Per
// marker the products F w_x and w_y w_z are formed once and shared.  Same
// markers as above: 1114 us (192 global atomics per marker: 2468 us).
__global__ void __launch_bounds__(32 * CW, 6) k_spread_cells(GridDev g, const double* __restrict__ F,
                                                          const double* __restrict__ X, int n, const int* __restrict__ perm,
                                                          const int* __restrict__ lcell,
                                                          const int* __restrict__ lstart,
                                                          const int* __restrict__ lcnt, const int* __restrict__ ctr,
                                                          const unsigned long long* __restrict__ fmx, double scale,
                                                          unsigned long long* acc) {
  __shared__ BatchWeights sb[CW];
  __shared__ float2 sp[CW][MB][60];  // F w_x of the three components (4 each), then w_z w_y (16 each)
  __shared__ long long sa[CW][300];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nlist = ctr[BIN_CELLS], ncells = nlist + (ctr[BIN_SPARSE] < SPREAD_LIST_MIN ? ctr[BIN_SPARSE_CELLS] : 0);
  const int E = spread_exponent(ctr, fmx, scale);
  const dfl sc = df_split(scale);
  CellFaces cf;
  cf.init(g, lane);
  for (int s = lane; s < 300; s += 32) sa[w][s] = 0;
  for (int e = blockIdx.x * CW + w; e < ncells; e += gridDim.x * CW) {
    const int l = e < nlist ? e : n - 1 - (e - nlist), cnt = lcnt[l];
    const int* pm = perm + lstart[l];
    cf.move(g, lcell[l]);
    for (int b0 = 0; b0 < cnt; b0 += MB) {
      const int nm = min(MB, cnt - b0);
      __syncwarp();
      batch_weights(g, X, pm + b0, nm, lane, cf.ci, cf.cj, cf.ck, sb[w]);
      for (int e = lane; e < nm * 60; e += 32) {
        const int mk = e / 60, r = e - mk * 60;
        const float2* W = sb[w].w[mk];
        dfl v;
        if (r < 12) {
          const int c = r >> 2;
          const float2 a = W[(c == 0 ? 0 : 12) + (r & 3)];
          v = df_mul(df_mul(df_split(F[3 * pm[b0 + mk] + c]), sc), dfl{a.x, a.y});
        } else {
          const int q = r - 12, c = q >> 4;
          const float2 a = W[(c == 2 ? 8 : 20) + ((q >> 2) & 3)], b = W[(c == 1 ? 4 : 16) + (q & 3)];
          v = df_mul(dfl{a.x, a.y}, dfl{b.x, b.y});
        }
        sp[w][mk][r] = make_float2(v.h, v.l);
      }
      __syncwarp();
      for (int mk = 0; mk < nm; ++mk) {
        const float2* P = sp[w][mk];
#pragma unroll
        for (int t = 0; t < 6; ++t) {
          const int c = t >> 1, nx = c == 0 ? 4 : 5, ny = c == 1 ? 4 : 5;
          const int kx = lane & 3, ky = (lane >> 2) & 3, kz = (lane >> 4) + 2 * (t & 1);
          const float2 a = P[12 + 16 * c + 4 * kz + ky], b = P[4 * c + kx];
          const dfl v = df_mul(dfl{a.x, a.y}, dfl{b.x, b.y});
          long long* q = &sa[w][100 * c + (kz * ny + ky) * nx + kx + sb[w].off[mk][c]];
          *q += fixed_of(v.h, E) + fixed_of(v.l, E);
        }
        __syncwarp();
      }
    }
    if (cf.inner) {
#pragma unroll
      for (int t = 0; t < 10; ++t) {
        const int s = lane + 32 * t;
        const long long v = s < 300 ? sa[w][s] : 0;
        if (v != 0) {
          sa[w][s] = 0;
          atomicAdd(&acc[cf.face(lane, t)], (unsigned long long)v);
        }
      }
    } else {
#pragma unroll 1
      for (int s = lane; s < 300; s += 32) {
        const long long v = sa[w][s];
        if (v == 0) continue;
        sa[w][s] = 0;
        float sg;
        const size_t id = cf.folded_face(g, s, sg);
        if (sg != 0.0f) atomicAdd(&acc[id], (unsigned long long)(sg < 0.0f ? -v : v));
      }
    }
  }
}

// vel += acc 2^-E on the box's faces, acc cleared; blockIdx.y selects the component
__global__ void k_unfix(GridDev g, SpreadBox b, Vel<unsigned long long> acc, const int* __restrict__ ctr,
                        const unsigned long long* __restrict__ fmx, double scale, Vel<double> vel) {
  const int C = blockIdx.y;
  const int ex = b.hi[0] - b.lo[0] + 1 + (C == 0), ey = b.hi[1] - b.lo[1] + 1 + (C == 1);
  const int ez = b.hi[2] - b.lo[2] + 1 + (C == 2);
  const long long nb = (long long)ex * ey * ez;
  const double q = ldexp(1.0, -spread_exponent(ctr, fmx, scale));
  unsigned long long* ac = acc.q[C];
  double* v = vel.q[C];
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nb; t += (long long)gridDim.x * blockDim.x) {
    const int i = b.lo[0] + (int)(t % ex), j = b.lo[1] + (int)((t / ex) % ey), k = b.lo[2] + (int)(t / ((long long)ex * ey));
    const size_t id = fidx(g, C, i, j, k);
    const long long a = (long long)ac[id];
    if (a != 0) {
      v[id] += (double)a * q;
      ac[id] = 0ull;
    }
  }
}

// warps for the cell kernels: a warp per cell (at most a cell per marker) up
// to sixteen blocks per SM
static int cell_blocks(int n) { return std::min(cdiv(n, CW), 152 * 16); }
// blocks of 128 for the markers that get a thread each (the host doesn't know how
// many; with eight blocks 20000 markers outside the box took 1140 us to interpolate
// and 600 to spread, now 68 and 104)
static int list_blocks(int n) { return std::min(cdiv(n, 128), 152 * 4); }

void launch_ib_interp(const GridDev& g, const double* vel, const double* X, int n, const MarkerBins& b,
                      double* U, cudaStream_t st) {
  if (n <= 0) return;
  CVel<double> v{{vel, vel + fsize(g, 0), vel + fsize(g, 0) + fsize(g, 1)}};
  { k_interp_cells<<<cell_blocks(n), 32 * CW, 0, st>>>(g, vel, X, n, b.perm, b.lcell, b.lstart, b.lcnt, b.ctr, U); WSI_COUNT(); }
  { k_interp_list<<<list_blocks(n), 128, 0, st>>>(g, v, X, n, b.irr, b.perm, b.ctr, U); WSI_COUNT(); }
}

SpreadBox spread_box(const GridDev& g, const double mm[6]) {
  SpreadBox b;
  for (int d = 0; d < 3; ++d) {
    b.lo[d] = std::max(0, (int)std::floor(mm[d] * g.ih[d] - 0.5) - 3);
    b.hi[d] = std::min(g.n[d] - 1, (int)std::floor(mm[3 + d] * g.ih[d]) + 3);
    if (b.hi[d] < b.lo[d]) b.hi[d] = b.lo[d];
  }
  return b;
}

// |a| as ordered bits, 0 for NaN
__device__ __forceinline__ unsigned long long abs_bits(double a) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
  return u > 0x7FF0000000000000ull ? 0ull : u;
}
// block maximum of v, one atomic (maxima don't depend on the order)
__device__ __forceinline__ void block_max(unsigned long long v, unsigned long long* out) {
  __shared__ unsigned long long sh[32];
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = max(v, sh[w]);
    atomicMax(out, v);
  }
}

__global__ void __launch_bounds__(256) k_force_max(const double* __restrict__ F, int n3, unsigned long long* fmx) {
  unsigned long long v = 0;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n3; t += (long long)gridDim.x * blockDim.x)
    v = max(v, abs_bits(F[t]));
  block_max(v, fmx);
}

void launch_force_max(const double* F, int n, const MarkerBins& b, cudaStream_t st) {
  if (n <= 0) return;
  { k_force_max<<<std::min(cdiv(3LL * n, 256), 152 * 4), 256, 0, st>>>(F, 3 * n, b.fmx); WSI_COUNT(); }
}

// b.fmx holds max|F| (launch_body_velocity or launch_force_max)
void launch_ib_spread(const GridDev& g, const double* F, const double* X, int n, double dV, double* vel,
                      unsigned long long* accv, const MarkerBins& b, const SpreadBox& box, cudaStream_t st) {
  if (n <= 0) return;
  const double scale = dV / (g.h[0] * g.h[1] * g.h[2]);
  Vel<unsigned long long> acc{{accv, accv + fsize(g, 0), accv + fsize(g, 0) + fsize(g, 1)}};
  Vel<double> v{{vel, vel + fsize(g, 0), vel + fsize(g, 0) + fsize(g, 1)}};
  const long long nb = (long long)(box.hi[0] - box.lo[0] + 2) * (box.hi[1] - box.lo[1] + 2) * (box.hi[2] - box.lo[2] + 2);
  const int blocks = (int)std::min<long long>((nb + 255) / 256, 152 * 4);
  { k_spread_cells<<<cell_blocks(n), 32 * CW, 0, st>>>(g, F, X, n, b.perm, b.lcell, b.lstart, b.lcnt, b.ctr, b.fmx, scale,
                                                       accv); WSI_COUNT(); }
  { k_spread_list<<<list_blocks(n), 128, 0, st>>>(g, F, X, n, b.irr, b.perm, b.ctr, b.fmx, scale, acc); WSI_COUNT(); }
  { k_unfix<<<dim3(blocks, 3), 256, 0, st>>>(g, box, acc, b.ctr, b.fmx, scale, v); WSI_COUNT(); }
}

// ---------------------------------------------------------------- rigid sums
static constexpr int SB = 152;  // reduction blocks
static constexpr int ST = 256;
static constexpr int NS = 12;   // sums per marker
static constexpr int NM = 9;    // mean and box: three sums, three minima, three maxima

// float64 as an unsigned key of the same order (minima and maxima on the
// integer pipes), and back
__device__ __forceinline__ unsigned long long order_key(double a) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double order_value(unsigned long long k) {
  return __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k));
}

// Mean and extent of the markers: per-block partials, then one block over
// them.  NaN positions don't enter the extent.
__global__ void __launch_bounds__(ST) k_mean_box_part(const double* __restrict__ X, int n, double* part) {
  double s[3] = {0.0, 0.0, 0.0};
  const unsigned long long k0 = order_key(1e300), k1 = order_key(-1e300);
  unsigned long long mn[3] = {k0, k0, k0}, mx[3] = {k1, k1, k1};
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < n; m += gridDim.x * blockDim.x)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double x = X[3 * m + d];
      s[d] += x;
      const unsigned long long u = (unsigned long long)__double_as_longlong(x);
      if ((u & 0x7FFFFFFFFFFFFFFFull) <= 0x7FF0000000000000ull) {
        const unsigned long long k = order_key(x);
        mn[d] = min(mn[d], k);
        mx[d] = max(mx[d], k);
      }
    }
  __shared__ double sh[ST / 32][NM];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    for (int o = 16; o > 0; o >>= 1) {
      s[d] += __shfl_down_sync(0xffffffffu, s[d], o);
      mn[d] = min(mn[d], __shfl_down_sync(0xffffffffu, mn[d], o));
      mx[d] = max(mx[d], __shfl_down_sync(0xffffffffu, mx[d], o));
    }
    if (lane == 0) {
      sh[wid][d] = s[d];
      sh[wid][3 + d] = order_value(mn[d]);
      sh[wid][6 + d] = order_value(mx[d]);
    }
  }
  __syncthreads();
  if (threadIdx.x < NM) {
    const int q = threadIdx.x;
    double v = sh[0][q];
    for (int w = 1; w < ST / 32; ++w) v = q < 3 ? v + sh[w][q] : (q < 6 ? fmin(v, sh[w][q]) : fmax(v, sh[w][q]));
    part[blockIdx.x * NM + q] = v;
  }
}

// partials of all blocks staged in shared memory; the sums one thread each in
// block order (their order is fixed), the extrema one warp each
__global__ void __launch_bounds__(32 * 7) k_mean_box_final(const double* __restrict__ part, int n, double* xc,
                                                           double* box) {
  __shared__ double sp[SB * NM];
  for (int t = threadIdx.x; t < SB * NM; t += blockDim.x) sp[t] = part[t];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w == 0) {
    if (lane >= 3) return;
    double v = 0.0;
#pragma unroll 8
    for (int b = 0; b < SB; ++b) v += sp[b * NM + lane];
    xc[lane] = v / (double)n;
  } else if (box) {
    const int q = 2 + w;
    double v = sp[q];
    for (int b = lane; b < SB; b += 32) v = q < 6 ? fmin(v, sp[b * NM + q]) : fmax(v, sp[b * NM + q]);
    for (int o = 16; o > 0; o >>= 1) {
      const double p = __shfl_xor_sync(0xffffffffu, v, o);
      v = q < 6 ? fmin(v, p) : fmax(v, p);
    }
    if (lane == 0) box[q - 3] = v;
  }
}

void launch_marker_mean_box(const double* X, int n, double* xc_dev, double* box6, double* scratch, cudaStream_t st) {
  if (n <= 0) return;
  { k_mean_box_part<<<SB, ST, 0, st>>>(X, n, scratch); WSI_COUNT(); }
  { k_mean_box_final<<<1, 32 * 7, 0, st>>>(scratch, n, xc_dev, box6); WSI_COUNT(); }
}

// sums of U (0..2), R x U (3..5) and R.R I - R (x) R (6..11); float64-pipe bound
__global__ void __launch_bounds__(ST) k_rigid_part(const double* __restrict__ X, const double* __restrict__ U, int n,
                                                   const double* __restrict__ xc, double* part) {
  double acc[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) acc[q] = 0.0;
  const bool full = xc != nullptr;
  double cx = 0.0, cy = 0.0, cz = 0.0;
  if (full) {
    cx = xc[0];
    cy = xc[1];
    cz = xc[2];
  }
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < n; m += gridDim.x * blockDim.x) {
    const double ux = U[3 * m], uy = U[3 * m + 1], uz = U[3 * m + 2];
    acc[0] += ux;
    acc[1] += uy;
    acc[2] += uz;
    if (full) {
      const double rx = X[3 * m] - cx, ry = X[3 * m + 1] - cy, rz = X[3 * m + 2] - cz;
      acc[3] += ry * uz - rz * uy;
      acc[4] += rz * ux - rx * uz;
      acc[5] += rx * uy - ry * ux;
      const double rr = rx * rx + ry * ry + rz * rz;
      acc[6] += rr - rx * rx;
      acc[7] += rr - ry * ry;
      acc[8] += rr - rz * rz;
      acc[9] += -rx * ry;
      acc[10] += -rx * rz;
      acc[11] += -ry * rz;
    }
  }
  __shared__ double sh[ST / 32][NS];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    double v = acc[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wid][q] = v;
  }
  __syncthreads();
  if (threadIdx.x < NS) {
    double s = 0.0;
    for (int w = 0; w < ST / 32; ++w) s += sh[w][threadIdx.x];
    part[blockIdx.x * NS + threadIdx.x] = s;
  }
}

__global__ void __launch_bounds__(256) k_rigid_final(const double* __restrict__ part, double* out) {
  __shared__ double sp[SB * NS];
  for (int t = threadIdx.x; t < SB * NS; t += blockDim.x) sp[t] = part[t];
  __syncthreads();
  const int q = threadIdx.x;
  if (q >= NS) return;
  double s = 0.0;
  for (int b = 0; b < SB; ++b) s += sp[b * NS + q];
  out[q] = s;
}

void launch_rigid_sums(const double* X, const double* U, int n, const double* xc_dev, double* out, double* scratch,
                       cudaStream_t st) {
  { k_rigid_part<<<SB, ST, 0, st>>>(X, U, n, xc_dev, scratch); WSI_COUNT(); }
  { k_rigid_final<<<1, 256, 0, st>>>(scratch, out); WSI_COUNT(); }
}

// body velocity, F = U_b - U and max|F| (for the spreading's quantum)
__global__ void __launch_bounds__(256) k_body_vel(const double* __restrict__ X, const double* __restrict__ U, int n,
                                                  const double* __restrict__ rg, const double* __restrict__ xc,
                                                  double* Ub, double* F, unsigned long long* fmx) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long f = 0;
  if (m < n) {
    double rx = X[3 * m] - xc[0], ry = X[3 * m + 1] - xc[1], rz = X[3 * m + 2] - xc[2];
    double wx = rg[3], wy = rg[4], wz = rg[5];
    double bx = rg[0] + (wy * rz - wz * ry);
    double by = rg[1] + (wz * rx - wx * rz);
    double bz = rg[2] + (wx * ry - wy * rx);
    Ub[3 * m] = bx;
    Ub[3 * m + 1] = by;
    Ub[3 * m + 2] = bz;
    const double f0 = bx - U[3 * m], f1 = by - U[3 * m + 1], f2 = bz - U[3 * m + 2];
    F[3 * m] = f0;
    F[3 * m + 1] = f1;
    F[3 * m + 2] = f2;
    f = max(abs_bits(f0), max(abs_bits(f1), abs_bits(f2)));
  }
  block_max(f, fmx);
}

void launch_body_velocity(const double* X, const double* U, int n, const double* rigid_dev, const double* xc_dev,
                          double* Ub, double* F, const MarkerBins& b, cudaStream_t st) {
  if (n <= 0) return;
  { k_body_vel<<<cdiv(n, 256), 256, 0, st>>>(X, U, n, rigid_dev, xc_dev, Ub, F, b.fmx); WSI_COUNT(); }
}

// X = X^n + dt (U_b^{n+1} + U_b^n) / 2 (Sec. 4.2.5).  Device bound check: a
// position that is not finite or lies outside the box by more than half a
// cell sets *flag (the step then reports WSI_ERR_DEVICE); nothing traps.
__global__ void k_marker_update(GridDev g, const double* __restrict__ Xn, const double* __restrict__ Ub1,
                                const double* __restrict__ Ub0, int n3, double dt, double* X, int* flag) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n3) return;
  const double v = Xn[t] + dt * 0.5 * (Ub1[t] + Ub0[t]);
  X[t] = v;
  const int d = t % 3;
  const double tol = 0.5 * g.h[d];
  if (flag && !(v >= -tol && v <= g.n[d] * g.h[d] + tol)) atomicOr(flag, 1);
}

void launch_marker_update(const GridDev& g, const double* Xn, const double* Ub_new, const double* Ub_old, int n,
                          double dt, double* X, int* flag, cudaStream_t st) {
  if (n <= 0) return;
  { k_marker_update<<<cdiv(3LL * n, 256), 256, 0, st>>>(g, Xn, Ub_new, Ub_old, 3 * n, dt, X, flag); WSI_COUNT(); }
}

}  // namespace wsi
