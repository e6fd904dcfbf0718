// Float64 Krylov kernels for FGMRES (Sec. 4.2.4): block dot products against
// the Arnoldi basis, multi-axpy updates, norms and type casts.
//
// Reductions are deterministic: a fixed grid of RB blocks walks the vector
// with a grid stride, each block reduces its partial sums in shared memory
// in a fixed order, and one block adds the RB partials in block order.
#include <algorithm>

#include "internal.h"

namespace wsi {

static constexpr int NV = 8;        // basis vectors per pass

template <int M>
__global__ void k_mdot(const double* __restrict__ V, size_t ldv, int m, const double* __restrict__ w, size_t n,
                       double* part) {
  double acc[M];
#pragma unroll
  for (int t = 0; t < M; ++t) acc[t] = 0.0;
  // four independent elements per iteration keep enough loads in flight
  // to cover HBM latency
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
    double wi[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) wi[u] = (i + u * stride < n) ? w[i + u * stride] : 0.0;
#pragma unroll
    for (int t = 0; t < M; ++t)
      if (t < m) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * stride < n) acc[t] += V[(size_t)t * ldv + i + u * stride] * wi[u];
      }
  }
  __shared__ double sh[RT / 32][M];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int t = 0; t < M; ++t) {
    double v = acc[t];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wid][t] = v;
  }
  __syncthreads();
  if (threadIdx.x < M) {
    double s = 0.0;
    for (int q = 0; q < RT / 32; ++q) s += sh[q][threadIdx.x];
    part[(size_t)blockIdx.x * M + threadIdx.x] = s;
  }
}

// one block per output t < m: the block's threads stride over the nblocks
// partials in a fixed pattern and combine them with a fixed tree
__global__ void k_reduce_parts(const double* __restrict__ part, int nblocks, int M, int m, double* out) {
  int t = blockIdx.x;
  if (t >= m) return;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) s += part[(size_t)b * M + t];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  __shared__ double sh[32];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) a += sh[q];
    out[t] = a;
  }
}

void launch_mdot(const double* V, size_t ldv, int m, const double* w, size_t n, double* out, double* scratch,
                 cudaStream_t st) {
  for (int t0 = 0; t0 < m; t0 += NV) {
    int mm = std::min(NV, m - t0);
    ktimer_begin(KC_MDOT, st);
    // each distinct array read once: w is often the last basis row itself
    const bool w_in_v = w == V + (size_t)(t0 + mm - 1) * ldv;
    ktimer_bytes(KC_MDOT, 8.0 * (double)n * (mm + (w_in_v ? 0 : 1)));
    { k_mdot<NV><<<RB, RT, 0, st>>>(V + (size_t)t0 * ldv, ldv, mm, w, n, scratch); WSI_COUNT(); }
    ktimer_end(KC_MDOT, st);
    { k_reduce_parts<<<mm, 256, 0, st>>>(scratch, RB, NV, mm, out + t0); WSI_COUNT(); }
  }
}

// w = (w - sign * sum_t h[t] V_t) * scale[0]   (scale may be null: 1); w32 (may
// be null): the result in float32 as well, for the preconditioner
__global__ void k_maxpy(const double* __restrict__ V, size_t ldv, int m, const double* __restrict__ h, double* w,
                        size_t n, double sign, const double* __restrict__ scale, float* w32) {
  __shared__ double hs[64];
  if (threadIdx.x < m && threadIdx.x < 64) hs[threadIdx.x] = sign * h[threadIdx.x];
  __syncthreads();
  const double f = scale ? scale[0] : 1.0;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
    double s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] = (i + u * stride < n) ? w[i + u * stride] : 0.0;
    for (int t = 0; t < m; ++t) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + u * stride < n) s[u] -= hs[t] * V[(size_t)t * ldv + i + u * stride];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < n) {
        const double r = scale ? s[u] * f : s[u];
        w[i + u * stride] = r;
        if (w32) w32[i + u * stride] = d2f_fast(r);
      }
  }
}

void launch_maxpy(const double* V, size_t ldv, int m, const double* h, double* w, size_t n, double sign,
                  cudaStream_t st, const double* scale_dev, float* w32) {
  for (int t0 = 0; t0 < m; t0 += 64) {
    int mm = std::min(64, m - t0);
    const double* sc = (t0 + 64 >= m) ? scale_dev : nullptr;
    ktimer_begin(KC_MAXPY, st);
    ktimer_bytes(KC_MAXPY, 8.0 * (double)n * (mm + 2));  // mm rows and w read, w written
    { k_maxpy<<<RB, RT, 0, st>>>(V + (size_t)t0 * ldv, ldv, mm, h + t0, w, n, sign, sc,
                                 t0 + 64 >= m ? w32 : nullptr); WSI_COUNT(); }
    ktimer_end(KC_MAXPY, st);
  }
}

// The second pass of the orthogonalisation in one go: w -= sum_t h[t] V_t
// (t < m), and the partials of V^T w and w.w with the new w, element by element
// the operations of k_maxpy followed by k_mdot in their order.  Float64-pipe
// bound (2 m + 1 operations per element); V is read once from HBM (the second
// use hits L1) and w once: the four passes of a 256^3 step 2.61 -> 2.23 ms.
__global__ void __launch_bounds__(RT) k_orth(const double* __restrict__ V, size_t ldv, int m,
                                             const double* __restrict__ h, double* w, size_t n, double* part) {
  __shared__ double hs[NV];
  if (threadIdx.x < m) hs[threadIdx.x] = 1.0 * h[threadIdx.x];
  __syncthreads();
  double acc[NV];
#pragma unroll
  for (int t = 0; t < NV; ++t) acc[t] = 0.0;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
    double s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] = (i + u * stride < n) ? w[i + u * stride] : 0.0;
#pragma unroll
    for (int t = 0; t < NV - 1; ++t)
      if (t < m) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * stride < n) s[u] -= hs[t] * V[(size_t)t * ldv + i + u * stride];
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < n) w[i + u * stride] = s[u];
#pragma unroll
    for (int t = 0; t < NV; ++t)
      if (t < m) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * stride < n) acc[t] += V[(size_t)t * ldv + i + u * stride] * s[u];
      } else if (t == m) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * stride < n) acc[t] += s[u] * s[u];
      }
  }
  __shared__ double sh[RT / 32][NV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int t = 0; t < NV; ++t) {
    double v = acc[t];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wid][t] = v;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double a = 0.0;
    for (int q = 0; q < RT / 32; ++q) a += sh[q][threadIdx.x];
    part[(size_t)blockIdx.x * NV + threadIdx.x] = a;
  }
}

// w -= V h, out = (V^T w, w.w); w is row m of V
void launch_orth(const double* V, size_t ldv, int m, const double* h, double* w, size_t n, double* out, double* scratch,
                 cudaStream_t st) {
  if (m + 1 > NV) {
    launch_maxpy(V, ldv, m, h, w, n, 1.0, st);
    launch_mdot(V, ldv, m + 1, w, n, out, scratch, st);
    return;
  }
  ktimer_begin(KC_MDOT, st);
  ktimer_bytes(KC_MDOT, 8.0 * (double)n * (m + 2));  // m rows and w read, w written
  { k_orth<<<RB, RT, 0, st>>>(V, ldv, m, h, w, n, scratch); WSI_COUNT(); }
  ktimer_end(KC_MDOT, st);
  { k_reduce_parts<<<m + 1, 256, 0, st>>>(scratch, RB, NV, m + 1, out); WSI_COUNT(); }
}

__global__ void k_scale(double* x, size_t n, const double* __restrict__ s, float* x32) {
  const double f = s[0];
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = (i + u * stride < n) ? x[i + u * stride] : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < n) {
        const double r = v[u] * f;
        x[i + u * stride] = r;
        if (x32) x32[i + u * stride] = d2f_fast(r);
      }
  }
}

void launch_scale(double* x, size_t n, const double* s_dev, cudaStream_t st, float* x32) {
  { k_scale<<<RB, RT, 0, st>>>(x, n, s_dev, x32); WSI_COUNT(); }
}

void launch_reduce_sum(const double* part, double* out_dev, cudaStream_t st) {
  { k_reduce_parts<<<1, 256, 0, st>>>(part, RB, 1, 1, out_dev); WSI_COUNT(); }
}

template <typename T>
__global__ void k_sum(const T* __restrict__ x, size_t n, double* part) {
  double acc = 0.0;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) acc += cvt<double, T>(x[i]);
  block_sum_to(acc, part);
}

template <typename T>
void launch_sum(const T* x, size_t n, double* out_dev, double* scratch, cudaStream_t st) {
  { k_sum<T><<<RB, RT, 0, st>>>(x, n, scratch); WSI_COUNT(); }
  launch_reduce_sum(scratch, out_dev, st);
}

// r = b - r and the partials of its square sum in one pass: the same terms in
// the same order as k_mdot<1> over the finished r, which it needn't read again
// (365 -> 259 us at 256^3)
__global__ void __launch_bounds__(RT) k_residual_norm(const double* __restrict__ b, double* r, size_t n, double* part) {
  double acc = 0.0;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = (i + u * stride < n) ? b[i + u * stride] - r[i + u * stride] : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < n) {
        r[i + u * stride] = v[u];
        acc += v[u] * v[u];
      }
  }
  block_sum_to(acc, part);
}

static double read_norm(double* scratch, cudaStream_t st) {
  double h = 0.0;
  cudaMemcpyAsync(&h, scratch + RB, sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return sqrt(h);
}

double host_residual_norm2(const double* b, double* r, size_t n, double* scratch, cudaStream_t st) {
  { k_residual_norm<<<RB, RT, 0, st>>>(b, r, n, scratch); WSI_COUNT(); }
  launch_reduce_sum(scratch, scratch + RB, st);
  return read_norm(scratch, st);
}

double host_norm2(const double* x, size_t n, double* scratch, cudaStream_t st) {
  // scratch: RB + 1 doubles on the device
  { k_mdot<1><<<RB, RT, 0, st>>>(x, 0, 1, x, n, scratch); WSI_COUNT(); }
  launch_reduce_sum(scratch, scratch + RB, st);
  return read_norm(scratch, st);
}

// max |x_i|: per-block maxima, then one block over the RB partials (max is
// order-independent, so the result is exact and deterministic).  A NaN
// anywhere makes the result NaN (fmax alone would drop it and hide a blown-up
// field).
// The magnitudes are compared as bit patterns: unsigned integers order them, NaN
// above infinity, without float64 operations (418 -> 69 us for 50 M entries).
__device__ __forceinline__ unsigned long long warp_max(unsigned long long m) {
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  return m;
}
__device__ __forceinline__ void block_max_to(unsigned long long m, unsigned long long* out) {
  __shared__ unsigned long long sh[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  m = warp_max(m);
  if (lane == 0) sh[wid] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) a = max(a, sh[q]);
    *out = a;
  }
}

__global__ void k_maxabs_part(const unsigned long long* __restrict__ x, size_t n, unsigned long long* part) {
  unsigned long long m = 0;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 4 * stride) {
    unsigned long long v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = i + u * stride < n ? x[i + u * stride] : 0ull;
#pragma unroll
    for (int u = 0; u < 4; ++u) m = max(m, v[u] & 0x7FFFFFFFFFFFFFFFull);
  }
  block_max_to(m, part + blockIdx.x);
}

__global__ void k_max_parts(const unsigned long long* __restrict__ part, int nb, unsigned long long* out) {
  unsigned long long m = 0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) m = max(m, part[b]);
  block_max_to(m, out);
}

double host_maxabs(const double* x, size_t n, double* scratch, cudaStream_t st) {
  // scratch: RB + 1 doubles on the device
  unsigned long long* const part = (unsigned long long*)scratch;
  { k_maxabs_part<<<RB, RT, 0, st>>>((const unsigned long long*)x, n, part); WSI_COUNT(); }
  { k_max_parts<<<1, 256, 0, st>>>(part, RB, part + RB); WSI_COUNT(); }
  double h = 0.0;
  cudaMemcpyAsync(&h, scratch + RB, sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return h;
}

template <typename T>
__global__ void k_add_scalar(T* x, size_t n, const double* __restrict__ s, double factor) {
  T a = (T)(s[0] * factor);
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) x[i] += a;
}

template <typename T>
void launch_add_scalar_from(T* x, size_t n, const double* s_dev, double factor, cudaStream_t st) {
  { k_add_scalar<T><<<RB, RT, 0, st>>>(x, n, s_dev, factor); WSI_COUNT(); }
}

template void launch_sum<double>(const double*, size_t, double*, double*, cudaStream_t);
template void launch_sum<float>(const float*, size_t, double*, double*, cudaStream_t);
template void launch_add_scalar_from<double>(double*, size_t, const double*, double, cudaStream_t);
template void launch_add_scalar_from<float>(float*, size_t, const double*, double, cudaStream_t);

}  // namespace wsi
