// Batched GMRES building blocks (§2.5: right-preconditioned GMRES, one Krylov
// space per load case): FP64 dot products (norms), deterministic partial
// reductions, start of a cycle and the triangular solve at its end.  The
// Arnoldi step itself is in gs.cu.
#include <cstdint>

#include "kernels.cuh"

namespace cell {

namespace {

constexpr int kB = 256;
constexpr int kWarps = kB / 32;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block reduction of one value per thread; result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < kWarps ? sh[threadIdx.x] : 0.0;
    t = warp_sum(t);
  }
  return t;
}

// Per-thread partial sums use the vector type T (FP32 for the mixed path:
// FP64 arithmetic runs at 1/64 of the FP32 rate on this part and would cap
// the reductions far below HBM bandwidth); block and grid sums are FP64.

// Reduce G per-thread values over the block; thread i < G gets total i.
template <int G>
__device__ __forceinline__ void block_sum_many(double (&v)[G], double (*sh)[G]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < G; ++i) v[i] = warp_sum(v[i]);
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < G; ++i) sh[wid][i] = v[i];
  }
  __syncthreads();
  if (threadIdx.x < G) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += sh[w][threadIdx.x];
    v[0] = t;
  }
}

// grid (nblk, nrhs): each block computes the partial dot of v and w over a
// contiguous chunk of len.  The loop is unrolled so that each thread keeps
// several elements' loads in flight (bound by HBM latency and bandwidth).
template <typename T>
__global__ void __launch_bounds__(kB)
k_dot(const T* __restrict__ v, i64 vstride, const T* __restrict__ w, i64 wstride, i64 len,
      double* __restrict__ partial, int nvmax, const int* active) {
  __shared__ double sh[kWarps][1];
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const i64 chunk = (len + gridDim.x - 1) / gridDim.x;
  const i64 lo = (i64)blockIdx.x * chunk;
  const i64 hi = lo + chunk < len ? lo + chunk : len;
  const T* W = w + q * wstride;
  const T* V = v + q * vstride;
  T acc = T(0);
#pragma unroll 2
  for (i64 k = lo + threadIdx.x; k < hi; k += kB) acc = fma(V[k], W[k], acc);
  double d[1] = {(double)acc};
  block_sum_many<1>(d, sh);
  if (threadIdx.x == 0) partial[((i64)q * gridDim.x + blockIdx.x) * nvmax] = d[0];
}

// One warp per (rhs, i): fixed-order sum over blocks.
__global__ void k_reduce_partials(const double* __restrict__ partial, int nblk, int nv, int nvmax,
                                  double* __restrict__ out, int accumulate, const int* active) {
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const int i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= nv) return;
  double s = 0.0;
  for (int b = lane; b < nblk; b += 32) s += partial[((i64)q * nblk + b) * nvmax + i];
  s = warp_sum(s);
  if (lane == 0) out[q * nvmax + i] = accumulate ? out[q * nvmax + i] + s : s;
}

// Solve the k x k upper-triangular R y = g per rhs (mask: rhs that ran this cycle).
// The stored directions belong to basis vectors of norm nu_i: y_i / nu_i.
__global__ void k_backsolve(const double* H, const double* g, const double* nu2, const int* kcount, int m, double* y,
                            int nvmax, int nrhs, const int* mask) {
  const int q = threadIdx.x;
  if (q >= nrhs || !mask[q]) return;
  const int k = kcount[q];
  const double* Hq = H + (i64)q * (m + 1) * m;
  const double* gq = g + q * (m + 1);
  double* yq = y + q * nvmax;
  for (int i = k - 1; i >= 0; --i) {
    double t = gq[i];
    for (int l = i + 1; l < k; ++l) t -= Hq[(i64)l * (m + 1) + i] * yq[l];
    const double d = Hq[(i64)i * (m + 1) + i];
    yq[i] = d != 0.0 ? t / d : 0.0;
  }
  for (int i = 0; i < k; ++i) yq[i] /= sqrt(nu2[q * nvmax + i]);
}

// Start of a GMRES cycle: beta = ||r0||, g = beta e1, v0 scale = 1/beta.
__global__ void k_start_cycle(const double* beta2, double* g, double* nu2, int m, int nvmax, int* active,
                              const int* want, double* resid, double* invscale,
                              const double* tolabs, int* kcount, int nrhs) {
  const int q = threadIdx.x;
  if (q >= nrhs) return;
  const double beta = sqrt(fmax(beta2[q * nvmax], 0.0));
  double* gq = g + q * (m + 1);
  for (int i = 0; i <= m; ++i) gq[i] = 0.0;
  gq[0] = beta;
  nu2[q * nvmax] = 1.0;
  resid[q] = beta;
  kcount[q] = 0;
  const bool go = want[q] && beta > tolabs[q] && beta > 0.0;
  active[q] = go ? 1 : 0;
  invscale[q] = go ? 1.0 / beta : 1.0;
}

__global__ void k_to_f32(const double* __restrict__ r, i64 rs, float* __restrict__ v, i64 vs,
                         i64 len, const double* __restrict__ sc, const int* active) {
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const double f = sc[q];
  for (i64 k = (i64)blockIdx.x * blockDim.x + threadIdx.x; k < len; k += (i64)gridDim.x * blockDim.x)
    v[q * vs + k] = (float)(r[q * rs + k] * f);
}

inline unsigned stream_blocks(i64 len) {
  i64 b = (len + kB - 1) / kB;
  if (b > 4096) b = 4096;
  return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

template <typename T>
void dot(const T* v, i64 vstride, const T* w, i64 wstride, i64 len, double* partial, int nblk, int nvmax, int nrhs,
         const int* active, cudaStream_t s) {
  note_launch(), k_dot<T><<<dim3(nblk, nrhs), kB, 0, s>>>(v, vstride, w, wstride, len, partial, nvmax, active);
}

void reduce_partials(const double* partial, int nblk, int nv, int nvmax, double* out, int accumulate,
                     int nrhs, const int* active, cudaStream_t s) {
  const int wpb = 4;
  note_launch(), k_reduce_partials<<<dim3((nv + wpb - 1) / wpb, nrhs), 32 * wpb, 0, s>>>(partial, nblk, nv, nvmax,
                                                                         out, accumulate, active);
}

void backsolve(const double* H, const double* g, const double* nu2, const int* kcount, int m, double* y, int nrhs,
               const int* mask, cudaStream_t s) {
  note_launch(), k_backsolve<<<1, 32, 0, s>>>(H, g, nu2, kcount, m, y, kNvMax, nrhs, mask);
}

void start_cycle(const double* beta2, double* g, double* nu2, int m, int* active, const int* want, double* resid,
                 double* invscale, const double* tolabs, int* kcount, int nrhs, cudaStream_t s) {
  note_launch(), k_start_cycle<<<1, 32, 0, s>>>(beta2, g, nu2, m, kNvMax, active, want, resid, invscale, tolabs, kcount,
                                               nrhs);
}

void to_f32_scaled(const double* r, i64 rs, float* v, i64 vs, i64 len, const double* sc, int nrhs,
                   const int* active, cudaStream_t s) {
  note_launch(), k_to_f32<<<dim3(stream_blocks(len), nrhs), kB, 0, s>>>(r, rs, v, vs, len, sc, active);
}

template void dot<double>(const double*, i64, const double*, i64, i64, double*, int, int, int, const int*,
                          cudaStream_t);

}  // namespace cell
