// Arnoldi orthogonalisation of the batched flexible GMRES (§2.5): one Krylov
// space per load, low-synchronisation modified Gram-Schmidt.
//
// The new vector w = Ahat P^-1 v_j is projected off the basis with the
// coefficients of modified Gram-Schmidt, obtained from one pass of dots
// a_i = <v_i, w> and the Gram entries <v_i, v_k> that earlier steps left
// behind:  c_i = (a_i - sum_{k<i} <v_i, v_k> c_k) / <v_i, v_i>.  The second
// pass subtracts sum c_i v_i, scales by an estimate of 1 / |w'| (from |w|^2 -
// sum c_i^2 |v_i|^2) and forms the dots of the new vector with the basis and
// with itself: the Gram row of the next steps and the exact norm.  Basis
// vectors are therefore normalised only approximately; their measured norms
// nu_i enter every scalar.  (The low-synchronisation form of Swirydowicz, Langou,
// Ananthan, Yang and Thomas, "Low synchronization Gram-Schmidt and generalized
// minimal residual algorithms", 2021.)  Two basis passes and four launches per
// step; classical Gram-Schmidt with selective reorthogonalisation takes three
// passes, a scaling and eleven launches (64^3: 310 us per step at 7 vectors, half
// of them FP64 additions of the block sums, which run at 1/64 rate).  Block sums
// are pairs of FP32 with error-free additions.
#include <algorithm>
#include <cstdint>

#include "cell.h"
#include "kernels.cuh"

namespace cell {

namespace {

constexpr int kB = 256;
constexpr int kWarps = kB / 32;

// Sums of per-thread partials: an unevaluated FP32 pair for FP32 partials
// (error-free additions), FP64 for FP64 ones.
struct Sum2 {
  float h, l;
  __device__ __forceinline__ void add(float b) {
    const float s = __fadd_rn(h, b), t = __fsub_rn(s, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(b, t)));
    h = s;
  }
  __device__ __forceinline__ void merge(int o) {
    const float bh = __shfl_xor_sync(0xffffffffu, h, o), bl = __shfl_xor_sync(0xffffffffu, l, o);
    add(bh);
    l = __fadd_rn(l, bl);
  }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};
struct Sum1 {
  double h;
  __device__ __forceinline__ void add(double b) { h += b; }
  __device__ __forceinline__ void merge(int o) { h += __shfl_xor_sync(0xffffffffu, h, o); }
  __device__ __forceinline__ double value() const { return h; }
};
template <typename T> struct SumOf;
template <> struct SumOf<float> { typedef Sum2 type; };
template <> struct SumOf<double> { typedef Sum1 type; };

// Block totals of G (a power of two, at most 32) values per thread: value i
// lands in thread i * (kB / G).  sh: G x (kB + 1) values.
template <typename T, int G>
__device__ __forceinline__ double block_totals(const T (&v)[G], T* sh) {
  constexpr int S = kB / G;           // threads per value
  constexpr int W = S < 32 ? S : 32;  // of which W add it up
  const int t = threadIdx.x;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < G; ++i) sh[i * (kB + 1) + t] = v[i];
  __syncthreads();
  const int i = t / S, k = t % S;
  typename SumOf<T>::type s{};
  if (k < W) {
#pragma unroll
    for (int q = 0; q < kB / W; ++q) s.add(sh[i * (kB + 1) + k + q * W]);
  }
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) s.merge(o);
  return s.value();
}

// 16-byte vectors of T.
template <typename T> struct V16;
template <> struct V16<float> {
  static constexpr int N = 4;
  float4 v;
  __device__ __forceinline__ void fma_from(float k, const V16& a) {
    v.x = fmaf(k, a.v.x, v.x); v.y = fmaf(k, a.v.y, v.y); v.z = fmaf(k, a.v.z, v.z); v.w = fmaf(k, a.v.w, v.w);
  }
  __device__ __forceinline__ void scale(float k) { v.x *= k; v.y *= k; v.z *= k; v.w *= k; }
  __device__ __forceinline__ float dot(const V16& a, float acc) const {
    return fmaf(v.x, a.v.x, fmaf(v.y, a.v.y, fmaf(v.z, a.v.z, fmaf(v.w, a.v.w, acc))));
  }
  static __device__ __forceinline__ V16 load(const float* p, i64 k) { return {reinterpret_cast<const float4*>(p)[k]}; }
  __device__ __forceinline__ void store(float* p, i64 k) const { reinterpret_cast<float4*>(p)[k] = v; }
};
template <> struct V16<double> {
  static constexpr int N = 2;
  double2 v;
  __device__ __forceinline__ void fma_from(double k, const V16& a) { v.x = fma(k, a.v.x, v.x); v.y = fma(k, a.v.y, v.y); }
  __device__ __forceinline__ void scale(double k) { v.x *= k; v.y *= k; }
  __device__ __forceinline__ double dot(const V16& a, double acc) const { return fma(v.x, a.v.x, fma(v.y, a.v.y, acc)); }
  static __device__ __forceinline__ V16 load(const double* p, i64 k) { return {reinterpret_cast<const double2*>(p)[k]}; }
  __device__ __forceinline__ void store(double* p, i64 k) const { reinterpret_cast<double2*>(p)[k] = v; }
};

// Contiguous chunk of 16-byte elements of a block.
__device__ __forceinline__ void chunk_of(i64 n, i64& lo, i64& hi) {
  const i64 c = (n + gridDim.x - 1) / gridDim.x;
  lo = (i64)blockIdx.x * c;
  hi = lo + c < n ? lo + c : n;
}

// partial[(q * kNvMax + i) * nblk + block] = dots of w with vectors g0 .. of
// load q (vector nv - 1 is w itself).  Grid (nblk, loads, ceil(nv / G)).
template <typename T, int G>
__global__ void __launch_bounds__(kB)
k_gs_dots(const T* __restrict__ V, i64 vstride, i64 len, int nv, double* __restrict__ partial,
          const int* __restrict__ active) {
  __shared__ T sh[G * (kB + 1)];
  const int q = blockIdx.y;
  if (!active[q]) return;
  const int g0 = blockIdx.z * G, ng = min(G, nv - g0);
  const T* V0 = V + q * len + (i64)g0 * vstride;
  const T* w = V + q * len + (i64)(nv - 1) * vstride;
  i64 lo, hi;
  chunk_of(len / V16<T>::N, lo, hi);
  T acc[G];
#pragma unroll
  for (int i = 0; i < G; ++i) acc[i] = T(0);
  for (i64 k = lo + threadIdx.x; k < hi; k += kB) {
    const V16<T> x = V16<T>::load(w, k);
#pragma unroll
    for (int i = 0; i < G; ++i)
      if (i < ng) acc[i] = V16<T>::load(V0 + (i64)i * vstride, k).dot(x, acc[i]);
  }
  const double tot = block_totals<T, G>(acc, sh);
  constexpr int S = kB / G;
  const int i = threadIdx.x / S;
  if (threadIdx.x % S == 0 && i < ng) partial[((i64)q * kNvMax + g0 + i) * gridDim.x + blockIdx.x] = tot;
}

// w <- s (w - sum_{i<nb} c_i v_i), and the dots of the result with v_0 ..
// v_{nb-1} and itself (index nb).  Up to R basis values per element stay in
// registers between the two (4, 8, 16, in FP32 also 24); more are read again,
// 16 at a time.
template <typename T, int R>
__global__ void __launch_bounds__(kB)
k_gs_update(T* __restrict__ V, i64 vstride, i64 len, int nb, const double* __restrict__ coef, double* __restrict__ partial,
            const int* __restrict__ active) {
  constexpr int G = R == 0 ? 16 : (R <= 8 ? 8 : (R <= 16 ? 16 : 32));
  __shared__ T sh[G * (kB + 1)];
  __shared__ T c[kNvMax + 1];
  const int q = blockIdx.y;
  if (!active[q]) return;
  for (int i = threadIdx.x; i <= nb; i += kB)   // coefficient nb = the scale
    c[i] = (T)coef[q * (kNvMax + 1) + (i == nb ? kNvMax : i)];
  __syncthreads();
  const T* V0 = V + q * len;
  T* w = V + q * len + (i64)nb * vstride;
  const T s = c[nb];
  i64 lo, hi;
  chunk_of(len / V16<T>::N, lo, hi);
  constexpr int SP = kB / G;
  double* out = partial + (i64)q * kNvMax * gridDim.x + blockIdx.x;
  T nrm[G];
#pragma unroll
  for (int i = 0; i < G; ++i) nrm[i] = T(0);
  if (R > 0) {
    T acc[G];
#pragma unroll
    for (int i = 0; i < G; ++i) acc[i] = T(0);
    for (i64 k = lo + threadIdx.x; k < hi; k += kB) {
      V16<T> v[R > 0 ? R : 1];
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (i < nb) v[i] = V16<T>::load(V0 + (i64)i * vstride, k);
      V16<T> x = V16<T>::load(w, k);
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (i < nb) x.fma_from(-c[i], v[i]);
      x.scale(s);
      x.store(w, k);
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (i < nb) acc[i] = v[i].dot(x, acc[i]);
      nrm[0] = x.dot(x, nrm[0]);
    }
    const double tot = block_totals<T, G>(acc, sh);
    if (threadIdx.x % SP == 0 && (int)threadIdx.x / SP < nb) out[(i64)(threadIdx.x / SP) * gridDim.x] = tot;
  } else {
    for (i64 k = lo + threadIdx.x; k < hi; k += kB) {
      V16<T> x = V16<T>::load(w, k);
      for (int i = 0; i < nb; ++i) x.fma_from(-c[i], V16<T>::load(V0 + (i64)i * vstride, k));
      x.scale(s);
      x.store(w, k);
      nrm[0] = x.dot(x, nrm[0]);
    }
    for (int g0 = 0; g0 < nb; g0 += G) {
      T acc[G];
#pragma unroll
      for (int i = 0; i < G; ++i) acc[i] = T(0);
      for (i64 k = lo + threadIdx.x; k < hi; k += kB) {
        const V16<T> x = V16<T>::load(w, k);   // this thread's own values
#pragma unroll
        for (int i = 0; i < G; ++i)
          if (g0 + i < nb) acc[i] = V16<T>::load(V0 + (i64)(g0 + i) * vstride, k).dot(x, acc[i]);
      }
      const double tot = block_totals<T, G>(acc, sh);
      const int i = g0 + threadIdx.x / SP;
      if (threadIdx.x % SP == 0 && i < nb) out[(i64)i * gridDim.x] = tot;
    }
  }
  const double n2 = block_totals<T, G>(nrm, sh);
  if (threadIdx.x == 0) out[(i64)nb * gridDim.x] = n2;
}

// Block totals over the chunks: value i of load q into v[i].
__device__ __forceinline__ void reduce_chunks(const double* __restrict__ partial, int q, int nblk, int nv, double* v) {
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x >> 5; i < nv; i += kWarps) {
    const double* p = partial + ((i64)q * kNvMax + i) * nblk;
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += p[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) v[i] = s;
  }
  __syncthreads();
}

// After k_gs_dots of step j: coefficients c_0 .. c_j and the scale (entry
// kNvMax) of the update, and the Hessenberg column entries h_ij = c_i nu_i /
// nu_j.  One block per load.  G: Gram rows [load][i][k], k < i; nu2: squared
// norms [load][i].
__global__ void __launch_bounds__(kB)
k_gs_coef(const double* __restrict__ partial, int nblk, int j, const double* __restrict__ gram,
          const double* __restrict__ nu2, double* __restrict__ coef, double* __restrict__ hcol,
          const int* __restrict__ active) {
  __shared__ double a[kNvMax + 1];
  __shared__ double Gq[kNvMax * (kNvMax - 1) / 2];   // strict lower triangle, row i at i (i - 1) / 2
  const int q = blockIdx.x;
  if (!active[q]) return;
  for (int i = threadIdx.x >> 5; i <= j; i += kWarps)
    for (int k = threadIdx.x & 31; k < i; k += 32)
      Gq[i * (i - 1) / 2 + k] = gram[((i64)q * kNvMax + i) * kNvMax + k];
  reduce_chunks(partial, q, nblk, j + 2, a);   // synchronises
  if (threadIdx.x >= 32) return;
  // forward substitution: lane l holds entries l and l + 32
  const int lane = threadIdx.x;
  const double* nq = nu2 + q * kNvMax;
  double r0 = lane <= j ? a[lane] : 0.0, r1 = lane + 32 <= j ? a[lane + 32] : 0.0;
  const double n0 = lane <= j ? nq[lane] : 1.0, n1 = lane + 32 <= j ? nq[lane + 32] : 1.0;
  const double i0 = 1.0 / n0, i1 = 1.0 / n1;
  for (int i = 0; i <= j; ++i) {
    const double ci = __shfl_sync(0xffffffffu, i < 32 ? r0 * i0 : r1 * i1, i & 31);
    if (lane > i && lane <= j) r0 = fma(-Gq[lane * (lane - 1) / 2 + i], ci, r0);
    const int l1 = lane + 32;
    if (l1 > i && l1 <= j) r1 = fma(-Gq[l1 * (l1 - 1) / 2 + i], ci, r1);
  }
  double e = (lane <= j ? r0 * r0 * i0 : 0.0) + (lane + 32 <= j ? r1 * r1 * i1 : 0.0);   // sum c_i^2 |v_i|^2
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  const double nj = sqrt(nq[j]);
  double* cq = coef + q * (kNvMax + 1);
  if (lane <= j) {
    cq[lane] = r0 * i0;
    hcol[q * kNvMax + lane] = r0 / sqrt(n0) / nj;
  }
  if (lane + 32 <= j) {
    cq[lane + 32] = r1 * i1;
    hcol[q * kNvMax + lane + 32] = r1 / sqrt(n1) / nj;
  }
  if (lane == 0) {
    // the estimate cancels when w is almost in the span: its floor only
    // limits the scale, the exact norm is measured on the result
    const double w2 = a[j + 1], est = fmax(w2 - e, 1e-6 * w2);
    cq[kNvMax] = est > 0.0 ? 1.0 / sqrt(est) : 0.0;
  }
}

// After k_gs_update of step j: Gram row and norm of the new vector, Givens
// update of the least-squares problem, convergence of the load; the last block
// to finish sets the condition of the next step (if the solve is one graph).
__global__ void __launch_bounds__(kB)
k_gs_finish(const double* __restrict__ partial, int nblk, int j, int m, double* __restrict__ gram,
            double* __restrict__ nu2, const double* __restrict__ coef, const double* __restrict__ hcol,
            double* __restrict__ H, double* __restrict__ cs, double* __restrict__ sn, double* __restrict__ g, int* active,
            double* resid, const double* tolabs, int* kcount, int* ticket, int set_next,
            cudaGraphConditionalHandle next) {
  __shared__ double a[kNvMax + 1], hc[kNvMax + 1], c_[kNvMax], s_[kNvMax];
  const int q = blockIdx.x;
  if (active[q]) {
    for (int i = threadIdx.x; i < j; i += kB) {
      c_[i] = cs[q * m + i];
      s_[i] = sn[q * m + i];
    }
    for (int i = threadIdx.x; i <= j; i += kB) hc[i] = hcol[q * kNvMax + i];
    reduce_chunks(partial, q, nblk, j + 2, a);   // synchronises
    if (j + 1 < kNvMax) {
      for (int i = threadIdx.x; i <= j; i += kB) gram[((i64)q * kNvMax + j + 1) * kNvMax + i] = a[i];
      if (threadIdx.x == 0) nu2[q * kNvMax + j + 1] = a[j + 1] > 0.0 ? a[j + 1] : 1.0;
    }
    if (threadIdx.x == 0) {
      const double sc = coef[q * (kNvMax + 1) + kNvMax];
      const double hn = sc > 0.0 ? sqrt(fmax(a[j + 1], 0.0)) / (sc * sqrt(nu2[q * kNvMax + j])) : 0.0;
      double* Hq = H + (i64)q * (m + 1) * m + (i64)j * (m + 1);
      double x = hc[0];
      for (int i = 0; i < j; ++i) {
        const double y = hc[i + 1];
        Hq[i] = c_[i] * x + s_[i] * y;
        x = -s_[i] * x + c_[i] * y;
      }
      const double rr = hypot(x, hn);
      const double c = rr > 0.0 ? x / rr : 1.0, s = rr > 0.0 ? hn / rr : 0.0;
      cs[q * m + j] = c;
      sn[q * m + j] = s;
      Hq[j] = rr;
      Hq[j + 1] = 0.0;
      double* gq = g + q * (m + 1);
      const double gj = gq[j], gn = -s * gj;
      gq[j] = c * gj;
      gq[j + 1] = gn;
      resid[q] = fabs(gn);
      kcount[q] = j + 1;
      // breakdown (invariant subspace) or convergence: this space is done
      const bool brk = !(hn > 1e-300) || !(hn > 1e-14 * fabs(rr));
      if (fabs(gn) <= tolabs[q] || brk || j + 1 >= m) active[q] = 0;
    }
  }
  if (!set_next) return;
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(ticket, 1) == (int)gridDim.x - 1) {
      __threadfence();
      int any = 0;
      for (int k = 0; k < (int)gridDim.x; ++k) any |= *(volatile int*)(active + k);
      *ticket = 0;
      cudaGraphSetConditional(next, any ? 1u : 0u);
    }
  }
}

// x += sum_{i<k} y_i z_i of load q (FP64 iterate); FP32: also its pair (xh, xl).
template <typename T>
__global__ void __launch_bounds__(kB)
k_gs_solution(const T* __restrict__ Z, i64 vstride, i64 len, const double* __restrict__ y, const int* __restrict__ kcount,
              double* __restrict__ x, float* __restrict__ xh, float* __restrict__ xl, const int* __restrict__ ran) {
  __shared__ T ys[kNvMax];
  const int q = blockIdx.y;
  if (!ran[q]) return;
  const int kq = kcount[q];
  for (int i = threadIdx.x; i < kq; i += kB) ys[i] = (T)y[q * kNvMax + i];
  __syncthreads();
  const T* Z0 = Z + q * len;
  for (i64 k = (i64)blockIdx.x * kB + threadIdx.x; k < len / V16<T>::N; k += (i64)gridDim.x * kB) {
    V16<T> u{};
    for (int i = 0; i < kq; ++i) u.fma_from(ys[i], V16<T>::load(Z0 + (i64)i * vstride, k));
    if constexpr (sizeof(T) == 4) {
      const i64 o = q * len + 4 * k;
      double2* X = reinterpret_cast<double2*>(x + o);
      double2 a = X[0], b = X[1];
      a.x += (double)u.v.x; a.y += (double)u.v.y; b.x += (double)u.v.z; b.y += (double)u.v.w;
      X[0] = a;
      X[1] = b;
      const float4 h = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
      *reinterpret_cast<float4*>(xh + o) = h;
      *reinterpret_cast<float4*>(xl + o) = make_float4((float)(a.x - (double)h.x), (float)(a.y - (double)h.y),
                                                      (float)(b.x - (double)h.z), (float)(b.y - (double)h.w));
    } else {
      double2* X = reinterpret_cast<double2*>(x + q * len + 2 * k);
      double2 a = *X;
      a.x += u.v.x;
      a.y += u.v.y;
      *X = a;
    }
  }
}

}  // namespace

// Blocks per load: enough to fill the chip with nine loads, at least two
// 16-byte elements per thread; on grids of more than 2e6 values a load, as many
// (up to 1024) as keep a thread's FP32 chain at 32 products.  Error of a dot at
// 128^3 against 64 bits, relative to sum |v w|: 4.5e-10 with 256 blocks (128
// products a chain), 6.1e-11 with 1024; the FP32-pair block sums add at most
// 1e-16 at any size.
int gs_blocks(i64 len) {
  const i64 fill = std::min<i64>(256, len / (4 * 2 * kB)), chain = std::min<i64>(1024, (len + 32 * kB - 1) / (32 * kB));
  return (int)std::max<i64>(1, std::max(fill, chain));
}

template <typename T>
void gs_step(const GsArgs<T>& a, int j, cudaGraphConditionalHandle next, bool set_next, cudaStream_t s) {
  const int nv = j + 2, nb = j + 1;   // basis vectors v_0 .. v_j and w = v_{j+1}
  const dim3 g(a.nblk, a.nrhs);
  if (nv <= 4) note_launch(), k_gs_dots<T, 4><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nv, a.partial, a.active);
  else if (nv <= 8) note_launch(), k_gs_dots<T, 8><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nv, a.partial, a.active);
  else
    note_launch(), k_gs_dots<T, 16><<<dim3(a.nblk, a.nrhs, (nv + 15) / 16), kB, 0, s>>>(a.V, a.vstride, a.len, nv,
                                                                                      a.partial, a.active);
  note_launch(), k_gs_coef<<<a.nrhs, kB, 0, s>>>(a.partial, a.nblk, j, a.gram, a.nu2, a.coef, a.hcol, a.active);
  if (nb <= 4) note_launch(), k_gs_update<T, 4><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nb, a.coef, a.partial, a.active);
  else if (nb <= 8) note_launch(), k_gs_update<T, 8><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nb, a.coef, a.partial, a.active);
  else if (nb <= 16) note_launch(), k_gs_update<T, 16><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nb, a.coef, a.partial, a.active);
  else if (nb <= 24 && sizeof(T) == 4)
    note_launch(), k_gs_update<T, sizeof(T) == 4 ? 24 : 0><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nb, a.coef, a.partial, a.active);
  else note_launch(), k_gs_update<T, 0><<<g, kB, 0, s>>>(a.V, a.vstride, a.len, nb, a.coef, a.partial, a.active);
  note_launch(), k_gs_finish<<<a.nrhs, kB, 0, s>>>(a.partial, a.nblk, j, a.m, a.gram, a.nu2, a.coef, a.hcol, a.H, a.cs,
                                                  a.sn, a.g, a.active, a.resid, a.tolabs, a.kcount, a.ticket,
                                                  set_next ? 1 : 0, next);
}

template <typename T>
void gs_solution(const T* Z, i64 vstride, i64 len, const double* y, const int* kcount, double* x, float* xh, float* xl,
                 int nrhs, const int* ran, cudaStream_t s) {
  const i64 b = (len / V16<T>::N + kB - 1) / kB;
  note_launch(), k_gs_solution<T><<<dim3((unsigned)(b < 1024 ? b : 1024), nrhs), kB, 0, s>>>(Z, vstride, len, y, kcount, x,
                                                                                           xh, xl, ran);
}

#define INST(T)                                                                                              \
  template void gs_step<T>(const GsArgs<T>&, int, cudaGraphConditionalHandle, bool, cudaStream_t);            \
  template void gs_solution<T>(const T*, i64, i64, const double*, const int*, double*, float*, float*, int,   \
                               const int*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace cell
