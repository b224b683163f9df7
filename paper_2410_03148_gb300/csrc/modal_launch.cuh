// Kernels and launchers of the modal operators for one scalar type (included
// by modal_f32.cu and modal_f64.cu).
#pragma once

#include "modal.cuh"

namespace cell {
namespace modal {

// Inputs and outputs of one load.
template <int KIND, int MODE, typename T>
struct IO {
  static constexpr int NI = Shape<KIND>::NI, NO = Shape<KIND>::NO;
  static constexpr bool kStep = MODE >= MM_STEP;
  static constexpr bool kB = MODE != MM_APPLY;
  static constexpr bool kXp = MODE == MM_STEP;
  struct Pre {
    T b[kB ? NO : 1], xp[kXp ? NO : 1], di;
  };
  const T* x;
  T* y;
  const T* b;
  const T* xp;
  const T* dinv;
  const T* rp;
  i64 nn;
  T c1;
  T k0[3], k2[3];   // c0 dk, c2 dk per component

  __device__ __forceinline__ static T ld(const T* p, i64 plane, unsigned o) { return __ldg(p + plane + o); }
  __device__ __forceinline__ T in(int d, unsigned o) const {
    if (MODE == MM_PRE) return k0[d] * ld(dinv, 0, o) * ld(b, d * nn, o);
    return ld(x, d * nn, o);
  }
  __device__ __forceinline__ T rho(unsigned o) const { return ld(rp, 0, o); }
  __device__ __forceinline__ void fetch(Pre& p, unsigned o) const {
    if (kStep) p.di = ld(dinv, 0, o);
#pragma unroll
    for (int c = 0; c < NO; ++c) {
      if (kB) p.b[c] = ld(b, c * nn, o);
      // not through the read-only path: y may be xp (each node reads its own)
      if (kXp) p.xp[c] = xp[c * nn + o];
    }
  }
  __device__ __forceinline__ static void l2(const T* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
  __device__ __forceinline__ void prefetch(unsigned o) const {
#pragma unroll
    for (int c = 0; c < NO; ++c) {
      if (kB && MODE != MM_PRE) l2(b + c * nn + o);
      if (kXp) l2(xp + c * nn + o);
    }
  }
  __device__ __forceinline__ void out(unsigned o, T (&acc)[NO], const T (&own)[NI], const Pre& p) const {
    if (KIND == MK_FULL) acc[NO - 1] = -acc[NO - 1];
#pragma unroll
    for (int c = 0; c < NO; ++c) {
      T v;
      if (MODE == MM_APPLY) {
        v = acc[c];
      } else if (MODE == MM_ADD) {
        v = p.b[c] + acc[c];
      } else if (MODE == MM_RESID) {
        v = p.b[c] - acc[c];
      } else {
        const T x0 = own[c < NI ? c : 0];
        v = x0 + k2[c] * p.di * (p.b[c] - acc[c]);
        if (MODE == MM_STEP) v += c1 * (x0 - p.xp[c]);
        if (MODE == MM_STEP0) v += c1 * (x0 - k0[c] * p.di * p.b[c]);
        if (MODE == MM_PRE) v += c1 * x0;
      }
      y[c * nn + o] = v;
    }
  }
};

template <int KIND, int MODE, int RE, int MINB, bool PF, typename T>
__global__ void __launch_bounds__(kThreads, MINB)
k_modal(const ModalArgs<T> a, const __grid_constant__ typename MatOf<KIND, T>::type K, int L) {
  __shared__ Exchange<KIND, T> ex;
  const int r1 = min(a.nrhs, ((int)blockIdx.y + 1) * a.rg);
#pragma unroll 1
  for (int r = blockIdx.y * a.rg; r < r1; ++r) {
    // a vote, so that the branch (and every address below) is warp-uniform
    if (a.active && !__any_sync(0xffffffffu, a.active[r])) continue;
    IO<KIND, MODE, T> io;
    io.x = a.x + r * a.xs;
    io.y = a.y + r * a.ys;
    io.b = a.b + r * a.bs;
    io.xp = a.xp + r * a.ps;
    io.dinv = a.dinv;
    io.rp = a.rho;
    io.nn = (i64)a.nx * a.ny * a.nz;
    if (MODE >= MM_STEP) {
      io.c1 = a.c12[0];
#pragma unroll
      for (int c = 0; c < Shape<KIND>::NO; ++c) {
        io.k2[c] = a.c12[1] * a.dk[c];
        if (MODE == MM_STEP0 || MODE == MM_PRE) io.k0[c] = *a.c0 * a.dk[c];
      }
    }
    if (r > (int)blockIdx.y * a.rg) __syncthreads();   // the buffers of the load before
    march<KIND, RE, PF, T>(K, io, ex, a.nx, a.ny, a.nz, L);
  }
}

template <int KIND, int MODE, int RE, int MINB, bool PF, typename T>
void launch(const ModalArgs<T>& a0, const typename MatOf<KIND, T>::type& K, cudaStream_t s) {
  ModalArgs<T> a = a0;
  if (a.rg < 1) a.rg = 1;
  int L = 0;
  const dim3 grid = grid_for(a.nx, a.ny, a.nz, (a.nrhs + a.rg - 1) / a.rg, RE, MINB, &L);
  note_launch(), k_modal<KIND, MODE, RE, MINB, PF, T><<<grid, kThreads, 0, s>>>(a, K, L);
}

}  // namespace modal
}  // namespace cell
