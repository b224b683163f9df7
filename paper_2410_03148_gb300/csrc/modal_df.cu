// FP64-grade coupled operator in pairs of FP32 (the refinement residual).
#include "modal.cuh"

namespace cell {

namespace {

struct DfIO {
  struct Pre {
    double b[4];
  };
  const float *xh, *xl, *rh, *rl;
  float un;   // 1 / scale of the rho pair (a power of two)
  const double* b;
  double* r;
  i64 nn;
  static __device__ __forceinline__ float ld(const float* p, i64 plane, unsigned o) {
    return __ldg(p + plane + o);
  }
  __device__ __forceinline__ DF in(int d, unsigned o) const { return {ld(xh, d * nn, o), ld(xl, d * nn, o)}; }
  __device__ __forceinline__ DF rho(unsigned o) const { return {ld(rh, 0, o), ld(rl, 0, o)}; }
  __device__ __forceinline__ void fetch(Pre& p, unsigned o) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) p.b[c] = b ? __ldg(b + c * nn + o) : 0.0;
  }
  __device__ __forceinline__ void prefetch(unsigned) const {}
  __device__ __forceinline__ void out(unsigned o, DF (&acc)[4], const DF (&)[4], const Pre& p) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      double v = (double)(acc[c].h * un) + (double)(acc[c].l * un);
      if (c == 3) v = -v;
      r[c * nn + o] = b ? p.b[c] - v : v;
    }
  }
};

// Element rows per warp at 128^3 / 64^3 / 32^3 with nine loads (us): one 3746 / 478
// / 74, two 4021 / 517 / 77 (the corner form took 8300 at 128^3).  Both spill at
// 255 registers; the arithmetic alone would take about 1.5 ms.
constexpr int kRows = 1, kBlocksPerSM = 2;

__global__ void __launch_bounds__(modal::kThreads, kBlocksPerSM)
k_modal_df(const float* __restrict__ xh, const float* __restrict__ xl, i64 xs, const double* __restrict__ b, i64 bs,
           double* __restrict__ r, i64 rs, const float* __restrict__ rho_h, const float* __restrict__ rho_l,
           const float* __restrict__ unscale, const __grid_constant__ ModalMat<DF, 4, 4> K, int nx, int ny, int nz, const int* active, int L) {
  const int q = blockIdx.y;
  if (active && !__any_sync(0xffffffffu, active[q])) return;
  DfIO io;
  io.xh = xh + q * xs;
  io.xl = xl + q * xs;
  io.rh = rho_h;
  io.rl = rho_l;
  io.un = __ldg(unscale);
  io.b = b ? b + q * bs : nullptr;
  io.r = r + q * rs;
  io.nn = (i64)nx * ny * nz;
  __shared__ modal::Exchange<MK_FULL, DF> ex;
  modal::march<MK_FULL, kRows, false, DF>(K, io, ex, nx, ny, nz, L);
}

}  // namespace

void modal_resid_df(const float* xh, const float* xl, i64 xs, const double* b, i64 bs, double* r, i64 rs,
                    const float* rho_h, const float* rho_l, const float* unscale, const ModalMat<DF, 4, 4>& K, int nx,
                    int ny, int nz, int nrhs, const int* active, cudaStream_t s) {
  int L = 0;
  const dim3 grid = modal::grid_for(nx, ny, nz, nrhs, kRows, kBlocksPerSM, &L);
  note_launch(), k_modal_df<<<grid, modal::kThreads, 0, s>>>(xh, xl, xs, b, bs, r, rs, rho_h, rho_l, unscale, K, nx, ny, nz, active, L);
}

}  // namespace cell
