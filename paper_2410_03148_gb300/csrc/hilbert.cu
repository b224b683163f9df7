// Hilbertian extension-regularisation and projection of the shape velocity
// (§2.6) on the device.
//
// The velocity space is periodic H^1 on the unit cell, <u, v>_H =
// int alpha^2 grad u . grad v + u v, discretised with the Q1 node basis:
// <u, v>_H = u^T A v, A = alpha^2 K + M.  On the structured periodic grid A is
// a constant 27-point stencil, the sum of tensor products of the 1D Q1
// stencils S = [-1, 2, -1] / h and M = h [1, 4, 1] / 6.  A nodal sensitivity
// d (a dual vector) has the Riesz representer g = A^-1 d, computed by a
// Chebyshev iteration: A's eigenvalues are the symbol values on the grid's
// Fourier modes, a multilinear function of the per-axis cosines, so its
// extremes (corners of the cosine box) bound the spectrum exactly and the
// iteration count for a given reduction follows in advance.  The objective and
// constraint representers are solved together (one launch per step, one
// vector per grid y index).
//
// Projection (null-space method): with the H Gram matrix G_ab = <g_a, g_b>_H
// = g_a . d_b, the constraint block factors as R^T R (R = the Gram-Schmidt
// coefficients of the constraint representers), theta = g R^-1 is their
// H-orthonormal basis, P g_J = g_J - sum_k <g_J, theta_k> theta_k, mu solves
// R^T mu = w_C C, and the velocity v = w_J P g_J / ||P g_J||_H + sum_k mu_k
// theta_k is formed as one linear combination of the representers.  To first
// order one step of Eq. HJ then lowers J (<g_J, v>_H = w_J ||P g_J||_H) and
// moves each constraint by -dt w_C C_i.
#include <cmath>
#include <vector>

#include "cell.h"
#include "kernels.cuh"

namespace cell {

namespace {

constexpr int kB = 256;
constexpr int kMaxVec = 1 + kHilbertMaxCons;

// The stencil is symmetric along every axis: c[x + 2 y + 4 z] is the
// coefficient of the neighbours at distance 1 along the axes whose bit is set.
struct Stencil {
  double c[8];
};

// x_1 = d / theta for every vector (grid y = vector)
__global__ void k_cheb_init(const double* const* __restrict__ rhs, double* __restrict__ x, i64 nn, double inv_theta) {
  const int v = blockIdx.y;
  const double* d = rhs[v];
  for (i64 n = (i64)blockIdx.x * blockDim.x + threadIdx.x; n < nn; n += (i64)gridDim.x * blockDim.x)
    x[v * nn + n] = d[n] * inv_theta;
}

// One Chebyshev step in three-term form,
//   x_{k+1} = x_k + ca (x_k - x_{k-1}) + cb (d - A x_k)
//           = S x_k - ca x_{k-1} + cb d,   S = (1 + ca) I - cb A,
// x_{k+1} over x_{k-1} (first: x_0 = 0, written only).  FP64 arithmetic (1/64
// rate) bounds it.
//
// Large grids: a warp marches a strip of kRows rows by 30 columns (lanes 1 ..
// 30; lanes 0 and 31 are halo) through z and adds the two neighbours along x,
// the rows of a strip along y and the planes along z once: 15 operations per
// node.  The columns of all strips form one sequence of nx + 2 positions each,
// cut into windows of 30.
constexpr int kRows = 4, kOut = 30, kStepThreads = 128, kStepWarps = kStepThreads / 32;

__global__ void __launch_bounds__(kStepThreads)
k_cheb_step(const __grid_constant__ Stencil S, const double* const* __restrict__ rhs, const double* __restrict__ xin,
            double* xio, int first, int nx, int ny, int nz, int L, double ca, double cb) {
  const int lane = threadIdx.x & 31;
  const int rl = nx + 2, strips = (ny + kRows - 1) / kRows;
  const int p0 = (int)(blockIdx.x * kStepWarps + (threadIdx.x >> 5)) * kOut;
  if (p0 >= strips * rl - 2) return;   // warp-uniform
  const int p = min(p0 + lane, strips * rl - 1);
  const int strip = p / rl, xi = p - strip * rl - 1;
  const bool vx = lane >= 1 && lane <= kOut && p0 + lane == p && xi >= 0 && xi < nx;
  const int i = xi < 0 ? nx - 1 : (xi >= nx ? 0 : xi);
  const int j0 = strip * kRows;
  unsigned ro[kRows + 2];
#pragma unroll
  for (int r = 0; r < kRows + 2; ++r) {
    int j = j0 - 1 + r;   // at most ny + kRows - 1: two subtractions wrap it
    j = j < 0 ? j + ny : j;
    j = j >= ny ? j - ny : j;
    j = j >= ny ? j - ny : j;
    ro[r] = (unsigned)(j * nx + i);
  }
  const unsigned nxy = (unsigned)(nx * ny);
  const i64 nn = (i64)nxy * nz;
  const double* X = xin + blockIdx.y * nn;
  double* Y = xio + blockIdx.y * nn;
  const double* D = rhs[blockIdx.y];
  const int z0 = blockIdx.z * L, Lc = min(L, nz - z0);
  // planes z0 - 1 .. z0 + Lc; U: in-plane part of the plane before plus the z
  // part of the one before that; W: z part of the plane before
  double U[kRows], W[kRows], vn[kRows + 2];
  unsigned zo = (unsigned)(z0 == 0 ? nz - 1 : z0 - 1) * nxy, zb = 0;
#pragma unroll
  for (int r = 0; r < kRows; ++r) U[r] = W[r] = 0.0;
#pragma unroll
  for (int r = 0; r < kRows + 2; ++r) vn[r] = __ldg(X + zo + ro[r]);
#pragma unroll 1
  for (int t = -1; t <= Lc; ++t) {
    const unsigned zn = zo + nxy == nxy * (unsigned)nz ? 0 : zo + nxy;
    double v[kRows + 2], xs[kRows + 2], d[kRows], xp[kRows];
#pragma unroll
    for (int r = 0; r < kRows + 2; ++r) {
      v[r] = vn[r];
      vn[r] = __ldg(X + zn + ro[r]);   // the plane after the last is read and not used
    }
    if (t > 0 && vx) {
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        if (j0 + r >= ny) continue;
        d[r] = __ldg(D + zb + ro[r + 1]);
        xp[r] = first ? 0.0 : Y[zb + ro[r + 1]];
      }
    }
#pragma unroll
    for (int r = 0; r < kRows + 2; ++r)
      xs[r] = __shfl_up_sync(0xffffffffu, v[r], 1) + __shfl_down_sync(0xffffffffu, v[r], 1);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const double P = v[r + 1], Xs = xs[r + 1], Ys = v[r] + v[r + 2], XY = xs[r] + xs[r + 2];
      const double w = fma(S.c[7], XY, fma(S.c[6], Ys, fma(S.c[5], Xs, S.c[4] * P)));
      const double ax = U[r] + w;   // S x on the plane before
      if (t > 0 && vx && j0 + r < ny)
        Y[zb + ro[r + 1]] = fma(-ca, xp[r], fma(cb, d[r], ax));
      U[r] = fma(S.c[3], XY, fma(S.c[2], Ys, fma(S.c[1], Xs, fma(S.c[0], P, W[r]))));
      W[r] = w;
    }
    zb = zo;
    zo = zn;
  }
}

// Small grids: one thread per node, 27 products in the grouped order of the
// symmetric stencil (19 additions and 8 products).
__global__ void __launch_bounds__(kStepThreads)
k_cheb_step_node(const __grid_constant__ Stencil S, const double* const* __restrict__ rhs, const double* __restrict__ xin,
                 double* xio, int first, int nx, int ny, int nz, double ca, double cb) {
  const int n = blockIdx.x * kStepThreads + threadIdx.x, nxy = nx * ny, nn = nxy * nz;
  if (n >= nn) return;
  const int k = n / nxy, ij = n - k * nxy, j = ij / nx, i = ij - j * nx;
  const int xo[3] = {i == 0 ? nx - 1 : i - 1, i, i == nx - 1 ? 0 : i + 1};
  const int yo[3] = {(j == 0 ? ny - 1 : j - 1) * nx, j * nx, (j == ny - 1 ? 0 : j + 1) * nx};
  const int zo[3] = {(k == 0 ? nz - 1 : k - 1) * nxy, k * nxy, (k == nz - 1 ? 0 : k + 1) * nxy};
  const i64 base = (i64)blockIdx.y * nn;
  const double* X = xin + base;
  const double dn = __ldg(rhs[blockIdx.y] + n);
  const double xp = first ? 0.0 : xio[base + n];
  // P, Xs, Ys, XY of the planes k and k - 1 + k + 1
  double s[2][4];
#pragma unroll
  for (int z = 0; z < 3; ++z) {
    double v[3][3];
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q / 3][q % 3] = __ldg(X + xo[q % 3] + yo[q / 3] + zo[z]);
    const double x0 = v[0][0] + v[0][2], x1 = v[1][0] + v[1][2], x2 = v[2][0] + v[2][2];
    const double t[4] = {v[1][1], x1, v[0][1] + v[2][1], x0 + x2};
    const int o = z == 1 ? 0 : 1;
#pragma unroll
    for (int c = 0; c < 4; ++c) s[o][c] = z == 2 ? s[o][c] + t[c] : t[c];
  }
  double ax = 0.0;
#pragma unroll
  for (int c = 0; c < 8; ++c) ax = fma(S.c[c], s[c >> 2][c & 3], ax);
  xio[base + n] = fma(-ca, xp, fma(cb, dn, ax));
}

// partial[(a * nblk + blk) * kNvMax + b] = block sum of g_a . d_b
__global__ void __launch_bounds__(kB)
k_gram(const double* __restrict__ g, const double* const* __restrict__ d, int nvec, i64 nn,
       double* __restrict__ partial) {
  __shared__ double sh[kB / 32][kMaxVec];
  const int a = blockIdx.y;
  const i64 chunk = (nn + gridDim.x - 1) / gridDim.x;
  const i64 lo = (i64)blockIdx.x * chunk, hi = lo + chunk < nn ? lo + chunk : nn;
  double acc[kMaxVec];
#pragma unroll
  for (int b = 0; b < kMaxVec; ++b) acc[b] = 0.0;
  for (i64 n = lo + threadIdx.x; n < hi; n += kB) {
    const double ga = g[a * nn + n];
#pragma unroll
    for (int b = 0; b < kMaxVec; ++b)
      if (b < nvec) acc[b] = fma(ga, d[b][n], acc[b]);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int b = 0; b < kMaxVec; ++b) {
    double v = acc[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh[w][b] = v;
  }
  __syncthreads();
  if (threadIdx.x < kMaxVec && (int)threadIdx.x < nvec) {
    double s = 0.0;
    for (int ww = 0; ww < kB / 32; ++ww) s += sh[ww][threadIdx.x];
    partial[((i64)a * gridDim.x + blockIdx.x) * kNvMax + threadIdx.x] = s;
  }
}

struct Coef {
  double c[kMaxVec];
};

__global__ void k_lincomb_vec(const double* __restrict__ g, const __grid_constant__ Coef C, int nvec, i64 nn,
                              double* __restrict__ v) {
  for (i64 n = (i64)blockIdx.x * blockDim.x + threadIdx.x; n < nn; n += (i64)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int a = 0; a < nvec; ++a) s = fma(C.c[a], g[a * nn + n], s);
    v[n] = s;
  }
}

// 1D Q1 stencils at offsets -1, 0, +1 (periodic grid of spacing h)
void stencils_1d(double h, double s[3], double m[3]) {
  s[0] = -1.0 / h; s[1] = 2.0 / h; s[2] = -1.0 / h;
  m[0] = h / 6.0; m[1] = 4.0 * h / 6.0; m[2] = h / 6.0;
}

// Symbol of A at per-axis cosines (cx, cy, cz).
double symbol(double alpha, const double h[3], const double c[3]) {
  double s[3], m[3];
  for (int d = 0; d < 3; ++d) {
    s[d] = (2.0 - 2.0 * c[d]) / h[d];
    m[d] = h[d] * (4.0 + 2.0 * c[d]) / 6.0;
  }
  return alpha * alpha * (s[0] * m[1] * m[2] + m[0] * s[1] * m[2] + m[0] * m[1] * s[2]) + m[0] * m[1] * m[2];
}

}  // namespace

int hilbert_velocity(int nx, int ny, int nz, double alpha, const double* dJ, const double* const* dC,
                     const double* C, int ncons, double wJ, double wC, double* v, double* work,
                     const double** dptrs_dev, double* partial, int nblk, double* red, double* info,
                     cudaStream_t s) {
  const i64 nn = (i64)nx * ny * nz;
  const int nvec = 1 + ncons;
  const double h[3] = {1.0 / nx, 1.0 / ny, 1.0 / nz};
  // exact spectral bounds: corners of the box of available cosines per axis
  const int n3[3] = {nx, ny, nz};
  double cmin[3];
  for (int d = 0; d < 3; ++d) cmin[d] = std::cos(2.0 * M_PI * (n3[d] / 2) / n3[d]);
  double lmin = 1e300, lmax = 0.0;
  for (int corner = 0; corner < 8; ++corner) {
    const double c[3] = {(corner & 1) ? cmin[0] : 1.0, (corner & 2) ? cmin[1] : 1.0, (corner & 4) ? cmin[2] : 1.0};
    const double l = symbol(alpha, h, c);
    lmin = std::min(lmin, l);
    lmax = std::max(lmax, l);
  }
  const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin);
  // iterations for an A-norm error reduction of 1e-13: 2 q^k / (1 + q^2k) <= 1e-13
  const double kap = lmax / lmin;
  const double q = (std::sqrt(kap) - 1.0) / (std::sqrt(kap) + 1.0);
  int iters = q <= 0.0 ? 1 : (int)std::ceil(std::log(1e-13 / 2.0) / std::log(q));
  iters = std::max(1, std::min(iters, 20000));
  const bool flat = !(delta > 1e-14 * theta);   // one eigenvalue: x = d / theta in one step
  // stencil of A: coefficient of a neighbour at distance (0 or 1) along the axes
  Stencil S;
  double sx[3], mx[3], sy[3], my[3], sz[3], mz[3];
  stencils_1d(h[0], sx, mx);
  stencils_1d(h[1], sy, my);
  stencils_1d(h[2], sz, mz);
  for (int o = 0; o < 8; ++o) {
    const int dx = (o & 1) ? 2 : 1, dy = (o & 2) ? 2 : 1, dz = (o & 4) ? 2 : 1;
    S.c[o] = alpha * alpha * (sx[dx] * my[dy] * mz[dz] + mx[dx] * sy[dy] * mz[dz] + mx[dx] * my[dy] * sz[dz]) +
             mx[dx] * my[dy] * mz[dz];
  }
  // workspace: two iterates of nvec x nn doubles
  double* x = work;
  double* x2 = x + nvec * nn;
  const double* hp[kMaxVec];
  hp[0] = dJ;
  for (int i = 0; i < ncons; ++i) hp[1 + i] = dC[i];
  cudaError_t e = cudaMemcpyAsync(dptrs_dev, hp, nvec * sizeof(double*), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return CELL_ECUDA;
  const unsigned nb = (unsigned)std::min<i64>((nn + kB - 1) / kB, 4096);
  note_launch(), k_cheb_init<<<dim3(nb, nvec), kB, 0, s>>>(dptrs_dev, x, nn, 1.0 / theta);
  // The march pays its longer serial chain back from about 4e5 node values on
  // (us a step, node kernel against march: 96^3 x 4 200 / 151, 64^3 x 3 48 / 40,
  // 48^3 x 3 24 / 26, 64^3 x 1 20 / 22, 30 x 33 x 27 x 2 7 / 17; 27 products a
  // node and the direction form take 216, 53 and 9 where the better is 151, 40 and 7);
  // two blocks per SM, a chunk reads two planes more than it writes.
  const bool march = nn * nvec >= 400000;
  const i64 windows = ((i64)((ny + kRows - 1) / kRows) * (nx + 2) - 2 + kOut - 1) / kOut;
  const i64 blocks = (windows + kStepWarps - 1) / kStepWarps;
  i64 chunks = std::max<i64>(1, modal::sm_count() * 2 / (blocks * nvec));
  chunks = std::min<i64>(chunks, std::min(nz, 4096));
  const int L = (int)((nz + chunks - 1) / chunks);
  const dim3 grid((unsigned)blocks, (unsigned)nvec, (unsigned)((nz + L - 1) / L));
  const dim3 nodes((unsigned)((nn + kStepThreads - 1) / kStepThreads), (unsigned)nvec);
  const double s1 = flat ? 1.0 : theta / delta;
  double rho0 = 1.0 / s1;
  // x_1 = d / theta is the first of the iterations
  for (int k = 0; k + 1 < (flat ? 1 : iters); ++k) {
    const double rho1 = 1.0 / (2.0 * s1 - rho0);
    const double ca = rho1 * rho0, cb = 2.0 * rho1 / delta;
    Stencil Sk;
    for (int o = 0; o < 8; ++o) Sk.c[o] = (o == 0 ? 1.0 + ca : 0.0) - cb * S.c[o];
    if (march)
      note_launch(), k_cheb_step<<<grid, kStepThreads, 0, s>>>(Sk, dptrs_dev, x, x2, k == 0, nx, ny, nz, L, ca, cb);
    else
      note_launch(), k_cheb_step_node<<<nodes, kStepThreads, 0, s>>>(Sk, dptrs_dev, x, x2, k == 0, nx, ny, nz, ca, cb);
    std::swap(x, x2);
    rho0 = rho1;
  }
  if (flat) iters = 1;
  note_launch(), k_gram<<<dim3(nblk, nvec), kB, 0, s>>>(x, dptrs_dev, nvec, nn, partial);
  reduce_partials(partial, nblk, nvec, kNvMax, red, 0, nvec, nullptr, s);
  std::vector<double> Gr((size_t)nvec * kNvMax);
  e = cudaMemcpyAsync(Gr.data(), red, Gr.size() * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return CELL_ECUDA;
  // symmetric H Gram matrix of (g_J, g_1..g_N)
  double G[kMaxVec][kMaxVec];
  for (int a = 0; a < nvec; ++a)
    for (int b = 0; b < nvec; ++b) G[a][b] = 0.5 * (Gr[a * kNvMax + b] + Gr[b * kNvMax + a]);
  // constraint block = R^T R (Cholesky, R upper triangular), Rinv = R^-1
  const int N = ncons;
  double R[kMaxVec][kMaxVec] = {}, Ri[kMaxVec][kMaxVec] = {};
  for (int j = 0; j < N; ++j) {
    for (int i = 0; i <= j; ++i) {
      double sum = G[1 + i][1 + j];
      for (int k = 0; k < i; ++k) sum -= R[k][i] * R[k][j];
      if (i == j) {
        // constraint sensitivities linearly dependent (to rounding)
        if (!(sum > 1e-12 * G[1 + i][1 + i])) return CELL_EINVAL;
        R[i][i] = std::sqrt(sum);
      } else {
        R[i][j] = sum / R[i][i];
      }
    }
  }
  for (int j = 0; j < N; ++j) {   // upper-triangular inverse, column by column
    Ri[j][j] = 1.0 / R[j][j];
    for (int i = j - 1; i >= 0; --i) {
      double sum = 0.0;
      for (int k = i + 1; k <= j; ++k) sum += R[i][k] * Ri[k][j];
      Ri[i][j] = -sum / R[i][i];
    }
  }
  // p_k = <g_J, theta_k> with theta_k = sum_i Ri[i][k] g_i
  double pk[kMaxVec] = {}, mu[kMaxVec] = {}, t[kMaxVec] = {};
  double pn2 = G[0][0];
  for (int k = 0; k < N; ++k) {
    for (int i = 0; i <= k; ++i) pk[k] += Ri[i][k] * G[0][1 + i];
    pn2 -= pk[k] * pk[k];
  }
  // R^T mu = w_C C (forward substitution)
  for (int i = 0; i < N; ++i) {
    double sum = wC * C[i];
    for (int k = 0; k < i; ++k) sum -= R[k][i] * mu[k];
    mu[i] = sum / R[i][i];
  }
  const double nP = pn2 > 0.0 ? std::sqrt(pn2) : 0.0;
  const double cJ = nP > 1e-14 * std::sqrt(std::max(G[0][0], 0.0)) && nP > 0.0 ? wJ / nP : 0.0;
  for (int k = 0; k < N; ++k) t[k] = mu[k] - cJ * pk[k];
  Coef co{};
  co.c[0] = cJ;
  for (int i = 0; i < N; ++i) {
    double c = 0.0;
    for (int k = i; k < N; ++k) c += Ri[i][k] * t[k];
    co.c[1 + i] = c;
  }
  note_launch(), k_lincomb_vec<<<nb, kB, 0, s>>>(x, co, nvec, nn, v);
  if (info) {
    info[0] = nP;
    info[1] = iters;
    for (int i = 0; i < N; ++i) info[2 + i] = mu[i];
  }
  e = cudaGetLastError();
  return e == cudaSuccess ? CELL_OK : CELL_ECUDA;
}

}  // namespace cell
