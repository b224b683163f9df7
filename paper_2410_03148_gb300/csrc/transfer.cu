// Grid transfers of the geometric multigrid on rediscretised levels (mm2
// materials): trilinear interpolation between periodic grids of any ratio up
// to 2 per axis, its transpose, coarse element scales and diagonals.
#include "kernels.cuh"

namespace cell {

namespace {

constexpr int kB = 256;
inline unsigned nblocks(i64 n) { return (unsigned)((n + kB - 1) / kB); }

// Fine node i of nf lies at i nc / nf in coarse spacings: coarse nodes i0 and
// i0 + 1 with weights 1 - w and w.
template <typename T>
__device__ __forceinline__ void interp(int i, int nf, int nc, int& i0, int& i1, T& w) {
  const int t = (int)((i64)i * nc / nf);
  w = (T)((i64)i * nc - (i64)t * nf) / (T)nf;
  i0 = t;
  i1 = t + 1 == nc ? 0 : t + 1;
}

// Fine nodes that interpolate from coarse node I: lo .. lo + cnt - 1 (not yet
// wrapped), at most 4, node i with weight 1 - |i nc - I nf| / nf.
__device__ __forceinline__ void support(int I, int nf, int nc, int& lo, int& cnt) {
  if (nf == nc) {
    lo = I;
    cnt = 1;
    return;
  }
  const i64 a = (i64)(I - 1) * nf;                     // open interval (a, b) / nc
  const i64 b = (i64)(I + 1) * nf;
  const i64 fl = a >= 0 ? a / nc : -((-a + nc - 1) / nc);
  lo = (int)fl + 1;
  cnt = (int)((b + nc - 1) / nc) - lo;
}
template <typename T>
__device__ __forceinline__ T weight(int i, int I, int nf, int nc) {
  const i64 d = (i64)i * nc - (i64)I * nf;
  return T(1) - (T)(d < 0 ? -d : d) / (T)nf;
}
__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <typename T, int NC>
__global__ void __launch_bounds__(kB)
k_prolong(const T* __restrict__ xc, i64 cs, T* __restrict__ xf, i64 fs, const GridPair g, const int* active) {
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const int nx = g.nf[0], ny = g.nf[1];
  const i64 nfn = (i64)nx * ny * g.nf[2], ncn = (i64)g.nc[0] * g.nc[1] * g.nc[2];
  const i64 f = (i64)blockIdx.x * kB + threadIdx.x;
  if (f >= nfn) return;
  const int i = (int)(f % nx), j = (int)((f / nx) % ny), k = (int)(f / ((i64)nx * ny));
  int x[2], y[2], z[2];
  T wx, wy, wz;
  interp(i, nx, g.nc[0], x[0], x[1], wx);
  interp(j, ny, g.nc[1], y[0], y[1], wy);
  interp(k, g.nf[2], g.nc[2], z[0], z[1], wz);
  T acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = T(0);
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const T w = ((a & 1) ? wx : T(1) - wx) * ((a & 2) ? wy : T(1) - wy) * ((a & 4) ? wz : T(1) - wz);
    if (w == T(0)) continue;
    const i64 m = x[a & 1] + (i64)g.nc[0] * (y[(a >> 1) & 1] + (i64)g.nc[1] * z[a >> 2]);
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = fma(w, __ldg(xc + q * cs + c * ncn + m), acc[c]);
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) xf[q * fs + c * nfn + f] += acc[c];
}

// Halved axes: one thread takes the 2 x 2 x 2 fine nodes above one coarse
// node, 8 coarse values for 8 fine ones, the pairs along x as one access.
template <typename T> struct Vec2;
template <> struct Vec2<float> { typedef float2 type; };
template <> struct Vec2<double> { typedef double2 type; };

template <typename T, int NC>
__global__ void __launch_bounds__(kB)
k_prolong2(const T* __restrict__ xc, i64 cs, T* __restrict__ xf, i64 fs, const GridPair g, const int* active) {
  typedef typename Vec2<T>::type V2;
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const int cx = g.nc[0], cy = g.nc[1], cz = g.nc[2];
  const i64 ncn = (i64)cx * cy * cz, nfn = 8 * ncn;
  const i64 m = (i64)blockIdx.x * kB + threadIdx.x;
  if (m >= ncn) return;
  const int I = (int)(m % cx), J = (int)((m / cx) % cy), K = (int)(m / ((i64)cx * cy));
  const int I1 = I + 1 == cx ? 0 : I + 1, J1 = J + 1 == cy ? 0 : J + 1, K1 = K + 1 == cz ? 0 : K + 1;
  const i64 r00 = (i64)cx * (J + (i64)cy * K), r10 = (i64)cx * (J1 + (i64)cy * K), r01 = (i64)cx * (J + (i64)cy * K1),
            r11 = (i64)cx * (J1 + (i64)cy * K1);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const T* C = xc + q * cs + c * ncn;
    // sums along x of the four coarse rows: at the node, and the mean with its right neighbour
    T e[4], o[4];
    const i64 rr[4] = {r00, r10, r01, r11};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const T a = __ldg(C + rr[t] + I), b = __ldg(C + rr[t] + I1);
      e[t] = a;
      o[t] = T(0.5) * (a + b);
    }
    T* F = xf + q * fs + c * nfn + 2 * I + (i64)(2 * cx) * (2 * J + (i64)(2 * cy) * (2 * K));
    const i64 sy = 2 * cx, sz = (i64)4 * cx * cy;
    auto add = [](T* p, T a, T b) {
      V2 v = *reinterpret_cast<V2*>(p);
      v.x += a;
      v.y += b;
      *reinterpret_cast<V2*>(p) = v;
    };
    add(F, e[0], o[0]);
    add(F + sy, T(0.5) * (e[0] + e[1]), T(0.5) * (o[0] + o[1]));
    add(F + sz, T(0.5) * (e[0] + e[2]), T(0.5) * (o[0] + o[2]));
    add(F + sz + sy, T(0.25) * ((e[0] + e[1]) + (e[2] + e[3])), T(0.25) * ((o[0] + o[1]) + (o[2] + o[3])));
  }
}

template <typename T, int NC>
__global__ void __launch_bounds__(kB)
k_restrict_g(const T* __restrict__ rf, i64 rs, T* __restrict__ bc, i64 cs, const GridPair g, const int* active) {
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const int cx = g.nc[0], cy = g.nc[1];
  const i64 ncn = (i64)cx * cy * g.nc[2], nfn = (i64)g.nf[0] * g.nf[1] * g.nf[2];
  const i64 m = (i64)blockIdx.x * kB + threadIdx.x;
  if (m >= ncn) return;
  const int I = (int)(m % cx), J = (int)((m / cx) % cy), K = (int)(m / ((i64)cx * cy));
  int x0, nx, y0, ny, z0, nz;
  support(I, g.nf[0], cx, x0, nx);
  support(J, g.nf[1], cy, y0, ny);
  support(K, g.nf[2], g.nc[2], z0, nz);
  T acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = T(0);
  for (int dz = 0; dz < nz; ++dz) {
    const T wz = weight<T>(z0 + dz, K, g.nf[2], g.nc[2]);
    const i64 oz = (i64)wrap(z0 + dz, g.nf[2]) * g.nf[1];
    for (int dy = 0; dy < ny; ++dy) {
      const T wy = wz * weight<T>(y0 + dy, J, g.nf[1], cy);
      const i64 oy = (oz + wrap(y0 + dy, g.nf[1])) * g.nf[0];
#pragma unroll
      for (int dx = 0; dx < 4; ++dx) {
        if (dx >= nx) break;
        const T w = wy * weight<T>(x0 + dx, I, g.nf[0], cx);
        const i64 f = oy + wrap(x0 + dx, g.nf[0]);
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = fma(w, __ldg(rf + q * rs + c * nfn + f), acc[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) bc[q * cs + c * ncn + m] = acc[c];
}

// Halved axes: weights 1/2, 1, 1/2 at compile time, all 27 loads in flight.
template <typename T, int NC>
__global__ void __launch_bounds__(kB)
k_restrict2(const T* __restrict__ rf, i64 rs, T* __restrict__ bc, i64 cs, const GridPair g, const int* active) {
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const int cx = g.nc[0], cy = g.nc[1], cz = g.nc[2];
  const i64 ncn = (i64)cx * cy * cz, nfn = 8 * ncn;
  const i64 m = (i64)blockIdx.x * kB + threadIdx.x;
  if (m >= ncn) return;
  const int I = (int)(m % cx), J = (int)((m / cx) % cy), K = (int)(m / ((i64)cx * cy));
  const int nx = 2 * cx, ny = 2 * cy, nz = 2 * cz;
  const int xs[3] = {I == 0 ? nx - 1 : 2 * I - 1, 2 * I, 2 * I + 1};
  const i64 ys[3] = {(i64)(J == 0 ? ny - 1 : 2 * J - 1) * nx, (i64)2 * J * nx, (i64)(2 * J + 1) * nx};
  const i64 nxy = (i64)nx * ny;
  const i64 zs[3] = {(i64)(K == 0 ? nz - 1 : 2 * K - 1) * nxy, (i64)2 * K * nxy, (i64)(2 * K + 1) * nxy};
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const T* R = rf + q * rs + c * nfn;
    T acc = T(0);
#pragma unroll
    for (int z = 0; z < 3; ++z) {
      T sz = T(0);
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        const T* p = R + zs[z] + ys[y];
        const T t = fma(T(0.5), __ldg(p + xs[0]) + __ldg(p + xs[2]), __ldg(p + xs[1]));
        sz = y == 1 ? sz + t : fma(T(0.5), t, sz);
      }
      acc = z == 1 ? acc + sz : fma(T(0.5), sz, acc);
    }
    bc[q * cs + c * ncn + m] = acc;
  }
}

template <typename T>
__global__ void __launch_bounds__(kB) k_rho_coarse(const T* __restrict__ rf, T* __restrict__ rc, const GridPair g) {
  const int cx = g.nc[0], cy = g.nc[1];
  const i64 ncn = (i64)cx * cy * g.nc[2];
  const i64 m = (i64)blockIdx.x * kB + threadIdx.x;
  if (m >= ncn) return;
  const int at[3] = {(int)(m % cx), (int)((m / cx) % cy), (int)(m / ((i64)cx * cy))};
  // fine elements [e, e + 1] nc that overlap the coarse one [I, I + 1] nf
  int lo[3], hi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lo[d] = (int)((i64)at[d] * g.nf[d] / g.nc[d]);
    hi[d] = (int)(((i64)(at[d] + 1) * g.nf[d] - 1) / g.nc[d]);
  }
  auto part = [&](int d, int e) {   // share of the coarse element's length
    const i64 a = max((i64)e * g.nc[d], (i64)at[d] * g.nf[d]);
    const i64 b = min((i64)(e + 1) * g.nc[d], (i64)(at[d] + 1) * g.nf[d]);
    return (T)(b - a) / (T)g.nf[d];
  };
  T acc = T(0);
  for (int z = lo[2]; z <= hi[2]; ++z) {
    const T wz = part(2, z);
    for (int y = lo[1]; y <= hi[1]; ++y) {
      const T wy = wz * part(1, y);
      for (int x = lo[0]; x <= hi[0]; ++x)
        acc = fma(wy * part(0, x), __ldg(rf + x + (i64)g.nf[0] * (y + (i64)g.nf[1] * z)), acc);
    }
  }
  rc[m] = acc;
}

template <typename T>
__global__ void __launch_bounds__(kB) k_dinv(const T* __restrict__ rho, T* __restrict__ dinv, int nx, int ny, int nz) {
  const i64 nxy = (i64)nx * ny, nn = nxy * nz;
  const i64 n = (i64)blockIdx.x * kB + threadIdx.x;
  if (n >= nn) return;
  const int i = (int)(n % nx), j = (int)((n / nx) % ny), k = (int)(n / nxy);
  const int xs[2] = {i == 0 ? nx - 1 : i - 1, i};
  const i64 ys[2] = {(i64)(j == 0 ? ny - 1 : j - 1) * nx, (i64)j * nx};
  const i64 zs[2] = {(i64)(k == 0 ? nz - 1 : k - 1) * nxy, (i64)k * nxy};
  T s = T(0);
#pragma unroll
  for (int o = 0; o < 8; ++o) s += __ldg(rho + xs[o & 1] + ys[(o >> 1) & 1] + zs[o >> 2]);
  dinv[n] = s > T(0) ? T(1) / s : T(0);
}

template <typename T, int NC>
__global__ void __launch_bounds__(kB)
k_scale0(const T* __restrict__ b, i64 bs, T* __restrict__ x, i64 xs, const T* __restrict__ dinv, T d0, T d1, T d2,
         const T* __restrict__ c0, i64 nn, const int* active) {
  const int q = blockIdx.y;
  if (active && !active[q]) return;
  const i64 n = (i64)blockIdx.x * kB + threadIdx.x;
  if (n >= nn) return;
  const T dk[3] = {d0, d1, d2};
  const T di = dinv[n], c = *c0;
#pragma unroll
  for (int k = 0; k < NC; ++k) x[q * xs + k * nn + n] = c * dk[k] * di * b[q * bs + k * nn + n];
}

bool halved(const GridPair& g) {
  return g.nf[0] == 2 * g.nc[0] && g.nf[1] == 2 * g.nc[1] && g.nf[2] == 2 * g.nc[2];
}

}  // namespace

template <typename T, int NC>
void mg_prolong(const T* xc, i64 cs, T* xf, i64 fs, const GridPair& g, int nrhs, const int* active, cudaStream_t s) {
  // pairs along x: the fine rows are even; base and load stride too
  if (halved(g) && fs % 2 == 0 && ((uintptr_t)xf % (2 * sizeof(T))) == 0) {
    const i64 ncn = (i64)g.nc[0] * g.nc[1] * g.nc[2];
    note_launch(), k_prolong2<T, NC><<<dim3(nblocks(ncn), nrhs), kB, 0, s>>>(xc, cs, xf, fs, g, active);
    return;
  }
  const i64 nfn = (i64)g.nf[0] * g.nf[1] * g.nf[2];
  note_launch(), k_prolong<T, NC><<<dim3(nblocks(nfn), nrhs), kB, 0, s>>>(xc, cs, xf, fs, g, active);
}
template <typename T, int NC>
void mg_restrict(const T* rf, i64 rs, T* bc, i64 cs, const GridPair& g, int nrhs, const int* active, cudaStream_t s) {
  const i64 ncn = (i64)g.nc[0] * g.nc[1] * g.nc[2];
  const dim3 grid(nblocks(ncn), nrhs);
  if (halved(g)) note_launch(), k_restrict2<T, NC><<<grid, kB, 0, s>>>(rf, rs, bc, cs, g, active);
  else note_launch(), k_restrict_g<T, NC><<<grid, kB, 0, s>>>(rf, rs, bc, cs, g, active);
}
template <typename T>
void mg_rho(const T* rf, T* rc, const GridPair& g, cudaStream_t s) {
  note_launch(), k_rho_coarse<T><<<nblocks((i64)g.nc[0] * g.nc[1] * g.nc[2]), kB, 0, s>>>(rf, rc, g);
}
template <typename T>
void mg_dinv(const T* rho, T* dinv, int nx, int ny, int nz, cudaStream_t s) {
  note_launch(), k_dinv<T><<<nblocks((i64)nx * ny * nz), kB, 0, s>>>(rho, dinv, nx, ny, nz);
}
template <typename T, int NC>
void mg_scale(const T* b, i64 bs, T* x, i64 xs, const T* dinv, const T* dk, const T* c0, i64 nn, int nrhs,
              const int* active, cudaStream_t s) {
  note_launch(), k_scale0<T, NC><<<dim3(nblocks(nn), nrhs), kB, 0, s>>>(b, bs, x, xs, dinv, dk[0], dk[1], dk[2], c0,
                                                                       nn, active);
}

#define INST(T, NC)                                                                                                  \
  template void mg_prolong<T, NC>(const T*, i64, T*, i64, const GridPair&, int, const int*, cudaStream_t);           \
  template void mg_restrict<T, NC>(const T*, i64, T*, i64, const GridPair&, int, const int*, cudaStream_t);          \
  template void mg_scale<T, NC>(const T*, i64, T*, i64, const T*, const T*, const T*, i64, int, const int*, cudaStream_t);
INST(float, 1)
INST(float, 3)
INST(double, 1)
INST(double, 3)
#undef INST
template void mg_rho<float>(const float*, float*, const GridPair&, cudaStream_t);
template void mg_rho<double>(const double*, double*, const GridPair&, cudaStream_t);
template void mg_dinv<float>(const float*, float*, int, int, int, cudaStream_t);
template void mg_dinv<double>(const double*, double*, int, int, int, cudaStream_t);

}  // namespace cell
