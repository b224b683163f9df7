// Element operators in their modal form (included by the modal_*.cu units).
//
// On a box element the 8 corner values of a component are replaced by their
// sums and differences along the axes, u^_m with m = (x, y, z) bits, bit set =
// difference (u(1) - u(0)), clear = sum.  In this basis the Q1 element matrix
// K = H^T K^ H is sparse: it couples only modes of the same number of
// differences (one: the constant strains; two: the linear ones; three), and
// constants drop out.  For a material with the mm2 mirror planes (no
// normal-shear coupling, e only e31 e32 e33 e15 e24, diagonal kappa: poled
// ceramics on an aligned grid) it couples only dofs of equal parity under
// the three mirrors as well: 82 products for the coupled operator against
// 1024 of the corner form, 45 (of 576) for the elastic block, 7 (of 64) for
// Sbar, 15 (of 192) for the coupling block.  The transforms are shared between
// neighbours: per node and component 2 operations along x, 4 along y and 7
// along z, and 19 back.  Other materials keep the corner form (apply.cu): with
// all 304 products of the modal matrix the registers of a thread do not hold
// the modes of an element.
//
// A block owns a strip of node rows by 30 columns (lanes 1..30; lanes 0 and 31
// are halo) and marches through z; its four warps take consecutive element rows.
// x neighbours are lane shuffles, y neighbours the rows a thread holds (the row
// between two warps goes through shared memory), z neighbours registers carried
// from the plane before: no atomics, and 4 RE element rows serve 4 RE - 1 node
// rows.  The columns of all strips form one sequence of nx + 2 positions per
// strip (both periodic ends included), cut into windows of 30 outputs, so any nx
// keeps about 30/32 of the lanes busy.
#pragma once

#include "kernels.cuh"

namespace cell {
namespace modal {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kOut = 30;   // output columns of a warp

// ---- arithmetic -------------------------------------------------------------
// Value types: float, double, and DF, an unevaluated pair h + l of floats with
// error-free products and sums of the leading parts (about 2^-46).
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ DF vadd(DF a, DF b) {
  const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
  return {s, __fadd_rn(__fadd_rn(a.l, b.l), e)};
}
__device__ __forceinline__ DF vsub(DF a, DF b) { return vadd(a, DF{-b.h, -b.l}); }
__device__ __forceinline__ DF vmul(DF a, DF b) {
  const float p = __fmul_rn(a.h, b.h);
  return {p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ DF vfma(DF a, DF b, DF c) { return vadd(c, vmul(a, b)); }

__device__ __forceinline__ float vdown(float v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double vdown(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ DF vdown(DF v) { return {vdown(v.h), vdown(v.l)}; }
__device__ __forceinline__ float vup(float v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double vup(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ DF vup(DF v) { return {vup(v.h), vup(v.l)}; }

// Two values that differ in the x mode (sum, difference).  FP32 pairs use the
// packed instructions (two results per issue slot); a - b is fma(b, -1, a),
// the same rounding.
template <typename V>
struct Pair {
  V s, d;
};
template <>
struct Pair<float> {
  float2 p;
};
template <>
struct Pair<DF> {
  float2 h, l;
};
template <typename V> __device__ __forceinline__ V sum_of(const Pair<V>& a) { return a.s; }
template <typename V> __device__ __forceinline__ V dif_of(const Pair<V>& a) { return a.d; }
__device__ __forceinline__ float sum_of(const Pair<float>& a) { return a.p.x; }
__device__ __forceinline__ float dif_of(const Pair<float>& a) { return a.p.y; }
__device__ __forceinline__ DF sum_of(const Pair<DF>& a) { return {a.h.x, a.l.x}; }
__device__ __forceinline__ DF dif_of(const Pair<DF>& a) { return {a.h.y, a.l.y}; }
template <typename V> __device__ __forceinline__ Pair<V> mk(V s, V d) { return {s, d}; }
template <> __device__ __forceinline__ Pair<DF> mk<DF>(DF s, DF d) {
  return {make_float2(s.h, d.h), make_float2(s.l, d.l)};
}
template <> __device__ __forceinline__ Pair<float> mk<float>(float s, float d) { return {make_float2(s, d)}; }
template <typename V> __device__ __forceinline__ Pair<V> padd(const Pair<V>& a, const Pair<V>& b) {
  return {vadd(a.s, b.s), vadd(a.d, b.d)};
}
template <typename V> __device__ __forceinline__ Pair<V> psub(const Pair<V>& a, const Pair<V>& b) {
  return {vsub(a.s, b.s), vsub(a.d, b.d)};
}
template <typename V> __device__ __forceinline__ Pair<V> pmul(V k, const Pair<V>& a) {
  return {vmul(k, a.s), vmul(k, a.d)};
}
__device__ __forceinline__ Pair<float> padd(const Pair<float>& a, const Pair<float>& b) {
  return {__fadd2_rn(a.p, b.p)};
}
__device__ __forceinline__ Pair<float> psub(const Pair<float>& a, const Pair<float>& b) {
  return {__ffma2_rn(b.p, make_float2(-1.f, -1.f), a.p)};
}
__device__ __forceinline__ Pair<float> pmul(float k, const Pair<float>& a) {
  return {__fmul2_rn(make_float2(k, k), a.p)};
}

// The error-free sums of vadd and vsub, two at a time.
__device__ __forceinline__ float2 minus(const float2 b, const float2 a) {   // a - b
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ Pair<DF> padd(const Pair<DF>& a, const Pair<DF>& b) {
  const float2 s = __fadd2_rn(a.h, b.h), t = minus(a.h, s);
  const float2 e = __fadd2_rn(minus(minus(t, s), a.h), minus(t, b.h));
  return {s, __fadd2_rn(__fadd2_rn(a.l, b.l), e)};
}
__device__ __forceinline__ Pair<DF> psub(const Pair<DF>& a, const Pair<DF>& b) {
  const float2 s = minus(b.h, a.h), t = minus(a.h, s);
  const float2 e = minus(__fadd2_rn(b.h, t), minus(minus(t, s), a.h));
  return {s, __fadd2_rn(minus(b.l, a.l), e)};
}
__device__ __forceinline__ Pair<DF> pmul(DF k, const Pair<DF>& a) {
  const float2 kh = make_float2(k.h, k.h), kl = make_float2(k.l, k.l);
  const float2 p = __fmul2_rn(kh, a.h);
  const float2 e = __ffma2_rn(kh, a.h, make_float2(-p.x, -p.y));
  return {p, __ffma2_rn(kh, a.l, __ffma2_rn(kl, a.h, e))};
}

// ---- element contraction ------------------------------------------------------
// Coupled input dofs before the k-th (k = j NI + d) in the row of output dof
// (c, mode); two: modes of two differences (7 without axis j).
template <int NI>
__host__ __device__ constexpr int before(int c, int m, int k, bool two) {
  int n = 0;
  for (int q = 0; q < k; ++q) n += modal_couples(c, m, q % NI, two ? 7 ^ (1 << (q / NI)) : 1 << (q / NI)) ? 1 : 0;
  return n;
}

// f[c][m] = sum K^[(c,m)][(d,n)] u[d][n] within the classes of one, two and
// three differences.  CO = component of the first output row.
template <int NO, int NI, int CO, typename V>
__device__ __forceinline__ void force(const ModalMat<V, NO, NI>& K, const V (&u)[NI][8], V (&f)[NO][8]) {
#pragma unroll
  for (int c = 0; c < NO; ++c) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int m1 = 1 << i, m2 = 7 ^ m1;
      const ModalRow<V> k1 = K.c[i * NO + c], k2 = K.q[i * NO + c];
      V f1 = V{}, f2 = V{};
#pragma unroll
      for (int k = 0; k < 3 * NI; ++k) {
        const int j = k / NI, d = k % NI, n1 = 1 << j, n2 = 7 ^ n1;
        if (modal_couples(CO + c, m1, d, n1)) {
          const int at = before<NI>(CO + c, m1, k, false);
          f1 = at == 0 ? vmul(k1.v[at], u[d][n1]) : vfma(k1.v[at], u[d][n1], f1);
        }
        if (modal_couples(CO + c, m2, d, n2)) {
          const int at = before<NI>(CO + c, m2, k, true);
          f2 = at == 0 ? vmul(k2.v[at], u[d][n2]) : vfma(k2.v[at], u[d][n2], f2);
        }
      }
      f[c][m1] = f1;
      f[c][m2] = f2;
    }
    const ModalRow<V> k3 = K.t[c];
    V f3 = V{};
    int at = 0;
#pragma unroll
    for (int d = 0; d < NI; ++d)
      if (modal_couples(CO + c, 7, d, 7)) {
        f3 = at == 0 ? vmul(k3.v[at], u[d][7]) : vfma(k3.v[at], u[d][7], f3);
        ++at;
      }
    f[c][7] = f3;
  }
}
// Sbar: the three mirrors leave every mode alone, S^ is diagonal.
template <typename V>
__device__ __forceinline__ void force_s(const ModalSch<V>& K, const V (&u)[1][8], V (&f)[1][8]) {
#pragma unroll
  for (int m = 1; m < 8; ++m) f[0][m] = vmul(K.s[m], u[0][m]);
}

template <int KIND>
struct Shape;   // input and output components
template <> struct Shape<MK_FULL> { static constexpr int NI = 4, NO = 4, CO = 0; };
template <> struct Shape<MK_UU> { static constexpr int NI = 3, NO = 3, CO = 0; };
template <> struct Shape<MK_PU> { static constexpr int NI = 3, NO = 1, CO = 3; };
template <> struct Shape<MK_SS> { static constexpr int NI = 1, NO = 1, CO = 0; };

template <int KIND, typename V>
struct MatOf { typedef ModalMat<V, Shape<KIND>::NO, Shape<KIND>::NI> type; };
template <typename V>
struct MatOf<MK_SS, V> { typedef ModalSch<V> type; };

// One element row of the march: modes of the element between node rows with
// (x pair, z sum / difference) values q0 (lower) and q1, scaled by rho;
// contributions to the lower (low) and upper (up) node row.
template <int KIND, typename V>
__device__ __forceinline__ void element(const typename MatOf<KIND, V>::type& K, const Pair<V> (&q0)[Shape<KIND>::NI][2],
                                        const Pair<V> (&q1)[Shape<KIND>::NI][2], V rho,
                                        Pair<V> (&low)[Shape<KIND>::NO][2], Pair<V> (&up)[Shape<KIND>::NO][2]) {
  constexpr int NI = Shape<KIND>::NI, NO = Shape<KIND>::NO;
  V u[NI][8], f[NO][8];
#pragma unroll
  for (int d = 0; d < NI; ++d)
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const Pair<V> ys = padd(q1[d][z], q0[d][z]), yd = psub(q1[d][z], q0[d][z]);
      u[d][4 * z] = sum_of(ys);
      u[d][4 * z + 1] = dif_of(ys);
      u[d][4 * z + 2] = sum_of(yd);
      u[d][4 * z + 3] = dif_of(yd);
    }
  if constexpr (KIND == MK_SS) force_s<V>(K, u, f);
  else force<NO, NI, Shape<KIND>::CO, V>(K, u, f);
#pragma unroll
  for (int c = 0; c < NO; ++c)
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const Pair<V> fs = pmul(rho, mk<V>(z ? f[c][4] : V{}, f[c][4 * z + 1]));
      const Pair<V> fd = pmul(rho, mk<V>(f[c][4 * z + 2], f[c][4 * z + 3]));
      low[c][z] = psub(fs, fd);
      up[c][z] = padd(fs, fd);
    }
}

// ---- the march ------------------------------------------------------------------
// IO supplies the inputs and takes the outputs of one load (offsets from the
// start of a component plane):
//   V    in(d, offset)          input component d at a node
//   V    rho(offset)            element scale
//   void fetch(pre, offset)     operands of a node's output
//   void out(offset, acc, own, pre)   assembled values of the output components
//                               and the node's own inputs
//
// Block = window of 30 columns (blockIdx.x) of a strip of 4 RE - 1 node rows,
// warp w = the RE element rows from w RE.  Element row r of a warp lies between
// its node rows r and r + 1; the node row 0 of a warp also needs the last
// element row of the warp before, whose contribution comes through shared
// memory (one barrier per plane, two buffers).  Warp 0's node row 0 is the halo.
template <int KIND, typename V>
struct Exchange {
  Pair<V> p[2][kWarps][Shape<KIND>::NO][2][32];
};

template <int KIND, int RE, bool PF, typename V, typename IO>
__device__ __forceinline__ void march(const typename MatOf<KIND, V>::type& K, const IO& io, Exchange<KIND, V>& ex, int nx,
                                      int ny, int nz, int L) {
  constexpr int NI = Shape<KIND>::NI, NO = Shape<KIND>::NO;
  constexpr int S = kWarps * RE - 1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int rl = nx + 2;
  const int strips = (ny + S - 1) / S;
  const int p0 = (int)blockIdx.x * kOut;
  const int p = min(p0 + lane, strips * rl - 1);
  const int strip = p / rl;
  const int xi = p - strip * rl - 1;
  const bool vx = lane >= 1 && lane <= kOut && p0 + lane == p && xi >= 0 && xi < nx;
  const int i = xi < 0 ? nx - 1 : (xi >= nx ? 0 : xi);
  const int j0 = strip * S - 1 + w * RE;   // the warp's node row 0
  // in-plane offsets of its node rows (periodic); rows that this lane writes
  unsigned ro[RE + 1];
  bool ok[RE];
  {
    int j = j0 < 0 ? j0 + ny : j0 % ny;
#pragma unroll
    for (int r = 0; r < RE + 1; ++r) {
      ro[r] = (unsigned)(j * nx + i);
      j = j + 1 == ny ? 0 : j + 1;
    }
  }
#pragma unroll
  for (int r = 0; r < RE; ++r) ok[r] = vx && j0 + r < ny && (r > 0 || w > 0);
  const unsigned nxy = (unsigned)(nx * ny);
  const int z0 = blockIdx.z * L;
  const int Lc = min(L, nz - z0);
  Pair<V> ps[RE + 1][NI];   // x sums and differences of the plane before
  V own[RE][NI];            // its values
  Pair<V> carry[RE][NO];    // contributions of the layer below to the plane before
  unsigned zp = (unsigned)(z0 == 0 ? nz - 1 : z0 - 1) * nxy;   // the plane before
  unsigned zc = (unsigned)z0 * nxy;                             // the plane above the layer
  // the loads of the first two planes are in flight together
  V v0[RE + 1][NI], vn[PF ? RE + 1 : 1][NI], rn[PF ? RE : 1];
#pragma unroll
  for (int r = 0; r < RE + 1; ++r)
#pragma unroll
    for (int d = 0; d < NI; ++d) v0[r][d] = io.in(d, zp + ro[r]);
  if (PF) {
#pragma unroll
    for (int r = 0; r < RE + 1; ++r)
#pragma unroll
      for (int d = 0; d < NI; ++d) vn[PF ? r : 0][d] = io.in(d, zc + ro[r]);
#pragma unroll
    for (int r = 0; r < RE; ++r) rn[PF ? r : 0] = io.rho(zp + ro[r]);
  }
#pragma unroll
  for (int r = 0; r < RE + 1; ++r)
#pragma unroll
    for (int d = 0; d < NI; ++d) {
      const V u = vdown(v0[r][d]);
      ps[r][d] = mk<V>(vadd(u, v0[r][d]), vsub(u, v0[r][d]));
    }
#pragma unroll
  for (int r = 0; r < RE; ++r) {
#pragma unroll
    for (int c = 0; c < NO; ++c) carry[r][c] = mk<V>(V{}, V{});
#pragma unroll
    for (int d = 0; d < NI; ++d) own[r][d] = V{};
  }
#pragma unroll 1
  for (int t = 0; t <= Lc; ++t) {
    const unsigned zn = zc + nxy == nxy * (unsigned)nz ? 0 : zc + nxy;
    V v[RE + 1][NI], rho[RE];
    typename IO::Pre pre[RE];
    if (PF) {
#pragma unroll
      for (int r = 0; r < RE + 1; ++r)
#pragma unroll
        for (int d = 0; d < NI; ++d) {
          v[r][d] = vn[PF ? r : 0][d];
          vn[PF ? r : 0][d] = io.in(d, zn + ro[r]);
        }
#pragma unroll
      for (int r = 0; r < RE; ++r) {
        rho[r] = rn[PF ? r : 0];
        rn[PF ? r : 0] = io.rho(zc + ro[r]);
      }
    } else {
#pragma unroll
      for (int r = 0; r < RE + 1; ++r)
#pragma unroll
        for (int d = 0; d < NI; ++d) v[r][d] = io.in(d, zc + ro[r]);
#pragma unroll
      for (int r = 0; r < RE; ++r) rho[r] = io.rho(zp + ro[r]);
    }
    if (t > 0) {
#pragma unroll
      for (int r = 0; r < RE; ++r)
        if (ok[r]) io.fetch(pre[r], zp + ro[r]);
    }
    // tall strips of few warps: the next plane's operands come from DRAM to L2
    // meanwhile (Sbar step at 128^3 102 -> 93 us; no gain with more warps per SM)
    if (RE >= 6) {
#pragma unroll
      for (int r = 0; r < RE; ++r) io.prefetch(zc + ro[r]);
    }
    // output row r from its element rows' contributions
    auto emit = [&](int r, const Pair<V> (&up)[NO][2], const Pair<V> (&low)[NO][2]) {
      V acc[NO];
#pragma unroll
      for (int c = 0; c < NO; ++c) {
        const Pair<V> ts = padd(up[c][0], low[c][0]), td = padd(up[c][1], low[c][1]);
        const Pair<V> o = padd(carry[r][c], psub(ts, td));
        carry[r][c] = padd(ts, td);
        acc[c] = vadd(vsub(sum_of(o), dif_of(o)), vup(vadd(sum_of(o), dif_of(o))));
      }
      if (t > 0 && ok[r]) io.out(zp + ro[r], acc, own[r], pre[r]);
#pragma unroll
      for (int d = 0; d < NI; ++d) own[r][d] = v[r][d];
    };
    Pair<V> q0[NI][2], up[NO][2], low0[NO][2];
#pragma unroll
    for (int r = 0; r < RE + 1; ++r) {
      Pair<V> q1[NI][2];
#pragma unroll
      for (int d = 0; d < NI; ++d) {
        const V u = vdown(v[r][d]);
        const Pair<V> x = mk<V>(vadd(u, v[r][d]), vsub(u, v[r][d]));
        q1[d][0] = padd(x, ps[r][d]);
        q1[d][1] = psub(x, ps[r][d]);
        ps[r][d] = x;
      }
      if (r > 0) {
        Pair<V> low[NO][2], un[NO][2];
        element<KIND, V>(K, q0, q1, rho[r - 1], low, un);
        if (r == 1) {
#pragma unroll
          for (int c = 0; c < NO; ++c) low0[c][0] = low[c][0], low0[c][1] = low[c][1];
        } else {
          emit(r - 1, up, low);
        }
#pragma unroll
        for (int c = 0; c < NO; ++c) up[c][0] = un[c][0], up[c][1] = un[c][1];
      }
#pragma unroll
      for (int d = 0; d < NI; ++d) q0[d][0] = q1[d][0], q0[d][1] = q1[d][1];
    }
    // the last element row's upper contribution goes to the next warp
#pragma unroll
    for (int c = 0; c < NO; ++c)
#pragma unroll
      for (int z = 0; z < 2; ++z) ex.p[t & 1][w][c][z][lane] = up[c][z];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NO; ++c)
#pragma unroll
      for (int z = 0; z < 2; ++z) up[c][z] = ex.p[t & 1][w == 0 ? 0 : w - 1][c][z][lane];
    emit(0, up, low0);
    zp = zc;
    zc = zn;
  }
}

// ---- launch geometry -----------------------------------------------------------
int sm_count();   // modal_f32.cu

// Planes per chunk: the smallest waves x (planes + 2) for the blocks that the
// chip holds (a chunk evaluates one element layer and loads two node planes
// more than it writes).
inline int chunk_planes(int nz, i64 blocks, int blocks_per_sm) {
  const i64 slots = (i64)sm_count() * blocks_per_sm;
  int best = nz;
  const int most = nz < 4096 ? nz : 4096;   // grid z
  double cost = 1e300;
  for (int chunks = 1; chunks <= most;) {
    const int L = (nz + chunks - 1) / chunks;
    const i64 w = blocks * ((nz + L - 1) / L);
    const double c = (double)((w + slots - 1) / slots) * (L + 2.0);
    if (c < cost) {
      cost = c;
      best = L;
    }
    chunks = L > 1 ? (nz + L - 2) / (L - 1) : most + 1;   // the next count with shorter chunks
  }
  return best;
}

// Grid (windows, load groups, z chunks) and planes per chunk, RE element rows
// per warp.
inline dim3 grid_for(int nx, int ny, int nz, int groups, int re, int blocks_per_sm, int* L) {
  const int rows = kWarps * re - 1;
  const i64 seq = (i64)((ny + rows - 1) / rows) * (nx + 2) - 2;   // positions between the first and last halo
  const i64 windows = (seq + kOut - 1) / kOut;
  *L = chunk_planes(nz, windows * groups, blocks_per_sm);
  return dim3((unsigned)windows, (unsigned)groups, (unsigned)((nz + *L - 1) / *L));
}

}  // namespace modal
}  // namespace cell
