// Inverse of the coarsest multigrid level on the device (rediscretised
// hierarchies): assembly from the element scales, FP32 Gauss-Jordan in the
// registers of one block, two Newton-Schulz steps X <- X (2 I - A X) in FP64
// over the whole chip.  The FP64 factorisation of the default coarsest level
// (192 unknowns) takes 5 ms per design on the host, more than an 8^3 design step.
// FP64 elimination in one block would take 1.7 ms (n^3 multiply-adds at two per
// clock); the FP32 one takes 0.17 ms (0.9 us a pivot, bound by its chain of
// barrier, shared-memory reads and update) and Newton-Schulz (Schulz 1933)
// squares its residual.
#include "kernels.cuh"

namespace cell {

namespace {

constexpr int kTile = 7;                 // register tile of a thread: kTile x kTile
constexpr int kMaxN = 32 * kTile;        // 224 unknowns
// Largest max |I - A X| before the last Newton step whose result is kept.  The
// step leaves (I - A X)^2, entries of at most n times the square: 2^-53 for an
// FP64 inverse, 2^-26 for one that is stored in FP32.  Designs reach 1e-12 at
// contrasts of 1e-3 and about 1e-9 at 1e-8; beyond, the host factorises in FP64.
constexpr double kAccept64 = 7e-10, kAccept32 = 8e-6;
static_assert(kMaxN * kAccept64 * kAccept64 < 1.2e-16 && kMaxN * kAccept32 * kAccept32 < 1.5e-8, "accepted residual");

// Row (i, c) of A = sum_e rho_e P_e^T K P_e: block = row, thread = column.  On
// 2-node axes a node is several corners of one element: all matches count.
template <typename T>
__global__ void k_dense_rows(const T* __restrict__ rho, const double* __restrict__ K, int nc, int nx, int ny, int nz,
                             double* __restrict__ A) {
  const int nn = nx * ny * nz, n = nc * nn, R = 8 * nc;
  const int row = blockIdx.x, c = row / nn, p = row % nn;
  const int i = p % nx, j = (p / nx) % ny, k = p / (nx * ny);
  for (int col = threadIdx.x; col < n; col += blockDim.x) {
    const int d = col / nn, m = col % nn;
    double v = 0.0;
    for (int o = 0; o < 8; ++o) {   // element at (i - 1 + ex, ..), local corner of the row's node
      const int ei = (i - 1 + (o & 1) + nx) % nx, ej = (j - 1 + ((o >> 1) & 1) + ny) % ny,
                ek = (k - 1 + (o >> 2) + nz) % nz;
      const int la = 7 - o;
      double s = 0.0;
      for (int b = 0; b < 8; ++b) {
        const int node = (ei + (b & 1)) % nx + nx * ((ej + ((b >> 1) & 1)) % ny + ny * ((ek + (b >> 2)) % nz));
        if (node == m) s += K[(la * nc + c) * R + b * nc + d];
      }
      v += s * (double)rho[ei + nx * (ej + ny * ek)];
    }
    A[(size_t)row * n + col] = v;
  }
}

// Null-space regularisation (mean of every component, scaled by the mean
// diagonal) and X = A^-1 in FP32: in-place Gauss-Jordan without pivoting (A is
// symmetric positive definite), a 32 x 32 block of threads with entry
// (ty + 32 a, tx + 32 b) in register (a, b), TILE = ceil(n / 32).  The pivot row
// and column of the next step are written to the other buffer right after the
// update, so a step has one barrier.
template <int TILE>
__global__ void __launch_bounds__(1024, 1)
k_dense_invert(double* __restrict__ A, double* __restrict__ X, int n, int nn) {
  __shared__ float row[2][32 * TILE], col[2][32 * TILE];
  __shared__ double mean;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (ty == 0) {
    double tr = 0.0;
    for (int i = tx; i < n; i += 32) tr += A[(size_t)i * n + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (tx == 0) mean = tr / n / nn;
  }
  __syncthreads();
  float a[TILE][TILE];
#pragma unroll
  for (int p = 0; p < TILE; ++p)
#pragma unroll
    for (int q = 0; q < TILE; ++q) {
      const int i = ty + 32 * p, j = tx + 32 * q;
      a[p][q] = 0.f;
      if (i < n && j < n) {
        double v = A[(size_t)i * n + j];
        if (i / nn == j / nn) {
          v += mean;
          A[(size_t)i * n + j] = v;
        }
        a[p][q] = (float)v;
      }
    }
  // Pivot row and column into shared memory; their registers are cleared and
  // the pivot's entries set to 1 (row) and -1 (column), so that the rank-1
  // update a - f r gives every case: the pivot row becomes r, the pivot column
  // -f piv, the pivot piv.
  __shared__ float pivot[2];
  auto publish = [&](int k) {
    const int kt = k & 31, kb = k >> 5;
    float* rk = row[k & 1];
    float* ck = col[k & 1];
    if (ty == kt) {
#pragma unroll
      for (int p = 0; p < TILE; ++p)
        if (p == kb) {
#pragma unroll
          for (int q = 0; q < TILE; ++q) {
            if (q == kb && tx == kt) {
              pivot[k & 1] = a[p][q];
              rk[tx + 32 * q] = 1.f;
            } else {
              rk[tx + 32 * q] = a[p][q];
            }
            a[p][q] = 0.f;
          }
        }
    }
    if (tx == kt) {
#pragma unroll
      for (int q = 0; q < TILE; ++q)
        if (q == kb) {
#pragma unroll
          for (int p = 0; p < TILE; ++p) {
            // the pivot row's owner has cleared its register already
            ck[ty + 32 * p] = p == kb && ty == kt ? -1.f : a[p][q];
            a[p][q] = 0.f;
          }
        }
    }
  };
  publish(0);
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const float* rk = row[k & 1];
    const float* ck = col[k & 1];
    const float piv = 1.f / pivot[k & 1];
    float r[TILE];
#pragma unroll
    for (int q = 0; q < TILE; ++q) r[q] = rk[tx + 32 * q] * piv;
#pragma unroll
    for (int p = 0; p < TILE; ++p) {
      const float f = -ck[ty + 32 * p];
#pragma unroll
      for (int q = 0; q < TILE; ++q) a[p][q] = fmaf(f, r[q], a[p][q]);
    }
    if (k + 1 < n) publish(k + 1);
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < TILE; ++p)
#pragma unroll
    for (int q = 0; q < TILE; ++q) {
      const int i = ty + 32 * p, j = tx + 32 * q;
      if (i < n && j < n) X[(size_t)i * n + j] = (double)a[p][q];
    }
}

// C = A B (sub = 0) with max |I - C| in *dev as float bits, or C = 2 A - A B
// (sub = 1, written as T into out too).  Tiles of 16 x 16.
template <typename T>
__global__ void __launch_bounds__(256)
k_dense_mul(const double* __restrict__ A, const double* __restrict__ B, double* __restrict__ C, int n, int sub,
            T* __restrict__ out, unsigned* __restrict__ dev) {
  __shared__ double sa[16][17], sb[16][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i = blockIdx.y * 16 + ty, j = blockIdx.x * 16 + tx;
  double s = 0.0;
  for (int k0 = 0; k0 < n; k0 += 16) {
    sa[ty][tx] = i < n && k0 + tx < n ? A[(size_t)i * n + k0 + tx] : 0.0;
    sb[ty][tx] = k0 + ty < n && j < n ? B[(size_t)(k0 + ty) * n + j] : 0.0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) s = fma(sa[ty][k], sb[k][tx], s);
    __syncthreads();
  }
  if (i >= n || j >= n) return;
  if (sub) {
    const double v = 2.0 * A[(size_t)i * n + j] - s;
    C[(size_t)i * n + j] = v;
    if (out) out[(size_t)i * n + j] = (T)v;
  } else {
    C[(size_t)i * n + j] = s;
    const float e = (float)fabs(s - (i == j ? 1.0 : 0.0));
    // NaN compares false against every bound: report it as infinity
    if (dev) atomicMax(dev, __float_as_uint(e == e ? e : __int_as_float(0x7f800000)));
  }
}

}  // namespace

bool dense_invert_ok(int n) { return n <= kMaxN; }
size_t dense_invert_work(int n) { return (size_t)4 * n * n; }
bool dense_invert_failed(unsigned dev_bits, bool fp64) {
  float f;
  static_assert(sizeof(f) == sizeof(dev_bits), "float bits");
  __builtin_memcpy(&f, &dev_bits, 4);
  return !(f <= (fp64 ? kAccept64 : kAccept32));
}

template <typename T>
void dense_invert(const T* rho, const double* K, int nc, int nx, int ny, int nz, double* work, T* out, unsigned* dev,
                  cudaStream_t s) {
  const int nn = nx * ny * nz, n = nc * nn;
  const size_t n2 = (size_t)n * n;
  double *A = work, *X = work + n2, *R = work + 2 * n2, *Y = work + 3 * n2;
  cudaMemsetAsync(dev, 0, sizeof(unsigned), s);
  note_launch(), k_dense_rows<T><<<n, n < 256 ? (n + 31) / 32 * 32 : 256, 0, s>>>(rho, K, nc, nx, ny, nz, A);
  note_launch();
  switch ((n + 31) / 32) {
    case 1: k_dense_invert<1><<<1, 1024, 0, s>>>(A, X, n, nn); break;
    case 2: k_dense_invert<2><<<1, 1024, 0, s>>>(A, X, n, nn); break;
    case 3: k_dense_invert<3><<<1, 1024, 0, s>>>(A, X, n, nn); break;
    case 4: k_dense_invert<4><<<1, 1024, 0, s>>>(A, X, n, nn); break;
    case 5: k_dense_invert<5><<<1, 1024, 0, s>>>(A, X, n, nn); break;
    case 6: k_dense_invert<6><<<1, 1024, 0, s>>>(A, X, n, nn); break;
    default: k_dense_invert<kTile><<<1, 1024, 0, s>>>(A, X, n, nn); break;
  }
  const dim3 g((unsigned)((n + 15) / 16), (unsigned)((n + 15) / 16));
  note_launch(), k_dense_mul<T><<<g, 256, 0, s>>>(A, X, R, n, 0, nullptr, nullptr);
  note_launch(), k_dense_mul<T><<<g, 256, 0, s>>>(X, R, Y, n, 1, nullptr, nullptr);
  note_launch(), k_dense_mul<T><<<g, 256, 0, s>>>(A, Y, R, n, 0, nullptr, dev);
  note_launch(), k_dense_mul<T><<<g, 256, 0, s>>>(Y, R, X, n, 1, out, nullptr);
}
template void dense_invert<float>(const float*, const double*, int, int, int, int, double*, float*, unsigned*,
                                  cudaStream_t);
template void dense_invert<double>(const double*, const double*, int, int, int, int, double*, double*, unsigned*,
                                   cudaStream_t);

}  // namespace cell
