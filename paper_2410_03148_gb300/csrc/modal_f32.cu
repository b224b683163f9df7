// Modal element operators in FP32.
#include "modal_launch.cuh"

namespace cell {

namespace modal {
int sm_count() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  int v = cache[dev].load(std::memory_order_relaxed);
  if (!v) {
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 152;
    cache[dev].store(v, std::memory_order_relaxed);
  }
  return v;
}
}  // namespace modal

template <>
void modal_full<float>(const ModalArgs<float>& a, const ModalMat<float, 4, 4>& K, cudaStream_t s) {
  modal::launch<MK_FULL, MM_APPLY, 3, 2, true, float>(a, K, s);
}

// Element rows per warp (RE) and blocks per SM, measured with 9 loads at 128^3 /
// 64^3 / 16^3 (us).  Coupled operator: RE 3, 2 blocks 265 / 45 / 6.3; RE 2, 3
// blocks 291 / 47 / 6.3; RE 4, 2 blocks (no registers for the prefetch) 356 / 43.
// Elastic step: RE 2, 3 blocks 282 / 46 / 6.2; RE 4, 2 blocks 291 / 45 / 6.3; RE 3,
// 2 blocks 314 / 52; RE 1, 4 blocks 353 / 53.  Sbar step: RE 3, 6 blocks 111 /
// 18.6 / 4.2; RE 2, 6 blocks 127 / 20.6; RE 4, 5 blocks 113 / 20.6 / 6.2.  Coupling:
// RE 4, 4 blocks 125 / 20.6; RE 3, 4 blocks 196 / 25.  (Strips of single warps,
// each with its own halo element row, took 318 / 51, 286 / 46, 113 / 18.5 and
// 142 / 22.6.)  What is left: about 60 % issue use with 8 to 12 warps per SM, and
// 45 % of the instructions are not arithmetic (addresses, constant loads,
// shuffles); the elastic step's bytes alone would take 150 us at 128^3.
template <>
void modal_pu<float>(const ModalArgs<float>& a, const ModalMat<float, 1, 3>& K, cudaStream_t s) {
  modal::launch<MK_PU, MM_ADD, 4, 4, false, float>(a, K, s);
}

template <>
void modal_uu<float>(const ModalArgs<float>& a, const ModalMat<float, 3, 3>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: modal::launch<MK_UU, MM_APPLY, 2, 3, true, float>(a, K, s); break;
    case MM_RESID: modal::launch<MK_UU, MM_RESID, 2, 3, true, float>(a, K, s); break;
    case MM_STEP: modal::launch<MK_UU, MM_STEP, 2, 3, true, float>(a, K, s); break;
    case MM_STEP0: modal::launch<MK_UU, MM_STEP0, 2, 3, true, float>(a, K, s); break;
    case MM_PRE: modal::launch<MK_UU, MM_PRE, 2, 3, true, float>(a, K, s); break;
    default: modal::launch<MK_UU, MM_POST, 2, 3, true, float>(a, K, s); break;
  }
}

namespace {
// Sbar: six element rows per warp from 4e6 node values on (128^3 x 9: 93 us
// against 111 for three rows, 64^3 x 9 18.5 / 18.6, 32^3 x 9 8.2 / 6.3).
template <int MODE>
void go_ss(const ModalArgs<float>& a, const ModalSch<float>& K, cudaStream_t s) {
  if ((i64)a.nx * a.ny * a.nz * a.nrhs >= 4000000) modal::launch<MK_SS, MODE, 6, 4, true, float>(a, K, s);
  else modal::launch<MK_SS, MODE, 3, 6, true, float>(a, K, s);
}
}  // namespace

template <>
void modal_ss<float>(const ModalArgs<float>& a, const ModalSch<float>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: go_ss<MM_APPLY>(a, K, s); break;
    case MM_RESID: go_ss<MM_RESID>(a, K, s); break;
    case MM_STEP: go_ss<MM_STEP>(a, K, s); break;
    case MM_STEP0: go_ss<MM_STEP0>(a, K, s); break;
    case MM_PRE: go_ss<MM_PRE>(a, K, s); break;
    default: go_ss<MM_POST>(a, K, s); break;
  }
}

}  // namespace cell
