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
void modal_full<float>(const ModalArgs<float>& a, const ModalMat<float, 4, 4>& K, int, cudaStream_t s) {
  modal::launch<MK_FULL, MM_APPLY, 3, 2, true, float>(a, K, s);
}

// Rows per strip and blocks per SM, measured with 9 loads at 128^3 / 64^3 / 16^3
// (us).  Coupled operator: 3 rows, 2 blocks 321 / 53 / 8.2; 2 rows, 2 blocks
// 341 / 55 / 8.2; 1 row, 3 blocks 521 / 72 / 8.2.  Elastic step: 3 rows, 2
// blocks 290 / 47 / 6.3 (255 registers); 2 rows, 3 blocks 424 / 66 / 8.2 (spills
// at 168 registers); 1 row, 4 blocks 384 / 60 / 6.3.  Sbar step: 2 rows, 6
// blocks 113 / 18.7 / 6.1; 3 rows, 5 blocks 111 / 20.3; 4 rows, 5 blocks 177 /
// 22.7 / 6.3.  Coupling: 4 rows, 4 blocks 143 / 24.6 / 6.3; 3 rows 153 / 22.8.
// What is left: 128^3 runs at 60 % issue use with 8 warps per SM, 45 % of the
// instructions are not arithmetic (addresses, constant loads, shuffles).
template <>
void modal_pu<float>(const ModalArgs<float>& a, const ModalMat<float, 1, 3>& K, int, cudaStream_t s) {
  modal::launch<MK_PU, MM_ADD, 4, 4, false, float>(a, K, s);
}

template <>
void modal_uu<float>(const ModalArgs<float>& a, const ModalMat<float, 3, 3>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: modal::launch<MK_UU, MM_APPLY, 3, 2, true, float>(a, K, s); break;
    case MM_RESID: modal::launch<MK_UU, MM_RESID, 3, 2, true, float>(a, K, s); break;
    case MM_STEP: modal::launch<MK_UU, MM_STEP, 3, 2, true, float>(a, K, s); break;
    case MM_STEP0: modal::launch<MK_UU, MM_STEP0, 3, 2, true, float>(a, K, s); break;
    case MM_PRE: modal::launch<MK_UU, MM_PRE, 3, 2, true, float>(a, K, s); break;
    default: modal::launch<MK_UU, MM_POST, 3, 2, true, float>(a, K, s); break;
  }
}

template <>
void modal_ss<float>(const ModalArgs<float>& a, const ModalSch<float>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: modal::launch<MK_SS, MM_APPLY, 2, 6, true, float>(a, K, s); break;
    case MM_RESID: modal::launch<MK_SS, MM_RESID, 2, 6, true, float>(a, K, s); break;
    case MM_STEP: modal::launch<MK_SS, MM_STEP, 2, 6, true, float>(a, K, s); break;
    case MM_STEP0: modal::launch<MK_SS, MM_STEP0, 2, 6, true, float>(a, K, s); break;
    case MM_PRE: modal::launch<MK_SS, MM_PRE, 2, 6, true, float>(a, K, s); break;
    default: modal::launch<MK_SS, MM_POST, 2, 6, true, float>(a, K, s); break;
  }
}

}  // namespace cell
