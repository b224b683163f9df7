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

template <>
void modal_pu<float>(const ModalArgs<float>& a, const ModalMat<float, 1, 3>& K, int, cudaStream_t s) {
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

template <>
void modal_ss<float>(const ModalArgs<float>& a, const ModalSch<float>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: modal::launch<MK_SS, MM_APPLY, 4, 5, true, float>(a, K, s); break;
    case MM_RESID: modal::launch<MK_SS, MM_RESID, 4, 5, true, float>(a, K, s); break;
    case MM_STEP: modal::launch<MK_SS, MM_STEP, 4, 5, true, float>(a, K, s); break;
    case MM_STEP0: modal::launch<MK_SS, MM_STEP0, 4, 5, true, float>(a, K, s); break;
    case MM_PRE: modal::launch<MK_SS, MM_PRE, 4, 5, true, float>(a, K, s); break;
    default: modal::launch<MK_SS, MM_POST, 4, 5, true, float>(a, K, s); break;
  }
}

}  // namespace cell
