// Modal element operators in FP64.
#include "modal_launch.cuh"

namespace cell {


template <>
void modal_full<double>(const ModalArgs<double>& a, const ModalMat<double, 4, 4>& K, int mode, cudaStream_t s) {
  if (mode == MM_APPLY) modal::launch<MK_FULL, MM_APPLY, 2, 2, false, double>(a, K, s);
  else modal::launch<MK_FULL, MM_RESID, 2, 2, false, double>(a, K, s);
}

template <>
void modal_pu<double>(const ModalArgs<double>& a, const ModalMat<double, 1, 3>& K, int, cudaStream_t s) {
  modal::launch<MK_PU, MM_ADD, 4, 2, false, double>(a, K, s);
}

template <>
void modal_uu<double>(const ModalArgs<double>& a, const ModalMat<double, 3, 3>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: modal::launch<MK_UU, MM_APPLY, 2, 2, false, double>(a, K, s); break;
    case MM_RESID: modal::launch<MK_UU, MM_RESID, 2, 2, false, double>(a, K, s); break;
    case MM_STEP: modal::launch<MK_UU, MM_STEP, 2, 2, false, double>(a, K, s); break;
    case MM_STEP0: modal::launch<MK_UU, MM_STEP0, 2, 2, false, double>(a, K, s); break;
    case MM_PRE: modal::launch<MK_UU, MM_PRE, 2, 2, false, double>(a, K, s); break;
    default: modal::launch<MK_UU, MM_POST, 2, 2, false, double>(a, K, s); break;
  }
}

template <>
void modal_ss<double>(const ModalArgs<double>& a, const ModalSch<double>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: modal::launch<MK_SS, MM_APPLY, 4, 3, false, double>(a, K, s); break;
    case MM_RESID: modal::launch<MK_SS, MM_RESID, 4, 3, false, double>(a, K, s); break;
    case MM_STEP: modal::launch<MK_SS, MM_STEP, 4, 3, false, double>(a, K, s); break;
    case MM_STEP0: modal::launch<MK_SS, MM_STEP0, 4, 3, false, double>(a, K, s); break;
    case MM_PRE: modal::launch<MK_SS, MM_PRE, 4, 3, false, double>(a, K, s); break;
    default: modal::launch<MK_SS, MM_POST, 4, 3, false, double>(a, K, s); break;
  }
}

}  // namespace cell
