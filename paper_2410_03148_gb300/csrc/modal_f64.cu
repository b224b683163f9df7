// Modal element operators in FP64.
#include "modal_launch.cuh"

namespace cell {

namespace {

// FP64 arithmetic (1/64 rate) bounds large grids, so a warp takes two element
// rows (8 element rows serve 7 node rows); grids that do not fill the chip are
// bound by a warp's serial chain and take one row.  us with 9 loads, RE 1 / RE 2:
// elastic step 64^3 1337 / 1172, 32^3 242 / 211, 16^3 45 / 55, 8^3 19 / 31; coupled
// operator 64^3 1833 / 1590, 16^3 62 / 76.
template <typename T>
bool small_grid(const ModalArgs<T>& a) {
  return (i64)a.nx * a.ny * a.nz * a.nrhs <= 65536;
}

template <int KIND, int MODE, int MINB1, int MINB2, typename K>
void go(const ModalArgs<double>& a, const K& k, cudaStream_t s) {
  if (small_grid(a)) modal::launch<KIND, MODE, 1, MINB1, false, double>(a, k, s);
  else modal::launch<KIND, MODE, 2, MINB2, false, double>(a, k, s);
}

}  // namespace

template <>
void modal_full<double>(const ModalArgs<double>& a, const ModalMat<double, 4, 4>& K, cudaStream_t s) {
  go<MK_FULL, MM_APPLY, 3, 2>(a, K, s);
}
void modal_resid(const ModalArgs<double>& a, const ModalMat<double, 4, 4>& K, cudaStream_t s) {
  go<MK_FULL, MM_RESID, 3, 2>(a, K, s);
}

template <>
void modal_pu<double>(const ModalArgs<double>& a, const ModalMat<double, 1, 3>& K, cudaStream_t s) {
  go<MK_PU, MM_ADD, 4, 3>(a, K, s);
}

template <>
void modal_uu<double>(const ModalArgs<double>& a, const ModalMat<double, 3, 3>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: go<MK_UU, MM_APPLY, 3, 2>(a, K, s); break;
    case MM_RESID: go<MK_UU, MM_RESID, 3, 2>(a, K, s); break;
    case MM_STEP: go<MK_UU, MM_STEP, 3, 2>(a, K, s); break;
    case MM_STEP0: go<MK_UU, MM_STEP0, 3, 2>(a, K, s); break;
    case MM_PRE: go<MK_UU, MM_PRE, 3, 2>(a, K, s); break;
    default: go<MK_UU, MM_POST, 3, 2>(a, K, s); break;
  }
}

template <>
void modal_ss<double>(const ModalArgs<double>& a, const ModalSch<double>& K, int mode, cudaStream_t s) {
  switch (mode) {
    case MM_APPLY: go<MK_SS, MM_APPLY, 4, 4>(a, K, s); break;
    case MM_RESID: go<MK_SS, MM_RESID, 4, 4>(a, K, s); break;
    case MM_STEP: go<MK_SS, MM_STEP, 4, 4>(a, K, s); break;
    case MM_STEP0: go<MK_SS, MM_STEP0, 4, 4>(a, K, s); break;
    case MM_PRE: go<MK_SS, MM_PRE, 4, 4>(a, K, s); break;
    default: go<MK_SS, MM_POST, 4, 4>(a, K, s); break;
  }
}

}  // namespace cell
