// k_front_wide in complex128, cube-CDD boxes.
#include "wide.cuh"

namespace lsw {

template <>
WideKernel wide_kernel<double2, true>(const Wide& wp) {
  return pick_window<double2, true, 5, 6, 7, 8, 9, 10, 11, 13, 15>(wp);
}

}  // namespace lsw
