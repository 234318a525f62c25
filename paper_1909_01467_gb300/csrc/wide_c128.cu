// k_front_wide in complex128, beams and 2D lines.
#include "wide.cuh"

namespace lsw {

template <>
WideKernel wide_kernel<double2, false>(const Wide& wp) {
  return pick_window<double2, false, 0, 3, 4, 5, 6, 7, 8, 9, 10, 11, 13, 15>(wp);
}

}  // namespace lsw
