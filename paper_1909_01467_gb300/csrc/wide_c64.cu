// k_front_wide in complex64.
#include "wide.cuh"

namespace lsw {

template <>
WideKernel wide_kernel<float2, false>(const Wide& wp) {
  return pick_window<float2, false, 3, 5, 9, 14>(wp);
}
template <>
WideKernel wide_kernel<float2, true>(const Wide& wp) {
  return pick_window<float2, true, 5, 9, 14>(wp);
}

}  // namespace lsw
