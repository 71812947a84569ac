// Explicit instantiation of the world-aligned rollout kernels for storage float, D-solves
// in float pairs (tape on chip and in global memory; the units compile in parallel).
#include "kernels.cuh"

namespace abasim {
namespace host {

template <class T, class DT>
RolloutKernel<T> wrollout_kernel(bool onchip, bool fr) {
  if (fr) return onchip ? k_wrollout<T, DT, true, true> : k_wrollout<T, DT, false, true>;
  return onchip ? k_wrollout<T, DT, true, false> : k_wrollout<T, DT, false, false>;
}
template RolloutKernel<float> wrollout_kernel<float, FF>(bool, bool);

}  // namespace host
}  // namespace abasim
