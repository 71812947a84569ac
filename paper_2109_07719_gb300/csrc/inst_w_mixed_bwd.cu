// Explicit instantiation of the world-aligned adjoint kernels for storage float, D-solves
// in float pairs (tape on chip and in global memory; the units compile in parallel).
#include "kernels.cuh"

namespace abasim {
namespace host {

template <class T, class DT>
BackwardKernel<T> wbackward_kernel(bool onchip, bool fr) {
  if (fr) return onchip ? k_wbackward<T, DT, true, true> : k_wbackward<T, DT, false, true>;
  return onchip ? k_wbackward<T, DT, true, false> : k_wbackward<T, DT, false, false>;
}
template BackwardKernel<float> wbackward_kernel<float, FF>(bool, bool);

}  // namespace host
}  // namespace abasim
