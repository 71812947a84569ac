// Explicit instantiation of the pipelined world-aligned adjoint kernel for storage
// float, D-solves in float pairs (tapes on chip and in global memory; the units compile in parallel).
#include "kernels.cuh"

namespace abasim {
namespace host {

template <class T, class DT>
BackwardKernel<T> wbackward_pipe_kernel(bool onchip, bool fr) {
  if (fr) return onchip ? k_wbackward_pipe<T, DT, true, true> : k_wbackward_pipe<T, DT, false, true>;
  return onchip ? k_wbackward_pipe<T, DT, true, false> : k_wbackward_pipe<T, DT, false, false>;
}
template BackwardKernel<float> wbackward_pipe_kernel<float, FF>(bool, bool);

}  // namespace host
}  // namespace abasim
