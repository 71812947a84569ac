// Explicit instantiation of the pipelined world-aligned adjoint kernel for storage
// float, D-solves in float pairs (tapes on chip and in global memory; the units compile in parallel).
#include "kernels.cuh"

namespace abasim {
namespace host {

template <class T, class DT, bool SEG>
BackwardKernel<T> wbackward_pipe_kernel(bool onchip, bool fr) {
  if (fr) return onchip ? k_wbackward_pipe<T, DT, true, true, SEG> : k_wbackward_pipe<T, DT, false, true, SEG>;
  return onchip ? k_wbackward_pipe<T, DT, true, false, SEG> : k_wbackward_pipe<T, DT, false, false, SEG>;
}
template BackwardKernel<float> wbackward_pipe_kernel<float, FF, false>(bool, bool);

}  // namespace host
}  // namespace abasim
