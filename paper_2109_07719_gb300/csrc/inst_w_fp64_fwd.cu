// Explicit instantiation of the world-aligned rollout kernels for storage double, D-solves
// double (tape on chip and in global memory; the units compile in parallel).
#include "kernels.cuh"

namespace abasim {
namespace host {

template <class T, class DT>
RolloutKernel<T> wrollout_kernel(bool onchip, bool fr) {
  if (fr) return onchip ? k_wrollout<T, DT, true, true> : k_wrollout<T, DT, false, true>;
  return onchip ? k_wrollout<T, DT, true, false> : k_wrollout<T, DT, false, false>;
}
template RolloutKernel<double> wrollout_kernel<double, double>(bool, bool);

template <class T> RolloutKernel<T> wrollout_team_kernel() { return k_wrollout_team<T>; }
template RolloutKernel<double> wrollout_team_kernel<double>();

}  // namespace host
}  // namespace abasim
