// Instantiation of the FP64 y-axis column transforms (templates in pf_yz.cuh;
// one translation unit each so that they compile in parallel).
#include "pf_yz.cuh"

namespace pf {
template void launch_y_pass_sign<double, 1>(const Geo&, void*, int, cudaStream_t);
template void launch_y_pass_sign<double, -1>(const Geo&, void*, int, cudaStream_t);
}  // namespace pf
