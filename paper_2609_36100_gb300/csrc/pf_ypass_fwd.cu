// Instantiation of the FP32 forward y-axis column transform (templates in pf_yz.cuh;
// one translation unit each so that they compile in parallel).
#include "pf_yz.cuh"

namespace pf {
template void launch_y_pass_sign<float, -1>(const Geo&, void*, int, cudaStream_t);
}  // namespace pf
