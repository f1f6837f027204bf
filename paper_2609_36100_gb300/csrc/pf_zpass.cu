// Instantiation of the inverse and the FP64 forward z transforms (templates in pf_yz.cuh;
// one translation unit each so that they compile in parallel).
#include "pf_yz.cuh"

namespace pf {
template void launch_z_pass<float>(const Geo&, void*, int, cudaStream_t);
template void launch_z_pass<double>(const Geo&, void*, int, cudaStream_t);
template void launch_z_fwd<double>(const Geo&, const Phys&, const void*, void*, int, cudaStream_t, int);
}  // namespace pf
