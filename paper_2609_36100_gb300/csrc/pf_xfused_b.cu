// Fused x passes of part of the line lengths (templates in pf_xfused.cuh; the
// lengths are spread over four translation units that compile in parallel).
#include "pf_xfused.cuh"

namespace pf {
#define PF_XF_INST(N_)                                                                                       \
    template int launch_x_fused_n<N_>(const Geo&, const Phys&, int, const void*, void*, void*, const void*, \
                                      double*, double, double, cudaStream_t);
PF_XF_INST(36)
PF_XF_INST(64)
PF_XF_INST(100)
PF_XF_INST(144)
PF_XF_INST(200)
PF_XF_INST(288)
PF_XF_INST(384)
PF_XF_INST(512)
#undef PF_XF_INST
}  // namespace pf
