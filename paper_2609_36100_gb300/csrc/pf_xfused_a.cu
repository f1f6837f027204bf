// Fused x passes of part of the line lengths (templates in pf_xfused.cuh; the
// lengths are spread over four translation units that compile in parallel).
#include "pf_xfused.cuh"

namespace pf {
#define PF_XF_INST(N_)                                                                                       \
    template int launch_x_fused_n<N_>(const Geo&, const Phys&, int, const void*, void*, void*, const void*, \
                                      double*, double, double, cudaStream_t);
PF_XF_INST(32)
PF_XF_INST(60)
PF_XF_INST(96)
PF_XF_INST(128)
PF_XF_INST(192)
PF_XF_INST(256)
PF_XF_INST(360)
PF_XF_INST(480)
#undef PF_XF_INST
}  // namespace pf
