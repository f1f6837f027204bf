// Fused x passes of part of the line lengths (templates in pf_xfused.cuh; the
// lengths are spread over four translation units that compile in parallel).
#include "pf_xfused.cuh"

namespace pf {
#define PF_XF_INST(N_)                                                                                       \
    template int launch_x_fused_n<N_>(const Geo&, const Phys&, int, const void*, void*, void*, const void*, \
                                      double*, double, double, cudaStream_t);
PF_XF_INST(48)
PF_XF_INST(80)
PF_XF_INST(120)
PF_XF_INST(180)
PF_XF_INST(240)
PF_XF_INST(320)
PF_XF_INST(432)
#undef PF_XF_INST
}  // namespace pf
