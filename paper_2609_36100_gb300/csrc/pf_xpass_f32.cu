// Instantiation of the FP32 x passes (templates in pf_xpass.cuh) and the
// choice of the fused ones, which are instantiated in pf_xfused_a.cu to _d.cu.
#include "pf_xpass.cuh"

namespace pf {
template <int N>
int launch_x_fused_n(const Geo& g, const Phys& ph, int mode, const void* in, void* out, void* R, const void* Rin,
                     double* partials, double rtol, double atol, cudaStream_t s);

// the fused x pass for FP32 contexts where the line length has a fused plan;
// returns the number of CTAs launched, 0 if it does not apply
int launch_x_fused(const Geo& g, const Phys& ph, int mode, const void* in, void* out, void* R, const void* Rin,
                   double* partials, double rtol, double atol, cudaStream_t s) {
    // the obstacle barrier runs the staged passes (the fused ones carry only the double well)
    if (g.xf_off || ph.obst) return 0;
    switch (g.nx) {
#define PF_XF(N_) \
    case N_: return launch_x_fused_n<N_>(g, ph, mode, in, out, R, Rin, partials, rtol, atol, s);
        PF_XF(32) PF_XF(36) PF_XF(40) PF_XF(48) PF_XF(60) PF_XF(64)
        PF_XF(72) PF_XF(80) PF_XF(96) PF_XF(100) PF_XF(108) PF_XF(120)
        PF_XF(128) PF_XF(144) PF_XF(160) PF_XF(180) PF_XF(192) PF_XF(200)
        PF_XF(216) PF_XF(240) PF_XF(256) PF_XF(288) PF_XF(300) PF_XF(320)
        PF_XF(360) PF_XF(384) PF_XF(400) PF_XF(432) PF_XF(480) PF_XF(512)
        PF_XF(640)
#undef PF_XF
        default: return 0;
    }
}

template int launch_x_pass<float>(const Geo&, const Phys&, int, const void*, void*, void*, const void*, double*,
                                 double, double, const double*, double*, cudaStream_t);
}  // namespace pf
