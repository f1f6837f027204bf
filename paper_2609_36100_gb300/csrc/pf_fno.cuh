// Device helpers shared by the translation units of the surrogate: GELU and
// its derivative, the split BF16 tensor-core product, and the interface of
// the fused kernels of pf_fno_fused.cu.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace pf {

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_g(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// Normal distribution function Phi(z) = (1 + erf(z / sqrt 2)) / 2 of GELU(z) =
// z Phi(z).  The tail Phi(-|z|) is e = exp(-z^2 / 2) times a polynomial in t =
// 1 / (1 + p |z|), the form of Hastings' approximations of the error function,
// here of degree eight with coefficients fitted to 9e-8 relative over |z| <= 14.
// One exponential and one reciprocal serve GELU and its derivative.
struct GaussTail {
    float q, t, e;  // Phi(-|z|) = q t e
};
__device__ __forceinline__ GaussTail gauss_tail(float z) {
    GaussTail g;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(g.t) : "f"(fmaf(fabsf(z), 0.30452660f, 1.0f)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(g.e) : "f"(z * z * -0.72134752f));
    float q = 0.036764109f;
    q = fmaf(q, g.t, -0.15403491f);
    q = fmaf(q, g.t, 0.18868711f);
    q = fmaf(q, g.t, -0.040320144f);
    q = fmaf(q, g.t, 0.12216621f);
    q = fmaf(q, g.t, 0.10296576f);
    q = fmaf(q, g.t, 0.12232373f);
    g.q = fmaf(q, g.t, 0.12144818f);
    return g;
}
// GELU.  Measured error, and that of the formula with the library's erff (where
// 1 + erf cancels for negative z): |z| < 3 evenly 2.1e-7 at most, 4.0e-8 rms
// (2.9e-7, 4.5e-8), normal samples 2.6e-8 rms (2.5e-8, 3.4e-7 and 4.7e-7 at most).
__device__ __forceinline__ float gelu_of(float z, const GaussTail& g) {
    const float tail = g.q * g.t * g.e;
    return z * (z < 0.f ? tail : 1.0f - tail);
}
// GELU'(z) = Phi(z) + z e / sqrt(2 pi).  With both terms of the tail under one
// exponential, e (q t - |z| / sqrt(2 pi)) for negative z and 1 minus that for
// positive; for |z| < 1, where the tail is up to a half and its rounding shows,
// 1/2 and an odd polynomial (fitted to 2e-9).  Measured as above: 1.1e-7 at
// most and 2.5e-8 rms, normal samples 1.2e-7 and 2.3e-8; with the library's erff
// and expf 1.5e-7 and 3.0e-8, 1.6e-7 and 2.8e-8; the tail's form at every z, as
// it was, 2.5e-7 and 3.6e-8, 2.6e-7 and 4.4e-8.
__device__ __forceinline__ float gelu_deriv_of(float z, const GaussTail& g) {
    const float s = fmaf(g.q, g.t, fabsf(z) * -0.39894228f);
    const float far = z < 0.f ? s * g.e : fmaf(-s, g.e, 1.0f);
    const float u = z * z;
    float r = -8.69920405e-05f;
    r = fmaf(r, u, 0.00112302043f);
    r = fmaf(r, u, -0.00948031712f);
    r = fmaf(r, u, 0.0598360933f);
    r = fmaf(r, u, -0.265960872f);
    r = fmaf(r, u, 0.797884524f);
    return u < 1.0f ? fmaf(r, z, 0.5f) : far;
}
__device__ __forceinline__ float gelu_fast(float z) { return gelu_of(z, gauss_tail(z)); }
__device__ __forceinline__ float gelu_fast_g(float z) { return gelu_deriv_of(z, gauss_tail(z)); }

// D += A B on one 16x8x16 BF16 tile, FP32 accumulation
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// two FP32 values -> their BF16 leading parts packed (first value in the low
// half) and the BF16 roundings of their remainders
__device__ __forceinline__ void split2(float x0, float x1, unsigned& hi, unsigned& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __bfloat162float(h.x), x1 - __bfloat162float(h.y));
    hi = *reinterpret_cast<const unsigned*>(&h);
    lo = *reinterpret_cast<const unsigned*>(&l);
}
// (ah + al)(bh + bl) without the al bl term
__device__ __forceinline__ void mma3(float (&d)[4], const unsigned (&ah)[4], const unsigned (&al)[4], unsigned bh0,
                                     unsigned bh1, unsigned bl0, unsigned bl1) {
    mma_bf16_16816(d, ah, bh0, bh1);
    mma_bf16_16816(d, ah, bl0, bl1);
    mma_bf16_16816(d, al, bh0, bh1);
}

// ---------------------------------------------------------------------------
// fused path (pf_fno_fused.cu)
// ---------------------------------------------------------------------------
struct FnoFusedDims {
    int nx, ny, nz, C, m, H, L;
    long long N;
};

// sizes the fused kernels take (BF16 mode only)
bool fno_fused_ok(const FnoFusedDims& d);

// device tables of the fused path: x-axis cosines and sines (plain and scaled
// by w/N) as [4m rounded up to 4][padded nx/2 + 1], y/z ones as [n/2 + 1][m + 1]
struct FnoTables {
    float *xc = nullptr, *xs = nullptr, *xcw = nullptr, *xsw = nullptr;
    float2 *y = nullptr, *z = nullptr;
};
size_t fno_fused_xtab_len(const FnoFusedDims& d);  // floats of each x table
// fills host copies of the tables
void fno_fused_tables(const FnoFusedDims& d, float* xc, float* xs, float* xcw, float* xsw, float2* y, float2* z);
// floats of the per-block partial-sum buffer
size_t fno_fused_part_len(const FnoFusedDims& d);

struct FnoWork {
    float2 *T1, *T2, *Ok, *Gk;  // [nz ny][C m], [nz][2m][C m], [2m][2m][C m] twice
    float* part;
    double* dpart;
};

// spectral part of a layer: T1 (x-transformed rows) -> y, z transforms -> A,
// the mix with the layer's weights, and back to T1
cudaError_t fno_spectral_fwd(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, float2* A,
                             const __nv_bfloat162* w16, cudaStream_t s);
cudaError_t fno_spectral_bwd(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float2* A,
                             const __nv_bfloat162* w16, float2* GW, cudaStream_t s);
// x transform of the lifted input (P x + p) or of a raw [C][N] field (scaled by w/N) into T1
cudaError_t fno_row_lift(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float* x, const float* P,
                         const float* p, cudaStream_t s);
cudaError_t fno_row_raw(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float* g, cudaStream_t s);
// z = V a + v + (inverse x transform of T1); a is GELU(zprev), or P x + p when
// zprev is null; then the x transform of GELU(z) into T1 unless last
cudaError_t fno_row_layer(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float* zprev,
                          const float* x, const float* P, const float* p, const float* V, const float* v, float* z,
                          bool last, cudaStream_t s);
// dz (in place): da = V^T dz + (inverse x transform of T1), then
// da GELU'(zprev) and its x transform (scaled by w/N) into T1; gradients of V
// and v, and of P and p when zprev is null
cudaError_t fno_row_layer_bwd(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, float* dz,
                              const float* zprev, const float* x, const float* P, const float* p, const float* V,
                              float* gV, float* gv, float* gP, float* gp, cudaStream_t s);
// out = Q2 GELU(Q1 a + q1) + q2
cudaError_t fno_project(const FnoFusedDims& d, const float* a, const float* Q1, const float* q1, const float* Q2,
                        const float* q2, float* out, cudaStream_t s);
// the projection's forward, the squared error against tgt (sum over blocks in
// w.dpart, *blocks of them), its gradients and the gradient of a into da
cudaError_t fno_project_bwd(const FnoFusedDims& d, const FnoWork& w, const float* a, const float* tgt,
                            const float* Q1, const float* q1, const float* Q2, const float* q2, float* da, float* gQ1,
                            float* gq1, float* gQ2, float* gq2, int* blocks, cudaStream_t s);

}  // namespace pf
