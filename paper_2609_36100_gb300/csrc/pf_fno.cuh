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
// z Phi(z), with e = exp(-z^2 / 2) for the derivative Phi(z) + z e / sqrt(2 pi).
// The tail Phi(-|z|) is e times a polynomial in t = 1 / (1 + p |z|), the form of
// Hastings' approximations of the error function, here of degree eight with
// coefficients fitted to 9e-8 relative over |z| <= 14.  In FP32 the error of
// GELU (2.1e-7 at most, 4.0e-8 rms for |z| < 3) is that of the formula with
// the library's erff (2.5e-7, 4.4e-8): there 1 + erf cancels for negative z.
// One exponential serves both values: 16 instructions for GELU and 19 with its
// derivative, against about 31 and 60 with erff and expf.
__device__ __forceinline__ float gauss_cdf(float z, float& e) {
    float t;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(fmaf(fabsf(z), 0.30452660f, 1.0f)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(z * z * -0.72134752f));
    float q = 0.036764109f;
    q = fmaf(q, t, -0.15403491f);
    q = fmaf(q, t, 0.18868711f);
    q = fmaf(q, t, -0.040320144f);
    q = fmaf(q, t, 0.12216621f);
    q = fmaf(q, t, 0.10296576f);
    q = fmaf(q, t, 0.12232373f);
    q = fmaf(q, t, 0.12144818f);
    const float tail = q * t * e;
    return z < 0.f ? tail : 1.0f - tail;
}
__device__ __forceinline__ float gelu_fast(float z) {
    float e;
    return z * gauss_cdf(z, e);
}
__device__ __forceinline__ float gelu_fast_g(float z) {
    float e;
    const float c = gauss_cdf(z, e);
    return fmaf(z * 0.39894228f, e, c);
}

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
