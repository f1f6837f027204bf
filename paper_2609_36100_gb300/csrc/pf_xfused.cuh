// Fused x passes (FP32 compute type): packed real transforms along x with the
// real-space physics between them, organised so that the physics runs in the
// registers of the threads that finish the inverse transform and start the
// forward one.
//
// The forward transform of a line uses the radix order Fwd = (RM, ...); the
// inverse runs it reversed, so its last stage (radix RM, sub-transform size
// M = N/RM) leaves butterfly j holding the elements x = j + M t (t < RM) --
// exactly the inputs of butterfly j of the forward first stage.  One thread
// per (row pair, j) therefore takes the last inverse stage of every input
// field, evaluates the physics at its RM positions of both rows, and applies
// the first forward stage to every output field without a shared-memory
// round trip.  The C2R packing of two real rows into one complex line is
// folded into the first inverse stage (read straight from the staged
// half-spectrum rows), the R2C unpacking into the store.  Every stage runs in
// place in one shared-memory tile of skewed lines: two tiles, with a barrier
// less a stage, hold half the CTAs on an SM and were as fast at 64 points and
// slower from 96 on (right-hand-side pass at 256^3: 256 us against 200, h pass 182
// against 154 then, 201 and 161 with the stages as they are now); so was copying
// the real fields into shared memory ahead of the physics (213 against 200 us).
#pragma once
#include "pf_xpass.cuh"

namespace pf {

enum XFMode { XF_PHYS1_H = 0, XF_PHYS1_RHS = 1, XF_PHYS2 = 2, XF_WRMS = 3 };
template <int MODE>
struct XFIO {
    static constexpr int FIN = MODE == XF_PHYS2 ? 3 : 4;  // input lines per row pair
    static constexpr int FOUT = MODE == XF_WRMS ? 0 : (MODE == XF_PHYS1_H ? 3 : 4);
};

// Lines are skewed (one empty slot after every 16 elements) or not, as their
// plan says.  Power-of-two lengths are: their stages read and write with
// power-of-two strides.  Most others are not: an odd first radix is free of
// most conflicts as it stands, and with N / R no multiple of 16 the skew costs
// two integer instructions an element (right-hand-side pass at 480 points 1714
// us skewed, 1596 not; h pass 1516 and 1309).
template <int N, bool SKEW>
struct XFLine {
    static constexpr int LS = SKEW ? N + N / 16 : N + 2;  // stride: at least the two raw rows of a line
};

// In-place stage of NL lines (one shared buffer): every job's R inputs are
// loaded into registers, the CTA synchronises, then the butterflies are formed
// and stored, and the CTA synchronises again.
template <int R, int SIGN, int N, int NS, int NL, int NT, bool SK, typename T2>
__device__ __forceinline__ void xf_stage_inplace(T2* S, const T2* __restrict__ tw) {
    constexpr int M = N / R, TWS = N / (NS * R), JOBS = NL * M, JPT = (JOBS + NT - 1) / NT, LS = XFLine<N, SK>::LS;
    T2 v[JPT][R];
#pragma unroll
    for (int u = 0; u < JPT; ++u) {
        const int idx = threadIdx.x + u * NT;
        if (JOBS % NT == 0 || idx < JOBS) {
            const int line = idx / M, j = idx - line * M;
            const T2* s = S + line * LS;
            if constexpr (!SK) {
#pragma unroll
                for (int t = 0; t < R; ++t) v[u][t] = s[j + t * M];
            } else if constexpr (M % 16 == 0) {
                // skew(j + t M) = skew(j) + t (M + M/16)
                const T2* sj = s + skew<true>(j);
#pragma unroll
                for (int t = 0; t < R; ++t) v[u][t] = sj[t * (M + M / 16)];
            } else {
#pragma unroll
                for (int t = 0; t < R; ++t) v[u][t] = s[skew<true>(j + t * M)];
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < JPT; ++u) {
        const int idx = threadIdx.x + u * NT;
        if (JOBS % NT == 0 || idx < JOBS) {
            const int line = idx / M, j = idx - line * M;
            const int jq = j / NS, k = j - jq * NS;
            if constexpr (NS > 1)
                tw_bfly<R, SIGN>(v[u], tw, k * TWS, N);
            else
                Bfly<R, SIGN, T2>::run(v[u]);
            T2* d = S + line * LS;
            const int a = jq * NS * R;  // outputs at a + k + t NS
            if constexpr (!SK) {
                T2* dk = d + a + k;
#pragma unroll
                for (int t = 0; t < R; ++t) dk[t * NS] = v[u][t];
            } else if constexpr ((NS * R) % 16 == 0 && NS % 16 == 0) {
                T2* dk = d + skew<true>(a) + skew<true>(k);
#pragma unroll
                for (int t = 0; t < R; ++t) dk[t * (NS + NS / 16)] = v[u][t];
            } else if constexpr ((NS * R) % 16 == 0 && 16 % NS == 0) {
                // k + t NS crosses a 16-block boundary only at multiples of 16
                T2* dk = d + skew<true>(a) + k;
#pragma unroll
                for (int t = 0; t < R; ++t) dk[t * NS + ((t * NS) >> 4)] = v[u][t];
            } else if constexpr (NS == 1 && 16 % R == 0) {
                // a = j R and a + t stay inside one 16-block
                T2* dk = d + skew<true>(a);
#pragma unroll
                for (int t = 0; t < R; ++t) dk[t] = v[u][t];
            } else {
#pragma unroll
                for (int t = 0; t < R; ++t) d[skew<true>(a + k + t * NS)] = v[u][t];
            }
        }
    }
    __syncthreads();
}
template <int SIGN, int N, int NS, int NL, int NT, bool SK, typename T2>
__device__ __forceinline__ void xf_run_inplace(T2*, const T2*, Radices<>) {}
template <int SIGN, int N, int NS, int NL, int NT, bool SK, typename T2, int R, int... Rest>
__device__ __forceinline__ void xf_run_inplace(T2* S, const T2* tw, Radices<R, Rest...>) {
    xf_stage_inplace<R, SIGN, N, NS, NL, NT, SK>(S, tw);
    xf_run_inplace<SIGN, N, NS * R, NL, NT, SK>(S, tw, Radices<Rest...>{});
}

template <class Fwd, int P, bool SK>
struct XFShape {
    static constexpr int N = RadProd<Fwd>::value;
    static constexpr int RM = RadInfo<Fwd>::first;  // radix of the fused stages
    static constexpr int M = N / RM;                 // butterflies per line in the fused stages
    static constexpr int NT = P * M;                 // one thread per (row pair, butterfly)
    static_assert(NT % 32 == 0 && NT <= 1024, "whole warps, at most 1024 threads");
    static constexpr int LS = XFLine<N, SK>::LS;     // line stride
};

// registers bounded to 64 a thread, so that they do not cap the CTAs per SM
// before the shared memory does
template <class Fwd, int P, bool SK, int MODE>
__global__ void __launch_bounds__(XFShape<Fwd, P, SK>::NT, 65536 / (XFShape<Fwd, P, SK>::NT * 64) > 0
                                                               ? 65536 / (XFShape<Fwd, P, SK>::NT * 64)
                                                               : 1)
    k_x_fused(Geo g, Phys ph, const float2* __restrict__ in,
                                                                  float2* __restrict__ out, float* __restrict__ R,
                                                                  const float* __restrict__ Rin,
                                                                  double* __restrict__ partials, float rt, float at) {
    PF_SKIP_INACTIVE(g);
    using T2 = float2;
    using Sh = XFShape<Fwd, P, SK>;
    constexpr int N = Sh::N, RM = Sh::RM, M = Sh::M, NT = Sh::NT, LS = Sh::LS, NXH = N / 2 + 1;
    constexpr int FIN = XFIO<MODE>::FIN, FOUT = XFIO<MODE>::FOUT;
    using Inv = Reversed<Fwd>;
    constexpr int R1 = RadInfo<Inv>::first;  // first inverse stage
    extern __shared__ __align__(16) unsigned char smraw[];
    T2* A = reinterpret_cast<T2*>(smraw);
    T2* B = A;  // the raw rows, where the first stage's results go
    const int npairs = g.nz * g.ny / 2;
    const int rp0 = blockIdx.x * P;
    const long long NK = g.NK, N3 = g.N;
    const T2* tw = g.px.tw32;
    __shared__ double red[NT / 32 + 1];

    // 1. the raw half-spectrum rows of the input fields -> B (cp.async).  Raw
    //    row r = (rp FIN + f) 2 + (0: row y, 1: row y+1) goes to B + r NXH.
    //    NXH is odd and NK even, so row r starts 16-byte aligned in global and
    //    shared memory alike when r is even and one element later when r is
    //    odd: each row is NXH/2 16-byte copies from its first aligned element
    //    and one 8-byte copy of the element left over (the last or the first)
    {
        static_assert(NXH % 2 == 1, "odd half-spectrum rows");
        constexpr int NC = NXH / 2 + 1;  // copies per row: NXH/2 pairs and one single
        for (int e = threadIdx.x; e < P * FIN * 2 * NC; e += NT) {
            const int r = e / NC, c = e - r * NC;
            const int pf = r >> 1, rp = pf / FIN, f = pf - rp * FIN;
            const int head = r & 1;  // first element of the aligned pairs
            const int k = c < NXH / 2 ? head + 2 * c : (head ? 0 : NXH - 1);
            T2* dst = B + r * NXH + k;
            if (rp0 + rp < npairs) {
                const T2* src = in + (long long)f * NK + (2LL * (rp0 + rp) + head) * NXH + k;
                if (c < NXH / 2)
                    cp_async<16>(dst, src);
                else
                    cp_async<8>(dst, src);
            } else {
                dst[0] = T2{0.f, 0.f};
                if (c < NXH / 2) dst[1] = T2{0.f, 0.f};
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();
    // 2. first inverse stage (radix R1, no twiddles), packing Z = a + i b of
    //    the two rows' half spectra (Hermitian extension, imaginary parts of
    //    DC and Nyquist dropped), in place: all loads, a barrier, the stores
    {
        constexpr int M1 = N / R1, JOBS = P * FIN * M1, JPT = (JOBS + NT - 1) / NT;
        auto load = [&](int idx, T2* v) {
            const int line = idx / M1, j = idx - line * M1;
            const T2* ra = B + line * 2 * NXH;
            const T2* rb = ra + NXH;
#pragma unroll
            for (int t = 0; t < R1; ++t) {
                const int x = j + t * M1;
                const bool lo = x <= N / 2;
                const int k = lo ? x : N - x;
                T2 a = ra[k], b = rb[k];
                if (k == 0 || k == N / 2) {
                    a.y = 0.f;
                    b.y = 0.f;
                }
                v[t] = lo ? T2{a.x - b.y, a.y + b.x} : T2{a.x + b.y, b.x - a.y};
            }
        };
        auto store = [&](int idx, T2* v) {
            const int line = idx / M1, j = idx - line * M1;
            Bfly<R1, +1, T2>::run(v);
            T2* d = A + line * LS;
#pragma unroll
            for (int t = 0; t < R1; ++t) d[skew<SK>(j * R1 + t)] = v[t];
        };
        T2 v[JPT][R1];
#pragma unroll
        for (int u = 0; u < JPT; ++u)
            if (JOBS % NT == 0 || threadIdx.x + u * NT < JOBS) load(threadIdx.x + u * NT, v[u]);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < JPT; ++u)
            if (JOBS % NT == 0 || threadIdx.x + u * NT < JOBS) store(threadIdx.x + u * NT, v[u]);
    }
    __syncthreads();
    // 3. inverse stages between the first and the last
    xf_run_inplace<+1, N, R1, P * FIN, NT, SK>(A, tw, typename PlanInner<Inv>::type{});
    // 4. fused: last inverse stage, physics, first forward stage
    const int rp = threadIdx.x / M, j = threadIdx.x - (threadIdx.x / M) * M;
    const bool valid = rp0 + rp < npairs;
    const long long row = 2LL * (rp0 + rp);
    T2 vin[FIN][RM];
#pragma unroll
    for (int f = 0; f < FIN; ++f) {
        const T2* src = A + (rp * FIN + f) * LS;
#pragma unroll
        for (int t = 0; t < RM; ++t) vin[f][t] = src[skew<SK>(j + t * M)];
        tw_bfly<RM, +1>(vin[f], tw, j, N);  // NS = M: twiddle exponent j t
    }
    if constexpr (MODE == XF_WRMS) {
        // sum of squares of the weighted error w_i LTE_i (weights from the
        // stored real-space y_{n-1}); compensated FP32 sum per thread, FP64
        // across threads and CTAs
        float sh = 0.f, sl = 0.f;
        if (g.tol) {
            rt = step_tol<float>(*g.tol, 0);
            at = step_tol<float>(*g.tol, 1);
        }
        if (valid) {
#pragma unroll
            for (int t = 0; t < RM; ++t) {
                const int x = j + t * M;
#pragma unroll
                for (int f = 0; f < FIN; ++f) {
                    const float* yr = Rin + f * N3 + row * N + x;
                    const float a = __fdividef(vin[f][t].x, __fmaf_rn(rt, fabsf(yr[0]), at));
                    const float b = __fdividef(vin[f][t].y, __fmaf_rn(rt, fabsf(yr[N]), at));
                    const DF s1 = df_two_sum(sh, __fmul_rn(a, a));
                    const DF s2 = df_two_sum(s1.h, __fmul_rn(b, b));
                    sh = s2.h;
                    sl = __fadd_rn(sl, __fadd_rn(s1.l, s2.l));
                }
            }
        }
        double acc = f2d_bits(sh) + f2d_bits(sl);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int i = 0; i < (NT + 31) / 32; ++i) s += red[i];
            partials[blockIdx.x] = s;
        }
        return;
    } else {
        const PhysT<float>& pt = ph.t32;
        T2 vout[FOUT][RM];
#pragma unroll
        for (int t = 0; t < RM; ++t) {
            const int x = j + t * M;
            float Xr[2], pr[2][3], er[2][3];
            if constexpr (MODE == XF_PHYS2) {
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    const float* b = Rin + f * N3 + row * N + x;
                    const float u0 = valid ? b[0] : 0.f, u1 = valid ? b[N] : 0.f;
                    if (f == 0) {
                        Xr[0] = u0;
                        Xr[1] = u1;
                    } else {
                        pr[0][f - 1] = u0;
                        pr[1][f - 1] = u1;
                    }
                }
#pragma unroll
                for (int v = 0; v < 3; ++v) {
                    er[0][v] = vin[v][t].x;
                    er[1][v] = vin[v][t].y;
                }
            } else {
                Xr[0] = vin[0][t].x;
                Xr[1] = vin[0][t].y;
#pragma unroll
                for (int v = 0; v < 3; ++v) {
                    pr[0][v] = vin[1 + v][t].x;
                    pr[1][v] = vin[1 + v][t].y;
                    er[0][v] = 0.f;
                    er[1][v] = 0.f;
                }
                if (R && valid) {
#pragma unroll
                    for (int f = 0; f < 4; ++f) {
                        float* b = R + f * N3 + row * N + x;
                        b[0] = vin[f][t].x;
                        b[N] = vin[f][t].y;
                    }
                }
            }
            if constexpr (MODE == XF_PHYS1_H) {
#pragma unroll
                for (int v = 0; v < 3; ++v) vout[v][t] = T2{hfun(pr[0][v]), hfun(pr[1][v])};
            } else {
                float q[2], gv[2][3];
#pragma unroll
                for (int r = 0; r < 2; ++r) Pt::rhs<float, false>(pt, Xr[r], pr[r], er[r], q[r], gv[r]);
                vout[0][t] = T2{q[0], q[1]};
#pragma unroll
                for (int v = 0; v < 3; ++v) vout[1 + v][t] = T2{gv[0][v], gv[1][v]};
            }
        }
        __syncthreads();  // every input of the fused stage read before the stores
#pragma unroll
        for (int f = 0; f < FOUT; ++f) {
            Bfly<RM, -1, T2>::run(vout[f]);  // first forward stage: NS = 1, no twiddles
            T2* d = A + (rp * FOUT + f) * LS;
#pragma unroll
            for (int t = 0; t < RM; ++t) d[skew<SK>(j * RM + t)] = vout[f][t];
        }
        __syncthreads();
        // 5. the remaining forward stages
        xf_run_inplace<-1, N, RM, P * FOUT, NT, SK>(A, tw, typename DropFirst<Fwd>::type{});
        // 6. R2C unpacking of the two rows of each line and the store
        for (int e = threadIdx.x; e < P * FOUT * NXH; e += NT) {
            const int line = e / NXH, k = e - line * NXH, lrp = line / FOUT, f = line - lrp * FOUT;
            if (rp0 + lrp >= npairs) continue;
            const T2 Zk = A[line * LS + skew<SK>(k)];
            const T2 Zm = A[line * LS + skew<SK>(k == 0 ? 0 : N - k)];
            const T2 a = T2{(Zk.x + Zm.x) * 0.5f, (Zk.y - Zm.y) * 0.5f};
            const T2 b = T2{(Zk.y + Zm.y) * 0.5f, (Zm.x - Zk.x) * 0.5f};
            T2* base = out + (long long)f * NK + (2LL * (rp0 + lrp)) * NXH + k;
            base[0] = a;
            base[NXH] = b;
        }
    }
}

// Fused plans by line length (FP32): row pairs per CTA, whether the lines are
// skewed, and the radices.  The first forward radix is small, so that the fused
// stage holds few values per field; the row pairs give 100 to 400 threads (whole
// warps) and, below 128 points, at least about 150 CTAs for a cube of that side
// (at 32 points 16 CTAs of 32 pairs took 4 us more a pass).  Of the orders tried
// the fastest: an odd first radix and the power of two next (480 = 5 8 12: 1177
// and 1455 us for the h and the right-hand-side pass, 5 12 8: 1309 and 1596, 3 16
// 10: 1385 and 1633).
template <int N>
struct XFPlan {
    static constexpr bool ok = false;
};
#define PF_XF_PLAN(N_, P_, SK_, ...)         \
    template <>                              \
    struct XFPlan<N_> {                      \
        static constexpr bool ok = true;     \
        static constexpr int P = P_;         \
        static constexpr bool SK = SK_;      \
        using Fwd = Radices<__VA_ARGS__>;    \
    };
PF_XF_PLAN(32, 4, true, 2, 4, 4)
PF_XF_PLAN(36, 8, false, 3, 12)
PF_XF_PLAN(40, 4, false, 5, 8)
PF_XF_PLAN(48, 8, false, 3, 16)
PF_XF_PLAN(60, 8, false, 3, 4, 5)
PF_XF_PLAN(64, 8, true, 4, 16)
PF_XF_PLAN(72, 8, false, 3, 8, 3)
PF_XF_PLAN(80, 8, true, 5, 16)
PF_XF_PLAN(96, 8, true, 4, 8, 3)
PF_XF_PLAN(100, 8, false, 5, 4, 5)
PF_XF_PLAN(108, 8, false, 3, 12, 3)
PF_XF_PLAN(120, 4, false, 3, 8, 5)
PF_XF_PLAN(128, 8, true, 4, 8, 4)
PF_XF_PLAN(144, 4, false, 3, 8, 6)
PF_XF_PLAN(160, 4, false, 4, 8, 5)
PF_XF_PLAN(180, 8, false, 5, 12, 3)
PF_XF_PLAN(192, 4, true, 4, 16, 3)
PF_XF_PLAN(200, 4, false, 5, 8, 5)
PF_XF_PLAN(216, 4, false, 3, 12, 6)
PF_XF_PLAN(240, 4, false, 5, 8, 6)
PF_XF_PLAN(256, 4, true, 4, 16, 4)
PF_XF_PLAN(288, 2, false, 3, 8, 12)
PF_XF_PLAN(300, 8, false, 5, 6, 10)
PF_XF_PLAN(320, 2, false, 5, 8, 8)
PF_XF_PLAN(360, 4, false, 5, 8, 9)
PF_XF_PLAN(384, 2, true, 4, 12, 8)
PF_XF_PLAN(400, 4, false, 5, 8, 10)
PF_XF_PLAN(432, 2, false, 3, 12, 12)
PF_XF_PLAN(480, 2, false, 5, 8, 12)
PF_XF_PLAN(512, 2, true, 4, 16, 8)
PF_XF_PLAN(640, 2, true, 5, 16, 8)
#undef PF_XF_PLAN

template <int N, int MODE>
static int launch_x_fused_k(const Geo& g, const Phys& ph, const void* in, void* out, void* R, const void* Rin,
                            double* partials, double rtol, double atol, cudaStream_t s) {
    using Pl = XFPlan<N>;
    using Sh = XFShape<typename Pl::Fwd, Pl::P, Pl::SK>;
    const size_t sm = (size_t)Pl::P * 4 * Sh::LS * sizeof(float2);
    const int npairs = g.nz * g.ny / 2;
    const int nb = (npairs + Pl::P - 1) / Pl::P;
    auto k = k_x_fused<typename Pl::Fwd, Pl::P, Pl::SK, MODE>;
    set_smem(k, sm);
    k<<<nb, Sh::NT, sm, s>>>(g, ph, reinterpret_cast<const float2*>(in), reinterpret_cast<float2*>(out),
                             reinterpret_cast<float*>(R), reinterpret_cast<const float*>(Rin), partials, (float)rtol,
                             (float)atol);
    return nb;
}

// the fused x pass of line length N; returns the number of CTAs launched, 0
// for a mode it does not have
template <int N>
int launch_x_fused_n(const Geo& g, const Phys& ph, int mode, const void* in, void* out, void* R, const void* Rin,
                     double* partials, double rtol, double atol, cudaStream_t s) {
    static_assert(XFPlan<N>::ok, "no fused plan of this length");
    switch (mode) {
        case XM_PHYS1:
            return ph.elastic ? launch_x_fused_k<N, XF_PHYS1_H>(g, ph, in, out, R, Rin, partials, rtol, atol, s)
                              : launch_x_fused_k<N, XF_PHYS1_RHS>(g, ph, in, out, R, Rin, partials, rtol, atol, s);
        case XM_PHYS2:
            if (!ph.elastic) return 0;
            return launch_x_fused_k<N, XF_PHYS2>(g, ph, in, out, R, Rin, partials, rtol, atol, s);
        case XM_WRMS: return launch_x_fused_k<N, XF_WRMS>(g, ph, in, out, R, Rin, partials, rtol, atol, s);
        default: return 0;
    }
}

}  // namespace pf
