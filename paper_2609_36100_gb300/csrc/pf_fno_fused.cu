// Fused kernels of the Fourier neural operator surrogate (BF16 mode).
//
// One layer is two kinds of work: pointwise channel products and truncated
// transforms along the rows of the grid, both of which need all channels of a
// row, and transforms along y and z of the few retained x modes.  The row
// kernels do everything of the first kind in one pass over the activations:
// two warps hold one row of all channels in shared memory, apply GELU to the
// previous pre-activation, the channel product on the tensor cores, add the
// inverse x transform of the layer's spectral part, store the
// pre-activation, and leave the x transform of its GELU for the next layer.
// So a layer reads one [C][N] array and writes one; activations are
// recomputed from pre-activations instead of stored.  The transforms use the
// symmetry of cosines and sines under x -> n - x, which halves their products.
//
// Layout of the partial transforms: channels and x modes innermost,
// T1 [z][y][c][kx], T2 [z][jy][c][kx], A [jz][jy][c][kx] (jy, jz: 0..m-1, then
// -m..-1), so that every transform along y and z is a contraction over the
// middle index with a contiguous inner one.
#include <cmath>
#include <type_traits>

#include "pf_fno.cuh"

namespace pf {

namespace {

constexpr int kSMs = 152;
constexpr int kSmemMax = 227 * 1024;
constexpr int kMaxModes = 16;  // x modes a lane group of the row kernels covers
constexpr int kMaxRow = 256;   // points of a row
constexpr int kFoldIter = (kMaxRow / 2 + 31) / 32;  // pairs of positions a lane folds: 4, or 2 (rows of up to 128)

__host__ __device__ inline int up(int a, int b) { return (a + b - 1) / b * b; }
// padded half row, row pitch (16-byte units odd: rows 0..7 fall on different
// banks, also as the k rows 2t of a B fragment), padded inverse positions
__host__ __device__ inline int half_pad(int nx) { return up(nx / 2 + 1, 4); }
__host__ __device__ inline int row_pitch(int nx) {
    int r = 2 * half_pad(nx);
    if (r < up(nx, 8)) r = up(nx, 8);
    while (r % 8 != 4) r += 4;
    return r;
}
__host__ __device__ inline int inv_pad(int nx) { return up((nx + 1) / 2, 16); }
inline int chan_pad(int C) { return C <= 16 ? 16 : 32; }
inline int modes_pad(int m) { return up(m, 4); }

struct RowArgs {
    const float* zprev;  // previous pre-activation (GELU applied), raw field, or null (lift of x)
    const float* x;      // network input [4][N]
    const float *P, *pb; // lift
    const float *V, *vb;
    float2* T1;
    float* z;            // forward: pre-activation out; backward: dz in and out
    const float *fc, *fs, *ic, *is;  // forward and inverse x tables
    float* part;
    int nx, C, m;
    int dense;  // forward: the layer (else only the x transform)
    int raw;    // zprev is taken as it is
    int last;   // forward: no x transform afterwards
    int vec;    // rows of the [C][N] arrays start on 16-byte boundaries
    long long N, rows;
};

// shared memory of the row kernels, in floats
struct RowSmem {
    int tf, ti, sp, frag, bias, lift, warp, perwarp;
};
__host__ __device__ inline RowSmem row_smem(int nx, int CP, int MP) {
    RowSmem o;
    const int HP = half_pad(nx), XQ = inv_pad(nx), T = CP / 16;
    o.tf = 0;
    o.ti = o.tf + 2 * MP * HP;
    o.sp = o.ti + 2 * MP * XQ;
    o.frag = o.sp + MP;
    o.bias = o.frag + T * T * 256;
    o.lift = o.bias + CP;
    o.warp = o.lift + 5 * CP;
    o.perwarp = CP * row_pitch(nx) + 2 * MP * (CP + 4);
    return o;
}

// The warps of a row: `part` 0..W-1 of W, synchronised by a named barrier
// (W = 2) or within the warp.  Shared memory holds about ten rows an SM; with
// one warp a row that left two warps a scheduler.
template <int W>
struct Team {
    int part, id;
    __device__ __forceinline__ void sync() const {
        if constexpr (W == 1)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "n"(32 * W) : "memory");
    }
};

template <int CPL>
__device__ __forceinline__ void ld_chan(float (&v)[CPL], const float* p) {
    if constexpr (CPL == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2*>(p);
        v[0] = t.x, v[1] = t.y;
    }
}

// tables, fragments of V (or its transpose), bias and lift into shared memory
template <int CP, int MP, bool TRANS>
__device__ __forceinline__ void row_setup(const RowArgs& a, float* sm, const RowSmem& L) {
    const int HP = half_pad(a.nx), XQ = inv_pad(a.nx), XL = (a.nx + 1) / 2, C = a.C;
    for (int e = threadIdx.x; e < MP * HP; e += blockDim.x) {
        sm[L.tf + e] = a.fc[e];
        sm[L.tf + MP * HP + e] = a.fs[e];
    }
    // inverse positions in the order a lane group takes them: four positions
    // spaced by 4 are one 16-byte load
    for (int e = threadIdx.x; e < MP * XQ; e += blockDim.x) {
        const int k = e / XQ, q = e - k * XQ, r = q & 15, x = (q & ~15) + (r >> 2) + 4 * (r & 3);
        sm[L.ti + e] = x < XL ? a.ic[k * HP + x] : 0.f;
        sm[L.ti + MP * XQ + e] = x < XL ? a.is[k * HP + x] : 0.f;
    }
    for (int e = threadIdx.x; e < MP; e += blockDim.x) sm[L.sp + e] = a.ic[e * HP + a.nx / 2];
    if (a.V) {
        constexpr int T = CP / 16;
        unsigned* w = reinterpret_cast<unsigned*>(sm + L.frag);
        for (int e = threadIdx.x; e < T * T * 32; e += blockDim.x) {
            const int lane = e & 31, tile = e >> 5, mt = tile / T, kt = tile - mt * T, g = lane >> 2, t = lane & 3;
            auto wv = [&](int mm, int kk) -> float {
                if (mm >= C || kk >= C) return 0.f;
                return TRANS ? a.V[kk * C + mm] : a.V[mm * C + kk];
            };
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int mm = mt * 16 + g + ((r & 1) ? 8 : 0), kk = kt * 16 + 2 * t + ((r & 2) ? 8 : 0);
                split2(wv(mm, kk), wv(mm, kk + 1), w[tile * 256 + lane * 4 + r], w[tile * 256 + 128 + lane * 4 + r]);
            }
        }
    }
    for (int e = threadIdx.x; e < CP; e += blockDim.x) {
        sm[L.bias + e] = a.vb && e < C ? a.vb[e] : 0.f;
#pragma unroll
        for (int f = 0; f < 4; ++f) sm[L.lift + 4 * e + f] = a.P && e < C ? a.P[e * 4 + f] : 0.f;
        sm[L.lift + 4 * CP + e] = a.pb && e < C ? a.pb[e] : 0.f;
    }
    // padded channels stay zero in every row
    for (int e = L.warp + threadIdx.x; e < L.warp + (int)(blockDim.x / 64) * L.perwarp; e += blockDim.x) sm[e] = 0.f;
}

// asynchronous global -> shared copies: a warp has a whole row in flight
// without holding it in registers (loaded through registers, 8 channels at a
// time, a row cost 16 trips to memory one after another)
__device__ __forceinline__ void cp4(float* dst, const float* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp16(float* dst, const float* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// the row's retained x modes: T1 -> [kx][channel], channels of a lane adjacent
// (zeros at the padded ones)
template <int CP, int MP, int W>
__device__ __forceinline__ void row_load_modes(const RowArgs& a, long long row, float* T, Team<W> tm) {
    constexpr int CPL = CP / 8, TS = CP + 4;
    const float* src = reinterpret_cast<const float*>(a.T1 + row * a.C * a.m);
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int e = lane + 32 * tm.part; e < MP * CP; e += 32 * W) {
        const int c = e / MP, k = e - c * MP;
        const bool in = c < a.C && k < a.m;
        const float* t = src + (in ? 2 * (c * a.m + k) : 0);
        const int o = k * TS + (c & 7) * CPL + (c >> 3);
        cp4(T + o, t, in);
        cp4(T + MP * TS + o, t + 1, in);
    }
}

// a row of C channels of src [C][N] into A
template <int W>
__device__ __forceinline__ void row_load(const RowArgs& a, const float* src, long long r0, float* A, int RS,
                                         Team<W> tm) {
    const int lane = threadIdx.x & 31;
    if (a.vec) {  // rows start on 16-byte boundaries
        for (int x = 4 * lane; x < a.nx; x += 128)
#pragma unroll 8
            for (int c = tm.part; c < a.C; c += W) cp16(A + c * RS + x, src + (long long)c * a.N + r0 + x);
    } else {
        for (int x = lane; x < a.nx; x += 32)
#pragma unroll 8
            for (int c = tm.part; c < a.C; c += W) cp4(A + c * RS + x, src + (long long)c * a.N + r0 + x, true);
    }
}

// A <- W A column tile by column tile on the tensor cores (W's fragments in shared memory)
template <int CP, int W>
__device__ __forceinline__ void row_dense(float* A, int RS, int nx, const unsigned* w, Team<W> tm) {
    constexpr int T = CP / 16;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    unsigned ah[T][T][4], al[T][T][4];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j) {
            const uint4 h = *reinterpret_cast<const uint4*>(w + (i * T + j) * 256 + lane * 4);
            const uint4 l = *reinterpret_cast<const uint4*>(w + (i * T + j) * 256 + 128 + lane * 4);
            ah[i][j][0] = h.x, ah[i][j][1] = h.y, ah[i][j][2] = h.z, ah[i][j][3] = h.w;
            al[i][j][0] = l.x, al[i][j][1] = l.y, al[i][j][2] = l.z, al[i][j][3] = l.w;
        }
    // two column tiles at a time: their chains of products overlap
    for (int n0 = 16 * tm.part; n0 < nx; n0 += 16 * W) {
        const bool two = n0 + 8 < nx;
        float acc[2][T][4] = {};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float* col = A + n0 + (u && two ? 8 : 0) + g;
#pragma unroll
            for (int j = 0; j < T; ++j) {
                const float* b = col + (j * 16 + 2 * t) * RS;
                unsigned bh0, bl0, bh1, bl1;
                split2(b[0], b[RS], bh0, bl0);
                split2(b[8 * RS], b[9 * RS], bh1, bl1);
#pragma unroll
                for (int i = 0; i < T; ++i) mma3(acc[u][i], ah[i][j], al[i][j], bh0, bh1, bl0, bl1);
            }
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (u == 0 || two)
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    float* o = A + (i * 16 + g) * RS + n0 + 8 * u + 2 * t;
                    *reinterpret_cast<float2*>(o) = make_float2(acc[u][i][0], acc[u][i][1]);
                    *reinterpret_cast<float2*>(o + 8 * RS) = make_float2(acc[u][i][2], acc[u][i][3]);
                }
        __syncwarp();
    }
}

// A += bias + inverse x transform of the modes in T: a lane takes CP/8
// channels at four positions x and their mirrors n - x
template <int CP, int MP, int W>
__device__ __forceinline__ void row_inverse_add(float* A, int RS, int nx, const float* T, const float* tic,
                                                const float* tis, const float* sp, const float* bias, Team<W> tm) {
    constexpr int CPL = CP / 8, TS = CP + 4;
    const int lane = threadIdx.x & 31, g = lane & 7, xg = lane >> 3;
    const int XL = (nx + 1) / 2, XQ = inv_pad(nx);
    for (int x0 = 16 * tm.part; x0 < XQ; x0 += 16 * W) {
        float c[CPL][4] = {}, s[CPL][4] = {};
#pragma unroll
        for (int k = 0; k < MP; ++k) {
            float tr[CPL], ti[CPL];
            ld_chan<CPL>(tr, T + k * TS + g * CPL);
            ld_chan<CPL>(ti, T + (MP + k) * TS + g * CPL);
            const float4 cc = *reinterpret_cast<const float4*>(tic + k * XQ + x0 + xg * 4);
            const float4 ss = *reinterpret_cast<const float4*>(tis + k * XQ + x0 + xg * 4);
            const float cv[4] = {cc.x, cc.y, cc.z, cc.w}, sv[4] = {ss.x, ss.y, ss.z, ss.w};
#pragma unroll
            for (int i = 0; i < CPL; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    c[i][j] = fmaf(tr[i], cv[j], c[i][j]);
                    s[i][j] = fmaf(ti[i], sv[j], s[i][j]);
                }
        }
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            float* r = A + (g + 8 * i) * RS;
            const float b = bias[g + 8 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int x = x0 + xg + 4 * j;
                if (x < XL) {
                    r[x] += c[i][j] - s[i][j] + b;
                    if (x > 0) r[nx - x] += c[i][j] + s[i][j] + b;
                }
            }
        }
    }
    if ((nx & 1) == 0 && lane < CP && tm.part == W - 1) {  // the position that is its own mirror
        const int slot = (lane & 7) * CPL + (lane >> 3);
        float v = bias[lane];
#pragma unroll
        for (int k = 0; k < MP; ++k) v = fmaf(T[k * TS + slot], sp[k], v);
        A[lane * RS + nx / 2] += v;
    }
}

// T1 <- forward x transform of the folded rows (sums at [0, HP), differences
// at [HP, 2 HP)): a lane takes CP/(8 W) channels and MP/4 modes
template <int CP, int MP, int W>
__device__ __forceinline__ void row_forward(const RowArgs& a, long long row, const float* A, int RS, float* T,
                                            const float* tfc, const float* tfs, Team<W> tm) {
    constexpr int CPL = CP / (8 * W), KPL = MP / 4;
    const int lane = threadIdx.x & 31, g = (lane & 7) + 8 * CPL * tm.part, kg = lane >> 3, HP = half_pad(a.nx);
    float re[CPL][KPL] = {}, im[CPL][KPL] = {};
#pragma unroll 2
    for (int x = 0; x < HP; x += 4) {
        float4 c[KPL], s[KPL];
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
            c[j] = *reinterpret_cast<const float4*>(tfc + (kg * KPL + j) * HP + x);
            s[j] = *reinterpret_cast<const float4*>(tfs + (kg * KPL + j) * HP + x);
        }
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            const float4 e = *reinterpret_cast<const float4*>(A + (g + 8 * i) * RS + x);
            const float4 o = *reinterpret_cast<const float4*>(A + (g + 8 * i) * RS + HP + x);
#pragma unroll
            for (int j = 0; j < KPL; ++j) {
                re[i][j] = fmaf(e.w, c[j].w, fmaf(e.z, c[j].z, fmaf(e.y, c[j].y, fmaf(e.x, c[j].x, re[i][j]))));
                im[i][j] = fmaf(o.w, s[j].w, fmaf(o.z, s[j].z, fmaf(o.y, s[j].y, fmaf(o.x, s[j].x, im[i][j]))));
            }
        }
    }
    // through shared memory (the modes of this row are used up) for a contiguous store
    float2* st = reinterpret_cast<float2*>(T);
#pragma unroll
    for (int i = 0; i < CPL; ++i)
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
            const int c = g + 8 * i, k = kg * KPL + j;
            if (c < a.C && k < a.m) st[c * a.m + k] = make_float2(re[i][j], -im[i][j]);
        }
    tm.sync();
    float2* dst = a.T1 + row * a.C * a.m;
    for (int e = lane + 32 * tm.part; e < a.C * a.m; e += 32 * W) dst[e] = st[e];
    tm.sync();
}

// in place: a row's values -> sums and differences under x -> n - x, after
// val(channel, x, value, pre(channel, x)).  The two positions that are their
// own mirrors, 0 and n/2, share a lane.  CB channels at a time: first every
// pre (a load, say), then the values.
template <int FI, int CB, int W, class G, class F>
__device__ __forceinline__ void row_fold(float* A, int RS, int nx, int C, Team<W> tm, G pre, F val) {
    const int lane = threadIdx.x & 31, HP = half_pad(nx), Hx = nx / 2 + 1, XL = (nx + 1) / 2;
    const bool even = (nx & 1) == 0;
    for (int c0 = CB * tm.part; c0 < C; c0 += CB * W) {
        float v[CB][FI], u[CB][FI];
        using P = decltype(pre(0, 0));
        P pv[CB][FI], pu[CB][FI];
#pragma unroll
        for (int q = 0; q < FI; ++q) {
            if (32 * q >= XL) break;  // the same for every lane: no instructions for positions no row has
            const int x = lane + 32 * q, y = x ? nx - x : nx / 2;
#pragma unroll
            for (int b = 0; b < CB; ++b)
                if (c0 + b < C && x < XL) {
                    pv[b][q] = pre(c0 + b, x);
                    if (x || even) pu[b][q] = pre(c0 + b, y);
                }
        }
#pragma unroll
        for (int q = 0; q < FI; ++q) {
            if (32 * q >= XL) break;
            const int x = lane + 32 * q, y = x ? nx - x : nx / 2;
#pragma unroll
            for (int b = 0; b < CB; ++b) {
                v[b][q] = u[b][q] = 0.f;
                if (c0 + b < C && x < XL) {
                    const float* r = A + (c0 + b) * RS;
                    v[b][q] = val(c0 + b, x, r[x], pv[b][q]);
                    if (x || even) u[b][q] = val(c0 + b, y, r[y], pu[b][q]);
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < CB; ++b) {
            if (c0 + b >= C) break;
            float* r = A + (c0 + b) * RS;
#pragma unroll
            for (int q = 0; q < FI; ++q) {
                if (32 * q >= XL) break;
                const int x = lane + 32 * q;
                if (x < XL) {
                    r[x] = x ? v[b][q] + u[b][q] : v[b][q];
                    r[HP + x] = x ? v[b][q] - u[b][q] : 0.f;
                    if (x == 0 && even) {
                        r[nx / 2] = u[b][q];
                        r[HP + nx / 2] = 0.f;
                    }
                }
            }
            if (lane < HP - Hx) r[Hx + lane] = r[HP + Hx + lane] = 0.f;
        }
    }
    tm.sync();
}

// lift of the row's input: a_0 = P x + p
template <int CP, int W>
__device__ __forceinline__ void row_lift(const RowArgs& a, long long r0, float* A, int RS, const float* lift,
                                         Team<W> tm) {
    for (int x = (threadIdx.x & 31) + 32 * tm.part; x < a.nx; x += 32 * W) {
        float v[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) v[f] = a.x[f * a.N + r0 + x];
        for (int c = 0; c < a.C; ++c) {
            const float4 w = *reinterpret_cast<const float4*>(lift + 4 * c);
            A[c * RS + x] = fmaf(w.w, v[3], fmaf(w.z, v[2], fmaf(w.y, v[1], fmaf(w.x, v[0], lift[4 * CP + c]))));
        }
    }
}

// T1 of the lifted input: the x transform of the four input fields, then
// P X + p (whose transform is p nx at kx = 0), a warp per row: the transform is
// linear, so it is taken of four fields instead of C (44 us at 128^3, C = 32,
// where the lift as a row pass took a layer's 246)
template <int MP>
__global__ void __launch_bounds__(256) k_fno_lift_modes(RowArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int HP = half_pad(a.nx), RS = row_pitch(a.nx), nx = a.nx;
    float *tc = sm, *ts = tc + MP * HP, *lift = ts + MP * HP;  // lift: [32][4] P, [32] p
    for (int e = threadIdx.x; e < MP * HP; e += blockDim.x) {
        tc[e] = a.fc[e];
        ts[e] = a.fs[e];
    }
    for (int e = threadIdx.x; e < 32; e += blockDim.x) {
#pragma unroll
        for (int f = 0; f < 4; ++f) lift[4 * e + f] = e < a.C ? a.P[e * 4 + f] : 0.f;
        lift[128 + e] = e < a.C ? a.pb[e] * (float)nx : 0.f;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float* A = lift + 160 + warp * (4 * RS + 8 * MP);
    float2* X = reinterpret_cast<float2*>(A + 4 * RS);  // [4][MP]
    for (long long row = blockIdx.x * (long long)nw + warp; row < a.rows; row += (long long)gridDim.x * nw) {
        for (int x = lane; x < nx; x += 32)
#pragma unroll
            for (int f = 0; f < 4; ++f) cp4(A + f * RS + x, a.x + f * a.N + row * nx + x, true);
        cp_wait();
        __syncwarp();
        row_fold<kFoldIter, 4>(
            A, RS, nx, 4, Team<1>{0, 0}, [](int, int) { return 0; }, [](int, int, float v, int) { return v; });
        const int f = lane & 3;
        for (int k = lane >> 2; k < a.m; k += 8) {
            float re = 0.f, im = 0.f;
            for (int x = 0; x < HP; x += 4) {
                const float4 c = *reinterpret_cast<const float4*>(tc + k * HP + x);
                const float4 s = *reinterpret_cast<const float4*>(ts + k * HP + x);
                const float4 e = *reinterpret_cast<const float4*>(A + f * RS + x);
                const float4 o = *reinterpret_cast<const float4*>(A + f * RS + HP + x);
                re = fmaf(e.w, c.w, fmaf(e.z, c.z, fmaf(e.y, c.y, fmaf(e.x, c.x, re))));
                im = fmaf(o.w, s.w, fmaf(o.z, s.z, fmaf(o.y, s.y, fmaf(o.x, s.x, im))));
            }
            X[f * MP + k] = make_float2(re, -im);
        }
        __syncwarp();
        float2* dst = a.T1 + row * a.C * a.m;
        for (int e = lane; e < a.C * a.m; e += 32) {
            const int c = e / a.m, k = e - c * a.m;
            const float4 w = *reinterpret_cast<const float4*>(lift + 4 * c);
            const float2 x0 = X[k], x1 = X[MP + k], x2 = X[2 * MP + k], x3 = X[3 * MP + k];
            dst[e] = make_float2(fmaf(w.w, x3.x, fmaf(w.z, x2.x, fmaf(w.y, x1.x, fmaf(w.x, x0.x, k ? 0.f : lift[128 + c])))),
                                 fmaf(w.w, x3.y, fmaf(w.z, x2.y, fmaf(w.y, x1.y, w.x * x0.y))));
        }
        __syncwarp();
    }
}

constexpr int kTeam = 2;  // warps of a row

// A layer forward.  It moves 2 [C][N] arrays (79 us at 128^3, C = 32, and 6.8
// TB/s) and is bound by instruction issue: 246 us, two thirds of the cycles
// issuing, of the products along x, GELU and the split into BF16 parts.  A row
// of all channels fills 20 KB, so ten rows an SM: with one warp a row that left
// two and a half warps a scheduler (402 us, with erff); two warps share a row.
template <int CP, int MP, int FI>
__global__ void __launch_bounds__(640, 1) k_fno_row(RowArgs a) {
    extern __shared__ __align__(16) float sm[];
    const RowSmem L = row_smem(a.nx, CP, MP);
    row_setup<CP, MP, false>(a, sm, L);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nt = blockDim.x / (32 * kTeam);
    const Team<kTeam> tm{warp % kTeam, warp / kTeam};
    const int nx = a.nx, C = a.C, RS = row_pitch(nx), HP = half_pad(nx), XQ = inv_pad(nx);
    float* A = sm + L.warp + tm.id * L.perwarp;
    float* T = A + CP * RS;
    for (long long row = blockIdx.x * (long long)nt + tm.id; row < a.rows; row += (long long)gridDim.x * nt) {
        const long long r0 = row * nx;
        if (a.dense) row_load_modes<CP, MP>(a, row, T, tm);
        if (a.zprev) row_load(a, a.zprev, r0, A, RS, tm);
        cp_wait();
        tm.sync();
        if (!a.zprev) {
            row_lift<CP>(a, r0, A, RS, sm + L.lift, tm);
        } else if (!a.raw) {
            for (int x = lane; x < nx; x += 32)
#pragma unroll 8
                for (int c = tm.part; c < C; c += kTeam) A[c * RS + x] = gelu_fast(A[c * RS + x]);
        }
        tm.sync();
        if (a.dense) {
            row_dense<CP>(A, RS, nx, reinterpret_cast<const unsigned*>(sm + L.frag), tm);
            tm.sync();
            row_inverse_add<CP, MP>(A, RS, nx, T, sm + L.ti, sm + L.ti + MP * XQ, sm + L.sp, sm + L.bias, tm);
            tm.sync();
        }
        if (a.last) {
            for (int x = lane; x < nx; x += 32)
#pragma unroll 8
                for (int c = tm.part; c < C; c += kTeam) a.z[(long long)c * a.N + r0 + x] = A[c * RS + x];
            tm.sync();
            continue;
        }
        if (a.dense) {
            row_fold<FI, 2>(
                A, RS, nx, C, tm, [](int, int) { return 0; },
                [&](int c, int x, float v, int) {
                    a.z[(long long)c * a.N + r0 + x] = v;
                    return gelu_fast(v);
                });
        } else {
            row_fold<FI, 2>(
                A, RS, nx, C, tm, [](int, int) { return 0; }, [](int, int, float v, int) { return v; });
        }
        row_forward<CP, MP>(a, row, A, RS, T, sm + L.tf, sm + L.tf + MP * HP, tm);
    }
}

// Partial sums of a block of k_fno_row_bwd: [C C] V, [C] v, [4 C] P, [C] p
__host__ __device__ inline int row_part_len(int C) { return C * C + 6 * C; }

// A layer backward: the gradient of its pre-activation in place of the next
// one's, the weights' partial sums over the block's rows.  It moves 3 [C][N]
// arrays (118 us at 128^3, C = 32) in 449 us, half the cycles issuing: two row
// tiles a team leave eight teams an SM, and 128 registers a thread.  810 us with
// a warp a row, 590 with the fold of long rows kept in registers for short ones.
template <int CP, int MP, int FI>
__global__ void __launch_bounds__(512, 1) k_fno_row_bwd(RowArgs a) {
    extern __shared__ __align__(16) float sm[];
    const RowSmem L = row_smem(a.nx, CP, MP);
    row_setup<CP, MP, true>(a, sm, L);
    __syncthreads();
    constexpr int MT = CP / 16, NT = CP / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nt = blockDim.x / (32 * kTeam);
    const int g = lane >> 2, t = lane & 3;
    const Team<kTeam> tm{warp % kTeam, warp / kTeam};
    const int nx = a.nx, C = a.C, RS = row_pitch(nx), HP = half_pad(nx), XQ = inv_pad(nx);
    const bool first = a.zprev == nullptr;
    float* A = sm + L.warp + tm.id * L.perwarp;
    float* T = A + CP * RS;
    const float* lift = sm + L.lift;
    float gV[MT][NT][4] = {}, gP[MT][4] = {}, sv[MT][2] = {}, sp[MT][2] = {};
    // A fragments (rows = channels of the shared-memory row, k = 16 points) and the row sums
    auto rows_frag = [&](int p, unsigned (&ah)[MT][4], unsigned (&al)[MT][4], float (&sum)[MT][2]) {
#pragma unroll
        for (int i = 0; i < MT; ++i) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int q = p + ((r & 2) ? 8 : 0);
                float2 u = *reinterpret_cast<const float2*>(A + (i * 16 + g + ((r & 1) ? 8 : 0)) * RS + (q < nx ? q : 0));
                if (q >= nx) u.x = 0.f;
                if (q + 1 >= nx) u.y = 0.f;
                sum[i][r & 1] += u.x + u.y;
                split2(u.x, u.y, ah[i][r], al[i][r]);
            }
        }
    };
    for (long long row = blockIdx.x * (long long)nt + tm.id; row < a.rows; row += (long long)gridDim.x * nt) {
        const long long r0 = row * nx;
        row_load_modes<CP, MP>(a, row, T, tm);
        row_load(a, a.z, r0, A, RS, tm);
        if (!first)  // the row of zprev on its way while dz arrives
            for (int e = lane + 32 * tm.part; e < C * ((nx + 31) / 32 + 1); e += 32 * kTeam) {
                const int c = e % C, x = min(32 * (e / C), nx - 1);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a.zprev + (long long)c * a.N + r0 + x));
            }
        cp_wait();
        tm.sync();
        // gradient of V: dz a^T over the row's points, a in fragments straight from global memory
        const float* zp = first ? nullptr : a.zprev + (g < C ? (long long)g * a.N : 0) + r0;
        for (int k0 = 16 * tm.part; k0 < nx; k0 += 16 * kTeam) {
            const int p = k0 + 2 * t;
            float av[NT][4];
            if (!first) {
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const bool dc = j * 8 + g < C;
                    const float* z = zp + (dc ? (long long)(j * 8) * a.N : 0);
                    if (a.vec) {  // p even, pairs 8-byte aligned, and nx even
                        const float2 lo = dc && p < nx ? *reinterpret_cast<const float2*>(z + p) : make_float2(0.f, 0.f);
                        const float2 hi =
                            dc && p + 8 < nx ? *reinterpret_cast<const float2*>(z + p + 8) : make_float2(0.f, 0.f);
                        av[j][0] = lo.x, av[j][1] = lo.y, av[j][2] = hi.x, av[j][3] = hi.y;
                    } else {
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const int q = p + (r & 1) + ((r & 2) ? 8 : 0);
                            av[j][r] = dc && q < nx ? z[q] : 0.f;
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < NT; ++j)
#pragma unroll
                    for (int r = 0; r < 4; ++r) av[j][r] = gelu_fast(av[j][r]);
            } else {
                float xv[4][4];
#pragma unroll
                for (int f = 0; f < 4; ++f)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int q = p + (r & 1) + ((r & 2) ? 8 : 0);
                        xv[f][r] = q < nx ? a.x[f * a.N + r0 + q] : 0.f;
                    }
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const float4 w = *reinterpret_cast<const float4*>(lift + 4 * (j * 8 + g));
                    const float b = lift[4 * CP + j * 8 + g];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        av[j][r] = fmaf(w.w, xv[3][r], fmaf(w.z, xv[2][r], fmaf(w.y, xv[1][r], fmaf(w.x, xv[0][r], b))));
                }
            }
            unsigned ah[MT][4], al[MT][4];
            rows_frag(p, ah, al, sv);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                unsigned bh0, bl0, bh1, bl1;
                split2(av[j][0], av[j][1], bh0, bl0);
                split2(av[j][2], av[j][3], bh1, bl1);
#pragma unroll
                for (int i = 0; i < MT; ++i) mma3(gV[i][j], ah[i], al[i], bh0, bh1, bl0, bl1);
            }
        }
        tm.sync();
        row_dense<CP>(A, RS, nx, reinterpret_cast<const unsigned*>(sm + L.frag), tm);
        tm.sync();
        row_inverse_add<CP, MP>(A, RS, nx, T, sm + L.ti, sm + L.ti + MP * XQ, sm + L.sp, sm + L.bias, tm);
        tm.sync();
        if (first) {
            // gradients of the lift: da x^T and the row sums
            for (int k0 = 16 * tm.part; k0 < nx; k0 += 16 * kTeam) {
                const int p = k0 + 2 * t;
                float xv[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int q = p + (r & 1) + ((r & 2) ? 8 : 0);
                    xv[r] = g < 4 && q < nx ? a.x[g * a.N + r0 + q] : 0.f;
                }
                unsigned ah[MT][4], al[MT][4], bh0, bl0, bh1, bl1;
                rows_frag(p, ah, al, sp);
                split2(xv[0], xv[1], bh0, bl0);
                split2(xv[2], xv[3], bh1, bl1);
#pragma unroll
                for (int i = 0; i < MT; ++i) mma3(gP[i], ah[i], al[i], bh0, bh1, bl0, bl1);
            }
            tm.sync();
            continue;
        }
        row_fold<FI, 2>(
            A, RS, nx, C, tm, [&](int c, int x) { return a.zprev[(long long)c * a.N + r0 + x]; },
            [&](int c, int x, float v, float z) {
                const float d = v * gelu_fast_g(z);
                a.z[(long long)c * a.N + r0 + x] = d;
                return d;
            });
        row_forward<CP, MP>(a, row, A, RS, T, sm + L.tf, sm + L.tf + MP * HP, tm);
    }
    // the warps of a row add up in its shared memory one after another, then
    // the rows, each in order
    const int E = row_part_len(C);
    float* own = A;  // CP row_pitch + 2 MP (CP + 4) floats: E of them from nx = 32 on
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            sv[i][r] += __shfl_xor_sync(0xffffffffu, sv[i][r], 1);
            sv[i][r] += __shfl_xor_sync(0xffffffffu, sv[i][r], 2);
            sp[i][r] += __shfl_xor_sync(0xffffffffu, sp[i][r], 1);
            sp[i][r] += __shfl_xor_sync(0xffffffffu, sp[i][r], 2);
        }
    for (int w = 0; w < kTeam; ++w) {
        __syncthreads();
        if (tm.part != w) continue;
        auto put = [&](int e, float v) { own[e] = w ? own[e] + v : v; };
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int c = i * 16 + g + ((r & 2) ? 8 : 0);
                if (c < C) {
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        const int d = j * 8 + 2 * t + (r & 1);
                        if (d < C) put(c * C + d, gV[i][j][r]);
                    }
                    if (2 * t + (r & 1) < 4) put(C * C + C + c * 4 + 2 * t + (r & 1), gP[i][r]);
                }
            }
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int c = i * 16 + g + 8 * r;
                if (t == 0 && c < C) {
                    put(C * C + c, sv[i][r]);
                    put(C * C + 5 * C + c, sp[i][r]);
                }
            }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        float v = 0.f;
        for (int w = 0; w < nt; ++w) v += sm[L.warp + w * L.perwarp + e];
        a.part[(long long)blockIdx.x * E + e] = v;
    }
}

// ---------------------------------------------------------------------------
// transforms along y or z of the retained modes: modes 0..m-1 and -m..-1.
// With E(j) = v(j) + v(J - j), O(j) = v(j) - v(J - j), the sums
// P_k = sum_j E cos, Q_k = sum_j O sin give F(+-k) = P_k -+ i Q_k, a quarter
// of the products of the plain contraction.  tab[j][k] = (cos, sin), k <= m.
// A thread takes a column of the contiguous inner index and all modes of it in
// registers, so rows come in whole (a thread per output read its J values again
// for every mode).  Along z there are few columns (144 blocks of 64 at 24 y
// modes), so forward four threads share a column's positions: 15.7 us a launch
// at 128^3, 12 modes, C = 32, mean of y and z, where one thread a column took
// 24.9; back 11.
// ---------------------------------------------------------------------------
constexpr int kDftCols = 64;   // columns of a block
constexpr int kDftParts = 4;   // parts of the positions, each summed by kDftCols threads
template <int MP>
constexpr size_t dft_sum_bytes() {  // two parts' sums P, Q
    return (kDftParts / 2) * 2 * (MP + 1) * kDftCols * sizeof(float2);
}
template <int MP>
__global__ void __launch_bounds__(kDftCols* kDftParts) k_dft_modes(const float2* __restrict__ in, float2* __restrict__ out,
                                                                   const float2* __restrict__ tab, int J, int m, int I) {
    extern __shared__ __align__(16) float2 st[];  // [J/2 + 1][MP + 2]; then the sums of two parts
    constexpr int TP = MP + 2;
    for (int e = threadIdx.x; e < (J / 2 + 1) * TP; e += blockDim.x) {
        const int j = e / TP, k = e - j * TP;
        st[e] = k <= m ? tab[j * (m + 1) + k] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int col = threadIdx.x % kDftCols, part = threadIdx.x / kDftCols;
    const int i = blockIdx.x * kDftCols + col;
    const bool ok = i < I;
    const float2* src = in + (long long)blockIdx.y * J * I + (ok ? i : 0);
    float2 P[MP + 1], Q[MP + 1];
#pragma unroll
    for (int k = 0; k <= MP; ++k) P[k] = Q[k] = make_float2(0.f, 0.f);
    auto add = [&](int j, float2 e, float2 o) {
        const float4* row = reinterpret_cast<const float4*>(st + j * TP);
#pragma unroll
        for (int k2 = 0; k2 < TP / 2; ++k2) {
            const float4 w = row[k2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = 2 * k2 + h;
                if (k <= MP) {
                    const float c = h ? w.z : w.x, s = h ? w.w : w.y;
                    P[k].x = fmaf(c, e.x, P[k].x);
                    P[k].y = fmaf(c, e.y, P[k].y);
                    Q[k].x = fmaf(s, o.x, Q[k].x);
                    Q[k].y = fmaf(s, o.y, Q[k].y);
                }
            }
        }
    };
    const float2 z = make_float2(0.f, 0.f);
    const int pairs = (J - 1) / 2, per = (pairs + kDftParts - 1) / kDftParts;
    const int end = min(pairs, (part + 1) * per);
    if (part == 0) add(0, src[0], z);
    if (part == kDftParts - 1 && (J & 1) == 0) add(J / 2, src[(long long)(J / 2) * I], z);
    // eight pairs' loads in flight: a thread's trips to memory, not its
    // products, set the time
    for (int j = 1 + part * per; j <= end; j += 8) {
        float2 a[8], b[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool in_part = j + u <= end;
            a[u] = in_part ? src[(long long)(j + u) * I] : z;
            b[u] = in_part ? src[(long long)(J - j - u) * I] : z;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j + u <= end)
                add(j + u, make_float2(a[u].x + b[u].x, a[u].y + b[u].y), make_float2(a[u].x - b[u].x, a[u].y - b[u].y));
    }
    // the upper half of the parts hands its sums to the lower one
#pragma unroll
    for (int n = kDftParts / 2; n > 0; n /= 2) {
        __syncthreads();  // the table, or the sums before, are read
        if (part >= n && part < 2 * n) {
            float2* d = st + (size_t)(part - n) * 2 * (MP + 1) * kDftCols + col;
#pragma unroll
            for (int k = 0; k <= MP; ++k) {
                d[(2 * k) * kDftCols] = P[k];
                d[(2 * k + 1) * kDftCols] = Q[k];
            }
        }
        __syncthreads();
        if (part < n) {
            const float2* d = st + (size_t)part * 2 * (MP + 1) * kDftCols + col;
#pragma unroll
            for (int k = 0; k <= MP; ++k) {
                const float2 p = d[(2 * k) * kDftCols], q = d[(2 * k + 1) * kDftCols];
                P[k] = make_float2(P[k].x + p.x, P[k].y + p.y);
                Q[k] = make_float2(Q[k].x + q.x, Q[k].y + q.y);
            }
        }
    }
    if (part > 0 || !ok) return;
    float2* dst = out + (long long)blockIdx.y * 2 * m * I + i;
#pragma unroll
    for (int k = 0; k <= MP; ++k) {
        if (k < m) dst[(long long)k * I] = make_float2(P[k].x + Q[k].y, P[k].y - Q[k].x);
        if (k > 0 && k <= m) dst[(long long)(2 * m - k) * I] = make_float2(P[k].x - Q[k].y, P[k].y + Q[k].x);
    }
}

// out(j) = sum over the modes of in e^{+2 pi i k j / J}, positions j and J - j
// together, blockIdx.z-th part of the positions
template <int MP>
__global__ void __launch_bounds__(64) k_dft_modes_inv(const float2* __restrict__ in, float2* __restrict__ out,
                                                      const float2* __restrict__ tab, int J, int m, int I) {
    extern __shared__ __align__(16) float2 st[];
    constexpr int TP = MP + 2;
    const int half = J / 2 + 1, per = (half + gridDim.z - 1) / gridDim.z;
    const int j0 = blockIdx.z * per, j1 = min(half, j0 + per);
    for (int e = threadIdx.x; e < (j1 - j0) * TP; e += blockDim.x) {
        const int j = e / TP, k = e - j * TP;
        st[e] = k <= m ? tab[(j0 + j) * (m + 1) + k] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= I) return;
    const float2* src = in + (long long)blockIdx.y * 2 * m * I + i;
    float2 U[MP + 1], V[MP + 1];
#pragma unroll
    for (int k = 0; k <= MP; ++k) {
        const float2 a = k < m ? src[(long long)k * I] : make_float2(0.f, 0.f);
        const float2 b = k > 0 && k <= m ? src[(long long)(2 * m - k) * I] : make_float2(0.f, 0.f);
        U[k] = make_float2(a.x + b.x, a.y + b.y);
        V[k] = make_float2(a.x - b.x, a.y - b.y);
    }
    float2* dst = out + (long long)blockIdx.y * J * I + i;
    for (int j = j0; j < j1; ++j) {
        const float4* row = reinterpret_cast<const float4*>(st + (j - j0) * TP);
        float2 P = make_float2(0.f, 0.f), Q = make_float2(0.f, 0.f);
#pragma unroll
        for (int k2 = 0; k2 < TP / 2; ++k2) {
            const float4 w = row[k2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = 2 * k2 + h;
                if (k <= MP) {
                    const float c = h ? w.z : w.x, s = h ? w.w : w.y;
                    P.x = fmaf(c, U[k].x, P.x);
                    P.y = fmaf(c, U[k].y, P.y);
                    Q.x = fmaf(s, V[k].x, Q.x);
                    Q.y = fmaf(s, V[k].y, Q.y);
                }
            }
        }
        dst[(long long)j * I] = make_float2(P.x - Q.y, P.y + Q.x);
        if (j > 0 && 2 * j != J) dst[(long long)(J - j) * I] = make_float2(P.x + Q.y, P.y - Q.x);
    }
}

// ---------------------------------------------------------------------------
// per-mode channel mix: one block per (jz, jy), a warp per kx.
// O[c] = sum_d W[c][d] A[d]: a lane takes row c of the mode's matrix, in
// 16-byte pieces where rows are 16-byte aligned (C a multiple of 4).  Every
// weight is read once: 28 MB of BF16 in 12 us at 12 modes, C = 32, and 37 us
// back, which writes 57 MB of gradients.
// ---------------------------------------------------------------------------
template <bool VEC>
__global__ void __launch_bounds__(256) k_mix_modes(const float2* __restrict__ A, float2* __restrict__ O,
                                                   const __nv_bfloat162* __restrict__ w16, int C, int m) {
    extern __shared__ __align__(16) float2 st[];  // [C m] in, [C m] out
    const long long b = blockIdx.x;
    float2* so = st + C * m;
    for (int e = threadIdx.x; e < C * m; e += blockDim.x) st[e] = A[b * C * m + e];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int kx = threadIdx.x >> 5; kx < m; kx += blockDim.x >> 5) {
        if (lane < C) {
            const __nv_bfloat162* w = w16 + ((b * m + kx) * C + lane) * C;
            float ar = 0.f, ai = 0.f;
            auto add = [&](unsigned u, int d) {
                const float wx = __uint_as_float(u << 16), wy = __uint_as_float(u & 0xffff0000u);
                const float2 v = st[d * m + kx];
                ar = fmaf(-wy, v.y, fmaf(wx, v.x, ar));
                ai = fmaf(wy, v.x, fmaf(wx, v.y, ai));
            };
            if constexpr (VEC) {
#pragma unroll 8
                for (int d = 0; d < C; d += 4) {
                    const uint4 u = __ldg(reinterpret_cast<const uint4*>(w + d));
                    add(u.x, d);
                    add(u.y, d + 1);
                    add(u.z, d + 2);
                    add(u.w, d + 3);
                }
            } else {
                for (int d = 0; d < C; ++d) add(*reinterpret_cast<const unsigned*>(w + d), d);
            }
            so[lane * m + kx] = make_float2(ar, ai);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < C * m; e += blockDim.x) O[b * C * m + e] = so[e];
}

// GA[d] = sum_c conj(W[c][d]) GO[c]; GW[c][d] = GO[c] conj(A[d]): a lane takes column d
__global__ void __launch_bounds__(256) k_mix_modes_bwd(const float2* __restrict__ GO, const float2* __restrict__ A,
                                                       float2* __restrict__ GA, float2* __restrict__ GW,
                                                       const __nv_bfloat162* __restrict__ w16, int C, int m) {
    extern __shared__ __align__(16) float2 st[];  // [C m] GO, A, GA
    const long long b = blockIdx.x;
    float2 *sa = st + C * m, *so = sa + C * m;
    for (int e = threadIdx.x; e < C * m; e += blockDim.x) {
        st[e] = GO[b * C * m + e];
        sa[e] = A[b * C * m + e];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int kx = threadIdx.x >> 5; kx < m; kx += blockDim.x >> 5) {
        if (lane < C) {
            const long long w0 = (b * m + kx) * C * C + lane;
            const float2 a = sa[lane * m + kx];
            float ar = 0.f, ai = 0.f;
#pragma unroll 8
            for (int c = 0; c < C; ++c) {
                const unsigned u = *reinterpret_cast<const unsigned*>(w16 + w0 + c * C);
                const float wx = __uint_as_float(u << 16), wy = __uint_as_float(u & 0xffff0000u);
                const float2 g = st[c * m + kx];
                ar = fmaf(wy, g.y, fmaf(wx, g.x, ar));
                ai = fmaf(-wy, g.x, fmaf(wx, g.y, ai));
                GW[w0 + c * C] = make_float2(g.x * a.x + g.y * a.y, g.y * a.x - g.x * a.y);
            }
            so[lane * m + kx] = make_float2(ar, ai);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < C * m; e += blockDim.x) GA[b * C * m + e] = so[e];
}

// ---------------------------------------------------------------------------
// projection: tiles of 64 points; a warp owns 16 of the H rows.
// ---------------------------------------------------------------------------
// points of a tile and the pitch of its rows: 8 (mod 32), so that the 8-byte
// reads of a fragment along the points (rows g) and, with the rows of a k tile
// taken in the order t, t + 4, t + 8, t + 12 (krow), the 4-byte ones across the
// rows are free of bank conflicts
constexpr int kPts = 64, kPS = 72;
// row of a k tile behind slot 2 t + i (i = 0, 1) and 2 t + 8 + i (i = 2, 3) of lane t
__device__ __forceinline__ int krow(int t, int i) { return t + 4 * i; }
__host__ __device__ inline int proj_part_len(int C, int H) { return H * C + 5 * H + 4; }
struct ProjArgs {
    const float *a, *tgt, *Q1, *q1, *Q2, *q2;
    float *out, *da, *part;
    double* dpart;
    int C, H;
    long long N;
    float sc;  // 2 / (4 N)
};
template <int CP, int NW, bool TRAIN, bool FULL>
constexpr int proj_smem() {
    constexpr int HP = 16 * NW, KT = CP / 16;
    return (2 * CP * kPS + HP * kPS + 4 * kPS + NW * 128 + 4 * HP + HP + 4 + (FULL ? HP * (CP + 4) : NW * KT * 256) +
            (TRAIN ? NW * KT * 256 : 0)) * 4;
}

// Hidden widths whose row tiles are no power of two (33 to 48, 65 to 112) have
// the product Q1 a in FP32, the others in BF16 parts: so it is in the kernels
// of one operation each (dense_mma has forms for 1, 2, 4 and 8 row tiles), and
// which of the two paths a size runs says nothing about its precision.  A forward
// pass at 64^3, C = 20, H = 100, 12 modes, four layers takes 441 us so, 423 with
// BF16 parts; at 160x160x40, C = 16, H = 112 1122 and 1029.
__host__ __device__ constexpr bool proj_full(int H) {
    const int tiles = (H + 15) / 16;
    return (tiles & (tiles - 1)) != 0;
}

// The products of a tile run on the tensor cores (1110 us forward and backward
// at 128^3, C = 32, H = 128, 1031 with GELU's derivative from the tail alone, 1708
// with the output and its weight gradient as scalar loops as well; 394 us forward
// at 160x96x120).  What bounds the kernel is
// the instructions around them, GELU of its H x 64 hidden values first, and the
// shared memory those pass through.  The next tile's columns of a are copied in
// while this one is worked on.
template <int CP, int NW, bool TRAIN, bool FULL>
__global__ void __launch_bounds__(32 * NW, 2) k_fno_project(ProjArgs p) {
    constexpr int HP = 16 * NW, KT = CP / 16, NT = kPts / 8;
    extern __shared__ __align__(16) float sm[];
    float* sa0 = sm;                  // [2][CP][kPS]
    float* sh = sa0 + 2 * CP * kPS;   // [HP][kPS]: h, then dh
    float* sd = sh + HP * kPS;        // [4][kPS]: d out
    uint4* w2 = reinterpret_cast<uint4*>(sd + 4 * kPS);  // Q2 fragments [NW][32]: rows 0..3, leading and remainder
    float* sq2 = sd + 4 * kPS + NW * 128;  // [HP][4]
    float* sq1 = sq2 + 4 * HP;             // [HP]
    float* sb2 = sq1 + HP;                 // [4]
    unsigned* w1 = reinterpret_cast<unsigned*>(sb2 + 4);  // Q1 fragments [NW][KT], or (FULL) Q1 itself
    float* f1 = sb2 + 4;                                  // [HP][FS]
    constexpr int FS = CP + 4;
    unsigned* wt = w1 + (FULL ? HP * FS : NW * KT * 256);  // Q1^T fragments [KT][NW]
    const int C = p.C, H = p.H;
    auto q1v = [&](int h, int c) -> float { return h < H && c < C ? p.Q1[h * C + c] : 0.f; };
    for (int e = threadIdx.x; e < NW * KT * 32; e += blockDim.x) {
        const int lane = e & 31, tile = e >> 5, g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int mm = g + ((r & 1) ? 8 : 0), k0 = krow(t, r & 2), k1 = krow(t, (r & 2) + 1);
            const int mt = tile / KT, kt = tile - mt * KT;
            if constexpr (!FULL)
                split2(q1v(mt * 16 + mm, kt * 16 + k0), q1v(mt * 16 + mm, kt * 16 + k1), w1[tile * 256 + lane * 4 + r],
                       w1[tile * 256 + 128 + lane * 4 + r]);
            if (TRAIN) {
                const int ct = tile / NW, ht = tile - ct * NW;
                split2(q1v(ht * 16 + k0, ct * 16 + mm), q1v(ht * 16 + k1, ct * 16 + mm),
                       wt[tile * 256 + lane * 4 + r], wt[tile * 256 + 128 + lane * 4 + r]);
            }
        }
    }
    if constexpr (FULL)
        for (int e = threadIdx.x; e < HP * CP; e += blockDim.x) f1[e / CP * FS + e % CP] = q1v(e / CP, e % CP);
    for (int e = threadIdx.x; e < NW * 32; e += blockDim.x) {
        const int g = (e & 31) >> 2, h = (e >> 5) * 16 + (e & 3);
        auto v = [&](int hh) -> float { return g < 4 && hh < H ? p.Q2[g * H + hh] : 0.f; };
        uint4 w;
        split2(v(h), v(h + 4), w.x, w.z);
        split2(v(h + 8), v(h + 12), w.y, w.w);
        w2[e] = w;
    }
    for (int e = threadIdx.x; e < HP; e += blockDim.x) {
#pragma unroll
        for (int f = 0; f < 4; ++f) sq2[4 * e + f] = e < H ? p.Q2[f * H + e] : 0.f;
        sq1[e] = e < H ? p.q1[e] : 0.f;
    }
    if (threadIdx.x < 4) sb2[threadIdx.x] = p.q2[threadIdx.x];
    for (int e = threadIdx.x; e < 2 * CP * kPS; e += blockDim.x) sa0[e] = 0.f;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const long long tiles = (p.N + kPts - 1) / kPts;
    auto load = [&](long long tile, float* dst) {
        const long long p0 = tile * kPts;
        if (p.N % 4 == 0 && p0 + kPts <= p.N) {
            for (int e = threadIdx.x; e < C * (kPts / 4); e += blockDim.x) {
                const int c = e / (kPts / 4), q = 4 * (e % (kPts / 4));
                cp16(dst + c * kPS + q, p.a + (long long)c * p.N + p0 + q);
            }
        } else {
            for (int e = threadIdx.x; e < C * kPts; e += blockDim.x) {
                const int c = e / kPts, q = e % kPts;
                const bool in = p0 + q < p.N;
                cp4(dst + c * kPS + q, p.a + (long long)c * p.N + (in ? p0 + q : 0), in);
            }
        }
    };
    // gradients kept over the block's tiles
    float gQ1[CP / 8][4] = {}, gq1[2] = {}, gQ2[4] = {};
    float gq2 = 0.f;
    double loss = 0.0;
    const int h0 = warp * 16;
    int cur = 0;
    if (blockIdx.x < tiles) load(blockIdx.x, sa0);
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x, cur ^= 1) {
        const long long p0 = tile * kPts;
        const int np = (int)min((long long)kPts, p.N - p0);
        const float* sa = sa0 + cur * CP * kPS;
        cp_wait();
        __syncthreads();
        if (tile + gridDim.x < tiles) load(tile + gridDim.x, sa0 + (cur ^ 1) * CP * kPS);
        // this warp's targets: fields 0..3 on the first 16 lanes
        float tg[TRAIN ? NT / NW + 1 : 1][2] = {};
        if constexpr (TRAIN) {
#pragma unroll
            for (int u = 0; u < NT / NW; ++u)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int q = (warp + u * NW) * 8 + 2 * t + r;
                    if (g < 4 && q < np) tg[u][r] = p.tgt[(long long)g * p.N + p0 + q];
                }
        }
        // h = GELU(Q1 a + q1) of this warp's rows; its derivative stays in registers
        float gp[TRAIN ? NT : 1][4];
        {
            const float b0 = sq1[h0 + g], b1 = sq1[h0 + g + 8];
            // column tile n of the pre-activations: GELU into sh
            auto hidden = [&](int n, const float (&acc)[4]) {
                float hv[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const GaussTail gt = gauss_tail(acc[r]);
                    hv[r] = gelu_of(acc[r], gt);
                    if (TRAIN) gp[n][r] = gelu_deriv_of(acc[r], gt);
                }
                float* o = sh + (h0 + g) * kPS + n * 8 + 2 * t;
                *reinterpret_cast<float2*>(o) = make_float2(hv[0], hv[1]);
                *reinterpret_cast<float2*>(o + 8 * kPS) = make_float2(hv[2], hv[3]);
            };
            if constexpr (FULL) {
                const float *q0 = f1 + (h0 + g) * FS, *q8 = q0 + 8 * FS;
                constexpr int NB = 4;  // column tiles at a time
#pragma unroll
                for (int n0 = 0; n0 < NT; n0 += NB) {
                    float acc[NB][4];
#pragma unroll
                    for (int u = 0; u < NB; ++u) acc[u][0] = acc[u][1] = b0, acc[u][2] = acc[u][3] = b1;
#pragma unroll 4
                    for (int c = 0; c < C; ++c) {
                        const float w0 = q0[c], w8 = q8[c];
#pragma unroll
                        for (int u = 0; u < NB; ++u) {
                            const float2 v = *reinterpret_cast<const float2*>(sa + c * kPS + (n0 + u) * 8 + 2 * t);
                            acc[u][0] = fmaf(w0, v.x, acc[u][0]);
                            acc[u][1] = fmaf(w0, v.y, acc[u][1]);
                            acc[u][2] = fmaf(w8, v.x, acc[u][2]);
                            acc[u][3] = fmaf(w8, v.y, acc[u][3]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < NB; ++u) hidden(n0 + u, acc[u]);
                }
            } else {
                unsigned ah[KT][4], al[KT][4];
#pragma unroll
                for (int k = 0; k < KT; ++k) {
                    const uint4 hv = *reinterpret_cast<const uint4*>(w1 + (warp * KT + k) * 256 + lane * 4);
                    const uint4 lv = *reinterpret_cast<const uint4*>(w1 + (warp * KT + k) * 256 + 128 + lane * 4);
                    ah[k][0] = hv.x, ah[k][1] = hv.y, ah[k][2] = hv.z, ah[k][3] = hv.w;
                    al[k][0] = lv.x, al[k][1] = lv.y, al[k][2] = lv.z, al[k][3] = lv.w;
                }
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    float acc[4] = {b0, b0, b1, b1};
#pragma unroll
                    for (int k = 0; k < KT; ++k) {
                        const float* b = sa + (k * 16 + t) * kPS + n * 8 + g;
                        unsigned bh0, bl0, bh1, bl1;
                        split2(b[0], b[4 * kPS], bh0, bl0);
                        split2(b[8 * kPS], b[12 * kPS], bh1, bl1);
                        mma3(acc, ah[k], al[k], bh0, bh1, bl0, bl1);
                    }
                    hidden(n, acc);
                }
            }
        }
        __syncthreads();
        // out = Q2 h + q2, eight points a warp at a time
#pragma unroll
        for (int u = 0; u < NT / NW; ++u) {
            const int n = warp + u * NW;
            const float b = g < 4 ? sb2[g] : 0.f;
            float acc[2][4] = {{b, b, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const float* hb = sh + (k * 16 + t) * kPS + n * 8 + g;
                unsigned bh0, bl0, bh1, bl1;
                split2(hb[0], hb[4 * kPS], bh0, bl0);
                split2(hb[8 * kPS], hb[12 * kPS], bh1, bl1);
                const uint4 w = w2[k * 32 + lane];
                const unsigned ah[4] = {w.x, 0u, w.y, 0u}, al[4] = {w.z, 0u, w.w, 0u};
                mma3(acc[k & 1], ah, al, bh0, bh1, bl0, bl1);
            }
            if (g < 4) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int q = n * 8 + 2 * t + r;
                    const float v = acc[0][r] + acc[1][r];
                    if constexpr (TRAIN) {
                        float d = 0.f;
                        if (q < np) {
                            d = v - tg[u][r];
                            loss += (double)d * d;
                            d *= p.sc;
                        }
                        sd[g * kPS + q] = d;
                        gq2 += d;
                    } else if (q < np) {
                        p.out[(long long)g * p.N + p0 + q] = v;
                    }
                }
            }
        }
        if constexpr (TRAIN) {
            __syncthreads();
            // gradient of Q2 (transposed: rows h, columns the fields): h d out^T
#pragma unroll
            for (int k = 0; k < kPts / 16; ++k) {
                unsigned ah[4], al[4], bh0, bl0, bh1, bl1;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float2 u = *reinterpret_cast<const float2*>(sh + (h0 + g + ((r & 1) ? 8 : 0)) * kPS + k * 16 +
                                                                      2 * t + ((r & 2) ? 8 : 0));
                    split2(u.x, u.y, ah[r], al[r]);
                }
                const float* d = sd + (g & 3) * kPS + k * 16 + 2 * t;
                float2 d0 = *reinterpret_cast<const float2*>(d), d1 = *reinterpret_cast<const float2*>(d + 8);
                if (g >= 4) d0 = d1 = make_float2(0.f, 0.f);
                split2(d0.x, d0.y, bh0, bl0);
                split2(d1.x, d1.y, bh1, bl1);
                mma3(gQ2, ah, al, bh0, bh1, bl0, bl1);
            }
            __syncwarp();
            // dh = GELU' (Q2^T d out) over h, and the gradient of Q1, dh a^T over
            // the tile's points: two column tiles of dh are an A fragment as
            // they stand in the registers
            {
                const float4 qa = *reinterpret_cast<const float4*>(sq2 + 4 * (h0 + g));
                const float4 qb = *reinterpret_cast<const float4*>(sq2 + 4 * (h0 + g + 8));
#pragma unroll
                for (int k = 0; k < NT / 2; ++k) {
                    unsigned ah[4], al[4];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int n = 2 * k + u;
                        const float* d = sd + n * 8 + 2 * t;
                        const float2 d0 = *reinterpret_cast<const float2*>(d);
                        const float2 d1 = *reinterpret_cast<const float2*>(d + kPS);
                        const float2 d2 = *reinterpret_cast<const float2*>(d + 2 * kPS);
                        const float2 d3 = *reinterpret_cast<const float2*>(d + 3 * kPS);
                        const float v0 = gp[n][0] * (qa.x * d0.x + qa.y * d1.x + qa.z * d2.x + qa.w * d3.x);
                        const float v1 = gp[n][1] * (qa.x * d0.y + qa.y * d1.y + qa.z * d2.y + qa.w * d3.y);
                        const float v2 = gp[n][2] * (qb.x * d0.x + qb.y * d1.x + qb.z * d2.x + qb.w * d3.x);
                        const float v3 = gp[n][3] * (qb.x * d0.y + qb.y * d1.y + qb.z * d2.y + qb.w * d3.y);
                        gq1[0] += v0 + v1;
                        gq1[1] += v2 + v3;
                        float* o = sh + (h0 + g) * kPS + n * 8 + 2 * t;
                        *reinterpret_cast<float2*>(o) = make_float2(v0, v1);
                        *reinterpret_cast<float2*>(o + 8 * kPS) = make_float2(v2, v3);
                        split2(v0, v1, ah[2 * u], al[2 * u]);
                        split2(v2, v3, ah[2 * u + 1], al[2 * u + 1]);
                    }
#pragma unroll
                    for (int j = 0; j < CP / 8; ++j) {
                        const float* b = sa + (j * 8 + g) * kPS + k * 16 + 2 * t;
                        const float2 u0 = *reinterpret_cast<const float2*>(b);
                        const float2 u1 = *reinterpret_cast<const float2*>(b + 8);
                        unsigned bh0, bl0, bh1, bl1;
                        split2(u0.x, u0.y, bh0, bl0);
                        split2(u1.x, u1.y, bh1, bl1);
                        mma3(gQ1[j], ah, al, bh0, bh1, bl0, bl1);
                    }
                }
            }
            __syncthreads();
            // da = Q1^T dh: a warp takes 16 channels of NT KT / NW column tiles
            {
                constexpr int NG = NW / KT, NU = NT / NG;
                const int i = warp % KT, ng = warp / KT;
                float acc[NU][4] = {};
#pragma unroll 4
                for (int k = 0; k < NW; ++k) {
                    const uint4 hv = *reinterpret_cast<const uint4*>(wt + (i * NW + k) * 256 + lane * 4);
                    const uint4 lv = *reinterpret_cast<const uint4*>(wt + (i * NW + k) * 256 + 128 + lane * 4);
                    const unsigned ah[4] = {hv.x, hv.y, hv.z, hv.w}, al[4] = {lv.x, lv.y, lv.z, lv.w};
#pragma unroll
                    for (int u = 0; u < NU; ++u) {
                        const float* b = sh + (k * 16 + t) * kPS + (ng * NU + u) * 8 + g;
                        unsigned bh0, bl0, bh1, bl1;
                        split2(b[0], b[4 * kPS], bh0, bl0);
                        split2(b[8 * kPS], b[12 * kPS], bh1, bl1);
                        mma3(acc[u], ah, al, bh0, bh1, bl0, bl1);
                    }
                }
#pragma unroll
                for (int u = 0; u < NU; ++u)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int c = i * 16 + g + ((r & 2) ? 8 : 0), q = (ng * NU + u) * 8 + 2 * t + (r & 1);
                        if (c < C && q < np) p.da[(long long)c * p.N + p0 + q] = acc[u][r];
                    }
            }
        }
    }
    if constexpr (TRAIN) {
        // block partials: [H C] Q1, [H] q1, [4 H] Q2, [4] q2; the loss in FP64
        float* o = p.part + (long long)blockIdx.x * proj_part_len(C, H);
#pragma unroll
        for (int j = 0; j < CP / 8; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int h = h0 + g + ((r & 2) ? 8 : 0), c = j * 8 + 2 * t + (r & 1);
                if (h < H && c < C) o[h * C + c] = gQ1[j][r];
            }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int h = h0 + g + ((r & 2) ? 8 : 0), f = 2 * t + (r & 1);
            if (h < H && f < 4) o[H * C + H + f * H + h] = gQ2[r];
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float v = gq1[r];
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            const int h = h0 + g + 8 * r;
            if (t == 0 && h < H) o[H * C + h] = v;
        }
        __shared__ double red[NW];
        __shared__ float red2[NW][4];
        gq2 += __shfl_xor_sync(0xffffffffu, gq2, 1);
        gq2 += __shfl_xor_sync(0xffffffffu, gq2, 2);
        if (t == 0 && g < 4) red2[warp][g] = gq2;
        for (int s = 16; s > 0; s >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, s);
        if (lane == 0) red[warp] = loss;
        __syncthreads();
        if (threadIdx.x < 4) {
            float v = 0.f;
            for (int w = 0; w < NW; ++w) v += red2[w][threadIdx.x];
            o[H * C + 5 * H + threadIdx.x] = v;
        }
        if (threadIdx.x == 0) {
            double v = 0.0;
            for (int w = 0; w < NW; ++w) v += red[w];
            p.dpart[blockIdx.x] = v;
        }
    }
}

// sums of the blocks' partials in a fixed order: 32 entries a block, eight
// warps over the partial blocks, up to four destinations
struct SumSeg {
    int off[4], len[4];
    float* dst[4];
    int n;
};
__global__ void __launch_bounds__(256) k_part_sum(const float* __restrict__ part, int nblk, int E, SumSeg sg) {
    __shared__ float red[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    float v = 0.f;
    if (e < E)
        for (int b = warp; b < nblk; b += 8) v += part[(long long)b * E + e];
    red[warp][lane] = v;
    __syncthreads();
    if (warp == 0 && e < E) {
        v = 0.f;
        for (int w = 0; w < 8; ++w) v += red[w][lane];
        for (int s = 0; s < sg.n; ++s)
            if (e >= sg.off[s] && e < sg.off[s] + sg.len[s]) sg.dst[s][e - sg.off[s]] = v;
    }
}

template <typename F>
void with_modes(int m, F f) {
    switch (modes_pad(m)) {
        case 4: f(std::integral_constant<int, 4>{}); break;
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 12: f(std::integral_constant<int, 12>{}); break;
        default: f(std::integral_constant<int, 16>{}); break;
    }
}

// rows of a block: as many as its shared memory holds, up to what its
// registers allow (640 threads of 96 forward, 512 of 128 backward)
int row_teams(const FnoFusedDims& d, bool bwd) {
    const int most = (bwd ? 512 : 640) / (32 * kTeam);
    const RowSmem L = row_smem(d.nx, chan_pad(d.C), modes_pad(d.m));
    const int w = (kSmemMax / 4 - L.warp) / L.perwarp;
    return w > most ? most : w;
}

cudaError_t row_launch(const FnoFusedDims& d, RowArgs& a, bool bwd, cudaStream_t s) {
    a.nx = d.nx;
    a.C = d.C;
    a.m = d.m;
    a.N = d.N;
    a.rows = (long long)d.nz * d.ny;
    a.vec = d.nx % 4 == 0 ? 1 : 0;  // N is then a multiple of 4 too; the arrays are the library's own
    const int CP = chan_pad(d.C), nw = row_teams(d, bwd);
    const RowSmem L = row_smem(d.nx, CP, modes_pad(d.m));
    const int sm = (L.warp + nw * L.perwarp) * 4;
    long long grid = (a.rows + nw - 1) / nw;
    if (grid > kSMs) grid = kSMs;
    cudaError_t e = cudaSuccess;
    with_modes(d.m, [&](auto M) {
        constexpr int MP = decltype(M)::value;
        const bool shortr = d.nx <= 128;
        auto k = bwd ? (CP == 16 ? (shortr ? k_fno_row_bwd<16, MP, 2> : k_fno_row_bwd<16, MP, kFoldIter>)
                                 : (shortr ? k_fno_row_bwd<32, MP, 2> : k_fno_row_bwd<32, MP, kFoldIter>))
                     : (CP == 16 ? (shortr ? k_fno_row<16, MP, 2> : k_fno_row<16, MP, kFoldIter>)
                                 : (shortr ? k_fno_row<32, MP, 2> : k_fno_row<32, MP, kFoldIter>));
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        if (e == cudaSuccess) k<<<(int)grid, 32 * kTeam * nw, sm, s>>>(a);
    });
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <bool TRAIN>
cudaError_t project_launch(const FnoFusedDims& d, ProjArgs& p, int* blocks, cudaStream_t s) {
    p.C = d.C;
    p.H = d.H;
    p.N = d.N;
    p.sc = 2.0f / (float)(4 * d.N);
    const long long tiles = (d.N + kPts - 1) / kPts;
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto cp, auto nwc, auto full) {
        constexpr int CP = decltype(cp)::value, NW = decltype(nwc)::value;
        constexpr bool FULL = decltype(full)::value;
        constexpr int sm = proj_smem<CP, NW, TRAIN, FULL>();
        auto k = k_fno_project<CP, NW, TRAIN, FULL>;
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        if (e != cudaSuccess) return;
        const int per = 2;  // 93 KB a block at C = 32, H = 128
        const long long grid = tiles < per * kSMs ? tiles : per * kSMs;
        if (blocks) *blocks = (int)grid;
        k<<<(int)grid, 32 * NW, sm, s>>>(p);
    };
    auto go = [&](auto cp, auto nwc) {
        if (proj_full(d.H))
            launch(cp, nwc, std::true_type{});
        else
            launch(cp, nwc, std::false_type{});
    };
    using I16 = std::integral_constant<int, 16>;
    using I32 = std::integral_constant<int, 32>;
    using I4 = std::integral_constant<int, 4>;
    using I8 = std::integral_constant<int, 8>;
    if (chan_pad(d.C) == 16)
        d.H <= 64 ? go(I16{}, I4{}) : go(I16{}, I8{});
    else
        d.H <= 64 ? go(I32{}, I4{}) : go(I32{}, I8{});
    return e == cudaSuccess ? cudaGetLastError() : e;
}

void dft_fwd(const float2* in, float2* out, const float2* tab, int J, int m, int I, int O, cudaStream_t s) {
    with_modes(m, [&](auto M) {
        constexpr int MP = decltype(M)::value;
        size_t sm = (size_t)(J / 2 + 1) * (MP + 2) * sizeof(float2);
        if (sm < dft_sum_bytes<MP>()) sm = dft_sum_bytes<MP>();
        if (sm > 48 * 1024)
            cudaFuncSetAttribute(k_dft_modes<MP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_dft_modes<MP><<<dim3((I + kDftCols - 1) / kDftCols, O), kDftCols * kDftParts, sm, s>>>(in, out, tab, J, m, I);
    });
}
void dft_inv(const float2* in, float2* out, const float2* tab, int J, int m, int I, int O, cudaStream_t s) {
    with_modes(m, [&](auto M) {
        constexpr int MP = decltype(M)::value;
        // parts of the positions: about eight resident blocks an SM
        const long long blocks = (long long)((I + 63) / 64) * O;
        int parts = (int)((8 * kSMs + blocks - 1) / blocks);
        const int half = J / 2 + 1;
        if (parts > (half + 7) / 8) parts = (half + 7) / 8;
        if (parts < 1) parts = 1;
        const size_t sm = (size_t)((half + parts - 1) / parts) * (MP + 2) * sizeof(float2);
        if (sm > 48 * 1024)
            cudaFuncSetAttribute(k_dft_modes_inv<MP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_dft_modes_inv<MP><<<dim3((I + 63) / 64, O, parts), 64, sm, s>>>(in, out, tab, J, m, I);
    });
}

}  // namespace

// The rule: a row of every channel has to fit the shared memory of its two warps
// (C <= 32, rows of 32 to 256 points), a lane group's registers cover the modes
// (m <= 16) and the projection's row tiles the hidden width (H <= 128).  Shorter
// rows leave most lanes of a warp idle; longer ones few rows an SM.
// Nothing bounds the lengths along y and z: their tables fit a block's shared
// memory up to 3227 points at 13 to 16 modes and 9683 at up to 4, and longer
// ones fail at the launch, as in the unfused kernels, whose matrices stay within
// 48 KB (2 m n <= 6144: 236 points at 13 modes).
// With an odd C the spectral weights are not aligned to (re, im) pairs.
bool fno_fused_ok(const FnoFusedDims& d) {
    return d.C <= 32 && d.C % 2 == 0 && d.H <= 128 && d.m <= kMaxModes && d.nx >= 32 && d.nx <= kMaxRow && d.nz <= 65535;
}

size_t fno_fused_xtab_len(const FnoFusedDims& d) { return (size_t)modes_pad(d.m) * half_pad(d.nx); }

void fno_fused_tables(const FnoFusedDims& d, float* xc, float* xs, float* xcw, float* xsw, float2* y, float2* z) {
    const double tp = 6.283185307179586476925286766559;
    const int HP = half_pad(d.nx);
    for (int k = 0; k < modes_pad(d.m); ++k)
        for (int x = 0; x < HP; ++x) {
            const bool in = k < d.m && x <= d.nx / 2;
            const double th = tp * (double)((long long)k * x % d.nx) / d.nx, w = (k == 0 ? 1.0 : 2.0) / (double)d.N;
            const double c = in ? std::cos(th) : 0.0, s = in ? std::sin(th) : 0.0;
            xc[k * HP + x] = (float)c;
            xs[k * HP + x] = (float)s;
            xcw[k * HP + x] = (float)(c * w);
            xsw[k * HP + x] = (float)(s * w);
        }
    auto axis = [&](int n, float2* o) {
        for (int j = 0; j <= n / 2; ++j)
            for (int k = 0; k <= d.m; ++k) {
                const double th = tp * (double)((long long)k * j % n) / n;
                o[j * (d.m + 1) + k] = make_float2((float)std::cos(th), (float)std::sin(th));
            }
    };
    axis(d.ny, y);
    axis(d.nz, z);
}

size_t fno_fused_part_len(const FnoFusedDims& d) {
    const size_t a = (size_t)kSMs * row_part_len(d.C), b = (size_t)2 * kSMs * proj_part_len(d.C, d.H);
    return a > b ? a : b;
}

cudaError_t fno_spectral_fwd(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, float2* A,
                             const __nv_bfloat162* w16, cudaStream_t s) {
    const int I = d.C * d.m, m2 = 2 * d.m;
    dft_fwd(w.T1, w.T2, t.y, d.ny, d.m, I, d.nz, s);
    dft_fwd(w.T2, A, t.z, d.nz, d.m, m2 * I, 1, s);
    const size_t sm = 2 * (size_t)I * sizeof(float2);
    if (d.C % 4 == 0)
        k_mix_modes<true><<<m2 * m2, 256, sm, s>>>(A, w.Ok, w16, d.C, d.m);
    else
        k_mix_modes<false><<<m2 * m2, 256, sm, s>>>(A, w.Ok, w16, d.C, d.m);
    dft_inv(w.Ok, w.T2, t.z, d.nz, d.m, m2 * I, 1, s);
    dft_inv(w.T2, w.T1, t.y, d.ny, d.m, I, d.nz, s);
    return cudaGetLastError();
}

cudaError_t fno_spectral_bwd(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float2* A,
                             const __nv_bfloat162* w16, float2* GW, cudaStream_t s) {
    const int I = d.C * d.m, m2 = 2 * d.m;
    dft_fwd(w.T1, w.T2, t.y, d.ny, d.m, I, d.nz, s);
    dft_fwd(w.T2, w.Gk, t.z, d.nz, d.m, m2 * I, 1, s);
    k_mix_modes_bwd<<<m2 * m2, 256, 3 * (size_t)I * sizeof(float2), s>>>(w.Gk, A, w.Ok, GW, w16, d.C, d.m);
    dft_inv(w.Ok, w.T2, t.z, d.nz, d.m, m2 * I, 1, s);
    dft_inv(w.T2, w.T1, t.y, d.ny, d.m, I, d.nz, s);
    return cudaGetLastError();
}

cudaError_t fno_row_lift(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float* x, const float* P,
                         const float* p, cudaStream_t s) {
    RowArgs a{};
    a.x = x;
    a.P = P;
    a.pb = p;
    a.T1 = w.T1;
    a.fc = t.xc;
    a.fs = t.xs;
    a.nx = d.nx;
    a.C = d.C;
    a.m = d.m;
    a.N = d.N;
    a.rows = (long long)d.nz * d.ny;
    long long grid = (a.rows + 7) / 8;
    if (grid > 4 * kSMs) grid = 4 * kSMs;
    cudaError_t e = cudaSuccess;
    with_modes(d.m, [&](auto M) {
        constexpr int MP = decltype(M)::value;
        const int sm = (2 * MP * half_pad(d.nx) + 160 + 8 * (4 * row_pitch(d.nx) + 8 * MP)) * 4;
        e = cudaFuncSetAttribute(k_fno_lift_modes<MP>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        if (e == cudaSuccess) k_fno_lift_modes<MP><<<(int)grid, 256, sm, s>>>(a);
    });
    return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t fno_row_raw(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float* g, cudaStream_t s) {
    RowArgs a{};
    a.zprev = g;
    a.raw = 1;
    a.T1 = w.T1;
    a.fc = a.ic = t.xcw;
    a.fs = a.is = t.xsw;
    return row_launch(d, a, false, s);
}

cudaError_t fno_row_layer(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, const float* zprev,
                          const float* x, const float* P, const float* p, const float* V, const float* v, float* z,
                          bool last, cudaStream_t s) {
    RowArgs a{};
    a.zprev = zprev;
    a.x = x;
    a.P = P;
    a.pb = p;
    a.V = V;
    a.vb = v;
    a.T1 = w.T1;
    a.z = z;
    a.fc = t.xc;
    a.fs = t.xs;
    a.ic = t.xcw;
    a.is = t.xsw;
    a.dense = 1;
    a.last = last ? 1 : 0;
    return row_launch(d, a, false, s);
}

cudaError_t fno_row_layer_bwd(const FnoFusedDims& d, const FnoTables& t, const FnoWork& w, float* dz,
                              const float* zprev, const float* x, const float* P, const float* p, const float* V,
                              float* gV, float* gv, float* gP, float* gp, cudaStream_t s) {
    RowArgs a{};
    a.zprev = zprev;
    a.x = x;
    a.P = P;
    a.pb = p;
    a.V = V;
    a.T1 = w.T1;
    a.z = dz;
    a.fc = t.xcw;
    a.fs = t.xsw;
    a.ic = t.xc;
    a.is = t.xs;
    a.part = w.part;
    cudaError_t e = row_launch(d, a, true, s);
    if (e != cudaSuccess) return e;
    const int C = d.C, nw = row_teams(d, true);
    const long long nb = (a.rows + nw - 1) / nw;
    SumSeg sg{{0, C * C, C * C + C, C * C + 5 * C}, {C * C, C, 4 * C, C}, {gV, gv, gP, gp}, zprev ? 2 : 4};
    const int E = row_part_len(C);
    k_part_sum<<<(E + 31) / 32, 256, 0, s>>>(w.part, (int)(nb < kSMs ? nb : kSMs), E, sg);
    return cudaGetLastError();
}

cudaError_t fno_project(const FnoFusedDims& d, const float* a, const float* Q1, const float* q1, const float* Q2,
                        const float* q2, float* out, cudaStream_t s) {
    ProjArgs p{};
    p.a = a;
    p.Q1 = Q1;
    p.q1 = q1;
    p.Q2 = Q2;
    p.q2 = q2;
    p.out = out;
    return project_launch<false>(d, p, nullptr, s);
}

cudaError_t fno_project_bwd(const FnoFusedDims& d, const FnoWork& w, const float* a, const float* tgt,
                            const float* Q1, const float* q1, const float* Q2, const float* q2, float* da, float* gQ1,
                            float* gq1, float* gQ2, float* gq2, int* blocks, cudaStream_t s) {
    ProjArgs p{};
    p.a = a;
    p.tgt = tgt;
    p.Q1 = Q1;
    p.q1 = q1;
    p.Q2 = Q2;
    p.q2 = q2;
    p.da = da;
    p.part = w.part;
    p.dpart = w.dpart;
    cudaError_t e = project_launch<true>(d, p, blocks, s);
    if (e != cudaSuccess) return e;
    const int C = d.C, H = d.H, E = proj_part_len(C, H);
    SumSeg sg{{0, H * C, H * C + H, H * C + 5 * H}, {H * C, H, 4 * H, 4}, {gQ1, gq1, gQ2, gq2}, 4};
    k_part_sum<<<(E + 31) / 32, 256, 0, s>>>(w.part, *blocks, E, sg);
    return cudaGetLastError();
}

}  // namespace pf
