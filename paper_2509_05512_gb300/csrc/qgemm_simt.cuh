// qgemm_simt.cuh -- tiled quaternion products on CUDA cores (fp32 FFMA): the convolution, its
// input gradient and its weight gradient for every shape the tensor-core kernels do not take
// (fp32 tensors, quaternion channel counts that are not multiples of 16, unaligned pointers).
//
// bf16 layers come here only where qconv_mma.cuh does not take them (unaligned tensors, very
// wide filters), layers of few products go to qconv_direct.cuh.  All three are the contraction
// out[i][j] = sum over k of A[i][k] (x) B[k][j]  of quaternions (Hamilton product of Eq. 3, 16
// FFMAs), or componentwise products for the separable form:
//   FWD    i = output channel, j = output pixel, k = (tap, input channel):
//          A = W, B = x  (Eq. 5; separable: the products c_p, mixed by Eq. 7 at the end)
//   DGRAD  i = input channel, j = input pixel, k = (tap, output channel):
//          A = conj(W), B = dy (separable: A = W, B = dy mixed by Eq. 9); the pixels of one
//          block share their row and column modulo the stride, so only the taps that reach
//          them are summed
//   WGRAD  i = output channel, j = (tap, input channel), k = output pixel:
//          A = dy, B = conj(x) (separable: A = dy mixed by Eq. 9, B = x); the pixels are split
//          over blockIdx.y and the partial sums added with atomics to zeroed outputs
//
// A block computes ITILE x JTILE quaternions from slices of 32 k's staged in shared memory as
// float4 quaternions, [k][i] and [k][j]; four groups of 128 threads take 8 k's of a slice each,
// TI x TJ quaternions per thread, and add up at the end (one group alone left a scheduler
// with 1.7 warps to issue from).  The next slice's global loads are
// in flight during the products.  ITILE = NI TI follows the channel count (10 channels: 5
// threads of 2), so little of a tile is padding.
// What bounds it: FFMA issue (TI = 2, TJ = 4: 6 LDS.128 per 128 FFMA).  A thread per output
// quaternion straight from global memory is bound by load instructions: 97 us for the fp32 layer
// of 8 images of 32 x 32, 64 -> 64 channels, 3x3, against 23 us.
#pragma once
#include <cuda_bf16.h>

#include "internal.h"

namespace quan {
namespace qg {

constexpr int GROUP = 128;  // threads of one k group
constexpr int KG = 4;       // k groups
constexpr int THREADS = GROUP * KG;
constexpr int KS = 8;       // k's of a slice per group
constexpr int KC = KS * KG;
constexpr int MAX_I = 16;   // ITILE: one pass of the loaders
constexpr int MAX_J = 64;   // JTILE
constexpr int PASSES = KC * MAX_J / THREADS;
enum Op { FWD = 0, DGRAD = 1, WGRAD = 2 };

struct Params {
    ConvShape s;
    const void* a[4];   // FWD, DGRAD: the letters; WGRAD: a[0] = dy
    const void* b;      // FWD, WGRAD: x; DGRAD: dy
    EpilogueArgs ep;    // FWD
    void* out;          // FWD: y, DGRAD: dx
    float* dw[4];       // WGRAD
    int I, ni, nj;      // rows; threads along i and j
    int itiles;
    int tj;             // j's per thread
    int ip, jp;         // powers of two >= ITILE, JTILE (loader strides)
    long long chunk;    // WGRAD: pixels per blockIdx.y
    long long jt;       // j tiles (DGRAD: of the largest class)
    int cw;             // DGRAD: classes along the columns
};

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void store(float* p, float v) { *p = v; }
__device__ __forceinline__ void store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

__device__ __forceinline__ float activate(float z, int act) {
    if (act == 1) return fmaxf(z, 0.0f);
    if (act == 2) return z / (1.0f + __expf(-z));
    return z;
}

// Four components of one quaternion, `step` elements apart.
template <typename T>
__device__ __forceinline__ float4 quat(const T* p, int step) {
    return make_float4(to_f32(__ldg(p)), to_f32(__ldg(p + step)), to_f32(__ldg(p + 2 * step)),
                       to_f32(__ldg(p + 3 * step)));
}
template <typename T>
__device__ __forceinline__ float4 letters(const Params& p, long long o) {
    return make_float4(to_f32(__ldg(static_cast<const T*>(p.a[0]) + o)),
                       to_f32(__ldg(static_cast<const T*>(p.a[1]) + o)),
                       to_f32(__ldg(static_cast<const T*>(p.a[2]) + o)),
                       to_f32(__ldg(static_cast<const T*>(p.a[3]) + o)));
}
__device__ __forceinline__ float4 conj(float4 q) { return make_float4(q.x, -q.y, -q.z, -q.w); }

// g = M dy, M of Eq. 9 (rows p, columns m):
//   [ 1  1  1  1 ]
//   [-1  1 -1  1 ]
//   [-1  1  1 -1 ]
//   [-1 -1  1  1 ]
__device__ __forceinline__ float4 mix_eq9(float4 d) {
    return make_float4(d.x + d.y + d.z + d.w, -d.x + d.y - d.z + d.w, -d.x + d.y + d.z - d.w,
                       -d.x - d.y + d.z + d.w);
}

template <bool SEP>
__device__ __forceinline__ void product(float4& c, const float4& a, const float4& b) {
    if constexpr (SEP) {
        c.x = fmaf(a.x, b.x, c.x);
        c.y = fmaf(a.y, b.y, c.y);
        c.z = fmaf(a.z, b.z, c.z);
        c.w = fmaf(a.w, b.w, c.w);
    } else {
        c.x = fmaf(a.x, b.x, c.x); c.x = fmaf(-a.y, b.y, c.x);
        c.x = fmaf(-a.z, b.z, c.x); c.x = fmaf(-a.w, b.w, c.x);
        c.y = fmaf(a.x, b.y, c.y); c.y = fmaf(a.y, b.x, c.y);
        c.y = fmaf(a.z, b.w, c.y); c.y = fmaf(-a.w, b.z, c.y);
        c.z = fmaf(a.x, b.z, c.z); c.z = fmaf(-a.y, b.w, c.z);
        c.z = fmaf(a.z, b.x, c.z); c.z = fmaf(a.w, b.y, c.z);
        c.w = fmaf(a.x, b.w, c.w); c.w = fmaf(a.y, b.z, c.w);
        c.w = fmaf(-a.z, b.y, c.w); c.w = fmaf(a.w, b.x, c.w);
    }
}

__device__ __forceinline__ bool not_finite(const float4& v) {
    // (NaN when one of them is not finite)
    return fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, v.w * 0.f))) != 0.f;
}

// One output quaternion from the taps inside the image (WGRAD: the pixels whose tap is) only:
// the tiles multiply the zeros that stand for the padding as well, which makes NaN of an
// infinite or NaN factor.  False where nothing is outside: the tile's sum stands.
// FWD: channel i, output pixel (n, h, w) by the input pixel of its first tap; DGRAD: channel i,
// dx pixel (n, h, w); WGRAD: channel i, input channel n, tap (h, w), pixels k0 .. k1 - 1.
template <typename T, int OP, bool SEP>
__device__ __forceinline__ bool sum_inside(const Params& p, int i, int n, int h, int w,
                                           long long k0, long long k1, float4& acc) {
    const ConvShape& s = p.s;
    const T* b = static_cast<const T*>(p.b);
    acc = make_float4(0.f, 0.f, 0.f, 0.f);
    bool outside = false;
    if constexpr (OP == WGRAD) {
        const T* dy = static_cast<const T*>(p.a[0]);
#pragma unroll 1
        for (long long k = k0; k < k1; ++k) {
            const long long r = k / s.Wo, img = r / s.Ho;
            const int y = static_cast<int>(r - img * s.Ho) * s.stride - s.pad + h;
            const int x = static_cast<int>(k - r * s.Wo) * s.stride - s.pad + w;
            if (y < 0 || y >= s.H || x < 0 || x >= s.W) {
                outside = true;
                continue;
            }
            const float4 g = quat(dy + k * s.Cout + i, s.Qout);
            const float4 q = quat(b + ((img * s.H + y) * s.W + x) * s.Cin + n, s.Qin);
            product<SEP>(acc, SEP ? mix_eq9(g) : g, SEP ? q : conj(q));
        }
    } else {
        const int C = OP == FWD ? s.Qin : s.Qout;
        const int hs = OP == FWD ? s.H : s.Ho, ws = OP == FWD ? s.W : s.Wo;
#pragma unroll 1
        for (int t = 0; t < s.kh * s.kw; ++t) {
            const int dh = t / s.kw, dw = t - dh * s.kw;
            int y = h + dh, x = w + dw;
            if constexpr (OP == DGRAD) {  // the output pixel this tap reads for dx (h, w)
                y = h + s.pad - dh;
                x = w + s.pad - dw;
                if (y % s.stride != 0 || x % s.stride != 0) continue;
                y /= s.stride;
                x /= s.stride;
            }
            if (y < 0 || y >= hs || x < 0 || x >= ws) {
                outside = true;
                continue;
            }
            const T* px = b + ((static_cast<long long>(n) * hs + y) * ws + x) * (4LL * C);
#pragma unroll 1
            for (int c = 0; c < C; ++c) {
                const long long row = OP == FWD ? i : c, col = OP == FWD ? c : i;
                const float4 q = letters<T>(p, (row * s.kh * s.kw + t) * s.Qin + col);
                const float4 g = quat(px + c, C);
                product<SEP>(acc, OP == DGRAD && !SEP ? conj(q) : q,
                             OP == DGRAD && SEP ? mix_eq9(g) : g);
            }
        }
    }
    return outside;
}

// The epilogue's vectors for output quaternion channel i.
__device__ __forceinline__ void vectors(const EpilogueArgs& ep, int Qout, int i, float (&bi)[4],
                                        float (&sc)[4], float (&sh)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = q * Qout + i;
        bi[q] = ep.bias ? __ldg(ep.bias + c) : 0.f;
        sc[q] = ep.scale ? __ldg(ep.scale + c) : 1.f;
        sh[q] = ep.scale ? __ldg(ep.shift + c) : 0.f;
    }
}

// One output quaternion of FWD at offset o (component q at o + q Qout): Eq. 7's mix of the
// separable form, then act(scale (y + bias) + shift + residual).
template <typename T, bool SEP>
__device__ __forceinline__ void finish(const ConvShape& s, const EpilogueArgs& ep, T* out,
                                       const float4& v, const float (&bi)[4],
                                       const float (&sc)[4], const float (&sh)[4], long long o) {
    const T* res = static_cast<const T*>(ep.residual);
    float z[4] = {v.x, v.y, v.z, v.w};
    if constexpr (SEP) {
        z[0] = v.x - v.y - v.z - v.w;
        z[1] = v.x + v.y + v.z - v.w;
        z[2] = v.x - v.y + v.z + v.w;
        z[3] = v.x + v.y - v.z + v.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float y = z[q] + bi[q];
        if (ep.scale) y = fmaf(sc[q], y, sh[q]);
        if (res) y += to_f32(res[o + q * s.Qout]);
        store(out + o + q * s.Qout, activate(y, s.act));
    }
}

template <typename T>
__device__ __forceinline__ void store4(T* o, int step, const float4& v) {
    store(o, v.x);
    store(o + step, v.y);
    store(o + 2 * step, v.z);
    store(o + 3 * step, v.w);
}

__device__ __forceinline__ void add4(float* const (&dw)[4], long long o, const float4& v) {
    atomicAdd(dw[0] + o, v.x);
    atomicAdd(dw[1] + o, v.y);
    atomicAdd(dw[2] + o, v.z);
    atomicAdd(dw[3] + o, v.w);
}

template <typename T, int OP, bool SEP, int TI, int TJ>
__global__ void __launch_bounds__(THREADS, 1) qgemm_kernel(const __grid_constant__ Params p) {
    __shared__ float4 sa[KC][MAX_I + 1];
    __shared__ float4 sb[KC][MAX_J + 1];
    __shared__ int4 tab[MAX_J];  // the tile's pixels: image, first row and column, valid
    const ConvShape& s = p.s;
    const int tid = threadIdx.x;
    const int itile = p.ni * TI, jtile = p.nj * TJ;
    const unsigned jtc = blockIdx.x / static_cast<unsigned>(p.itiles);
    const int i0 = static_cast<int>(blockIdx.x - jtc * p.itiles) * itile;
    const int cls = OP == DGRAD ? static_cast<int>(jtc / p.jt) : 0;
    const long long j0 = (jtc - cls * p.jt) * jtile;
    const int taps = s.kh * s.kw;

    // DGRAD: the pixel class (a, b), its grid and its taps
    int Hc = s.Ho, Wc = s.Wo, eh = 0, ew = 0, th = s.kh, tw = s.kw, ca = 0, cb = 0;
    long long J;
    int K;
    long long kbeg = 0;
    if constexpr (OP == DGRAD) {
        ca = cls / p.cw;
        cb = cls - ca * p.cw;
        Hc = (s.H - ca + s.stride - 1) / s.stride;
        Wc = (s.W - cb + s.stride - 1) / s.stride;
        eh = (ca + s.pad) % s.stride;
        ew = (cb + s.pad) % s.stride;
        th = eh < s.kh ? (s.kh - eh + s.stride - 1) / s.stride : 0;
        tw = ew < s.kw ? (s.kw - ew + s.stride - 1) / s.stride : 0;
        J = static_cast<long long>(s.N) * Hc * Wc;
        K = th * tw * s.Qout;
    } else if constexpr (OP == FWD) {
        J = s.M;
        K = taps * s.Qin;
    } else {
        J = static_cast<long long>(taps) * s.Qin;
        kbeg = blockIdx.y * p.chunk;
        const long long left = s.M - kbeg;
        K = static_cast<int>(left < p.chunk ? left : p.chunk);
    }
    if (j0 >= J) return;  // (a class with fewer pixels than the largest)
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if constexpr (OP != WGRAD) {
        for (int j = tid; j < jtile; j += THREADS) {
            const long long m = j0 + j;
            int4 t = make_int4(0, 0, 0, 0);
            if (m < J) {
                const long long r = m / Wc;
                const int c = static_cast<int>(m - r * Wc);
                const int n = static_cast<int>(r / Hc);
                const int h = static_cast<int>(r - static_cast<long long>(n) * Hc);
                if constexpr (OP == FWD)
                    t = make_int4(n, h * s.stride - s.pad, c * s.stride - s.pad, 1);
                else  // output row of the class's first tap
                    t = make_int4(n, h + (ca + s.pad - eh) / s.stride,
                                  c + (cb + s.pad - ew) / s.stride, 1);
            }
            tab[j] = t;
        }
        __syncthreads();
    }

    // loader coordinates.  k fastest (a slice of 8 contiguous channels per row): FWD's A,
    // FWD's and DGRAD's B; rows fastest (contiguous channels along i or j): the others
    const int kk = tid & (KC - 1), row = tid / KC;
    const int ai = OP == FWD ? row : (tid & (p.ip - 1)), ak = OP == FWD ? kk : tid / p.ip;
    const bool a_on = ai < itile && ak < KC && i0 + ai < p.I;
    // WGRAD's B: this thread's (tap, input channel)
    const int bj = tid & (p.jp - 1), bk = tid / p.jp, bstep = THREADS / p.jp;
    int b_dh = 0, b_dw = 0, b_ci = 0;
    bool b_on = false;
    int3 px0 = make_int3(0, 0, 0);  // the chunk's first pixel: image, row, column
    if constexpr (OP == WGRAD) {
        const long long r = kbeg / s.Wo;
        px0.x = static_cast<int>(r / s.Ho);
        px0.y = static_cast<int>(r - static_cast<long long>(px0.x) * s.Ho);
        px0.z = static_cast<int>(kbeg - r * s.Wo);
        const long long j = j0 + bj;
        b_on = bj < jtile && j < J;
        if (b_on) {
            const int tap = static_cast<int>(j / s.Qin);
            b_ci = static_cast<int>(j - static_cast<long long>(tap) * s.Qin);
            b_dh = tap / s.kw;
            b_dw = tap - b_dh * s.kw;
        }
    }
    const int passes = OP == WGRAD ? KC / bstep : (jtile + THREADS / KC - 1) / (THREADS / KC);
    const T* bp = static_cast<const T*>(p.b);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);

    float4 ra, rb[PASSES];
    auto load = [&](int k0) {
        ra = zero;
        if (a_on && k0 + ak < K) {
            const int k = k0 + ak;
            if constexpr (OP == FWD) {
                ra = letters<T>(p, static_cast<long long>(i0 + ai) * K + k);
            } else if constexpr (OP == DGRAD) {
                const int t = k / s.Qout, co = k - t * s.Qout;
                const int u = t / tw, v = t - u * tw;
                const long long o =
                    ((static_cast<long long>(co) * s.kh + eh + u * s.stride) * s.kw + ew +
                     v * s.stride) * s.Qin + i0 + ai;
                const float4 q = letters<T>(p, o);
                ra = SEP ? q : conj(q);
            } else {
                const float4 q = quat(static_cast<const T*>(p.a[0]) + (kbeg + k) * s.Cout + i0 + ai,
                                      s.Qout);
                ra = SEP ? mix_eq9(q) : q;
            }
        }
        if constexpr (OP == WGRAD) {
#pragma unroll
            for (int q = 0; q < PASSES; ++q) {
                const int k = k0 + bk + q * bstep;
                rb[q] = zero;
                if (q < passes && b_on && k < K) {
                    const int rr = (px0.z + k) / s.Wo, c = px0.z + k - rr * s.Wo;
                    const int dn = (px0.y + rr) / s.Ho, ho = px0.y + rr - dn * s.Ho;
                    const int n = px0.x + dn;
                    const int h = ho * s.stride - s.pad + b_dh, w = c * s.stride - s.pad + b_dw;
                    if (h >= 0 && h < s.H && w >= 0 && w < s.W) {
                        const float4 x = quat(
                            bp + ((static_cast<long long>(n) * s.H + h) * s.W + w) * s.Cin + b_ci,
                            s.Qin);
                        rb[q] = SEP ? x : conj(x);
                    }
                }
            }
        } else {
            // this thread's k, the same for every row
            const int k = k0 + kk;
            const int C = OP == FWD ? s.Qin : s.Qout, KW = OP == FWD ? s.kw : tw;
            const int t = k < K ? k / C : 0, c = k - t * C;
            const int dh = KW > 0 ? t / KW : 0, dw = t - dh * KW;
#pragma unroll
            for (int q = 0; q < PASSES; ++q) {
                if (q >= passes) break;
                const int j = row + q * (THREADS / KC);
                rb[q] = zero;
                if (j < jtile && k < K) {
                    const int4 px = tab[j];
                    if constexpr (OP == FWD) {
                        const int h = px.y + dh, w = px.z + dw;
                        if (px.w && h >= 0 && h < s.H && w >= 0 && w < s.W)
                            rb[q] = quat(
                                bp + ((static_cast<long long>(px.x) * s.H + h) * s.W + w) * s.Cin +
                                    c, s.Qin);
                    } else {
                        const int ho = px.y - dh, wo = px.z - dw;
                        if (px.w && ho >= 0 && ho < s.Ho && wo >= 0 && wo < s.Wo) {
                            const float4 g = quat(
                                bp + ((static_cast<long long>(px.x) * s.Ho + ho) * s.Wo + wo) *
                                         s.Cout + c, s.Qout);
                            rb[q] = SEP ? mix_eq9(g) : g;
                        }
                    }
                }
            }
        }
    };
    auto put = [&] {
        if (ai < itile && ak < KC) sa[ak][ai] = ra;
#pragma unroll
        for (int q = 0; q < PASSES; ++q) {
            if constexpr (OP == WGRAD) {
                if (q < passes && bj < jtile) sb[bk + q * bstep][bj] = rb[q];
            } else {
                const int j = row + q * (THREADS / KC);
                if (q < passes && j < jtile) sb[kk][j] = rb[q];
            }
        }
    };

    // thread (ti, tj) owns rows ti + r ni and columns tj + c nj
    const int grp = tid / GROUP, lt = tid % GROUP;
    const int ti = lt % p.ni, tj = lt / p.ni;
    const bool active = tj < p.nj;
    float4 acc[TI][TJ];
#pragma unroll
    for (int r = 0; r < TI; ++r)
#pragma unroll
        for (int c = 0; c < TJ; ++c) acc[r][c] = zero;

    if (K > 0) load(0);
    for (int k0 = 0; k0 < K; k0 += KC) {
        put();
        __syncthreads();
        if (k0 + KC < K) load(k0 + KC);
        if (active) {
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                float4 av[TI], bv[TJ];
#pragma unroll
                for (int r = 0; r < TI; ++r) av[r] = sa[grp * KS + k][ti + r * p.ni];
#pragma unroll
                for (int c = 0; c < TJ; ++c) bv[c] = sb[grp * KS + k][tj + c * p.nj];
#pragma unroll
                for (int r = 0; r < TI; ++r)
#pragma unroll
                    for (int c = 0; c < TJ; ++c) product<SEP>(acc[r][c], av[r], bv[c]);
            }
        }
        __syncthreads();
    }
    // The next kernel may start now.  (Triggered at the beginning, its blocks are placed while
    // this one's hold their SMs, several on some and none on others: the layer above took
    // 49 us among its like and 28 us alone.)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // groups 2 and 3 to 0 and 1, then 1 to 0 (through the tile's memory)
    float4* part = &sb[0][0];
    static_assert(2 * GROUP * TI * TJ <= KC * (MAX_J + 1), "partial sums fit");
#pragma unroll
    for (int half = KG / 2; half >= 1; half /= 2) {
        if (active && grp >= half && grp < 2 * half) {
#pragma unroll
            for (int e = 0; e < TI * TJ; ++e)
                part[((grp - half) * TI * TJ + e) * GROUP + lt] = acc[e / TJ][e % TJ];
        }
        __syncthreads();
        if (active && grp < half) {
#pragma unroll
            for (int e = 0; e < TI * TJ; ++e) {
                const float4 v = part[(grp * TI * TJ + e) * GROUP + lt];
                float4& a = acc[e / TJ][e % TJ];
                a.x += v.x;
                a.y += v.y;
                a.z += v.z;
                a.w += v.w;
            }
        }
        __syncthreads();
    }
    if (!active || grp != 0) return;

    float bi[4], sc[4], sh[4];  // FWD: the epilogue's vectors
    // DGRAD: dx pixel (n, h, w) of the class's pixel m
    auto dx_pixel = [&](long long m, long long& n, int& h, int& w) {
        const long long rr = m / Wc;
        w = static_cast<int>(m - rr * Wc) * s.stride + cb;
        n = rr / Hc;
        h = static_cast<int>(rr - n * Hc) * s.stride + ca;
    };
    T* out = static_cast<T*>(p.out);
    unsigned odd = 0;  // the quaternions that are not finite
#pragma unroll
    for (int r = 0; r < TI; ++r) {
        const int i = i0 + ti + r * p.ni;
        if (i >= p.I) continue;
        if constexpr (OP == FWD) vectors(p.ep, s.Qout, i, bi, sc, sh);
#pragma unroll
        for (int c = 0; c < TJ; ++c) {
            const long long m = j0 + tj + c * p.nj;
            if (m >= J) continue;
            const float4& v = acc[r][c];
            const bool bad = not_finite(v);
            if (bad) odd |= 1u << (r * TJ + c);
            if constexpr (OP == FWD) {
                finish<T, SEP>(s, p.ep, out, v, bi, sc, sh, m * s.Cout + i);
            } else if constexpr (OP == DGRAD) {
                long long n;
                int h, w;
                dx_pixel(m, n, h, w);
                store4(out + ((n * s.H + h) * s.W + w) * s.Cin + i, s.Qin, v);
            } else if (!bad) {
                add4(p.dw, static_cast<long long>(i) * J + m, v);
            }
        }
    }
    // rare: those once more without the padding
#pragma unroll 1
    for (; odd != 0; odd &= odd - 1) {
        const int e = __ffs(odd) - 1;
        const int i = i0 + ti + e / TJ * p.ni, jl = tj + e % TJ * p.nj;
        const long long m = j0 + jl;
        float4 v;
        if constexpr (OP == FWD) {
            const int4 px = tab[jl];
            if (!sum_inside<T, OP, SEP>(p, i, px.x, px.y, px.z, 0, 0, v)) continue;
            vectors(p.ep, s.Qout, i, bi, sc, sh);
            finish<T, SEP>(s, p.ep, out, v, bi, sc, sh, m * s.Cout + i);
        } else if constexpr (OP == DGRAD) {
            long long n;
            int h, w;
            dx_pixel(m, n, h, w);
            if (!sum_inside<T, OP, SEP>(p, i, static_cast<int>(n), h, w, 0, 0, v)) continue;
            store4(out + ((n * s.H + h) * s.W + w) * s.Cin + i, s.Qin, v);
        } else {
            const int tap = static_cast<int>(m / s.Qin), dh = tap / s.kw;
            const int ci = static_cast<int>(m - static_cast<long long>(tap) * s.Qin);
            sum_inside<T, OP, SEP>(p, i, ci, dh, tap - dh * s.kw, kbeg, kbeg + K, v);
            add4(p.dw, static_cast<long long>(i) * J + m, v);
        }
    }
}

// Thread grid of an I x J product: the fewest i tiles of at most 16 rows, TI rows per thread,
// and as many columns as a group's threads reach.
inline void layout(Params* p, int I, long long J, int ti, int tj) {
    const int per = MAX_I / ti;                       // threads along i at most
    const int rows = (I + ti - 1) / ti;               // thread rows needed
    p->I = I;
    p->itiles = (rows + per - 1) / per;
    p->ni = (rows + p->itiles - 1) / p->itiles;
    p->itiles = (rows + p->ni - 1) / p->ni;
    p->tj = tj;
    int nj = GROUP / p->ni;
    if (nj * tj > MAX_J) nj = MAX_J / tj;
    // no wider than J, and equal tiles
    const long long cols = (J + tj - 1) / tj;
    if (nj > cols) nj = static_cast<int>(cols);
    const long long jt = (cols + nj - 1) / nj;
    nj = static_cast<int>((cols + jt - 1) / jt);
    p->nj = nj;
    p->ip = 1;
    while (p->ip < p->ni * ti) p->ip <<= 1;
    p->jp = 16;
    while (p->jp < nj * tj) p->jp <<= 1;
}

inline long long jtiles(const Params& p, long long J) {
    const long long w = static_cast<long long>(p.nj) * p.tj;
    return (J + w - 1) / w;
}

constexpr int TILES[3][2] = {{2, 4}, {2, 2}, {1, 1}};

// The thread tile: 2 x 4 or 2 x 2 where that still gives four SMs of five a block, else (small
// problems, where the chain of products of one thread is the time) 1 x 1.
// outer: WGRAD's pixel chunks, DGRAD's pixel classes.  The index of TILES.
inline int pick(Params* p, int I, long long J, long long outer, int num_sms) {
    for (int v = 0;; ++v) {
        layout(p, I, J, TILES[v][0], TILES[v][1]);
        if (v == 2 || jtiles(*p, J) * p->itiles * outer * 5 >= 4LL * num_sms) return v;
    }
}

// Estimated time (us) of FWD: the waves of blocks, each a start and its slices of 32 products.
// (Fitted to 545 fp32 layers of random sizes: 80% between 0.9 and 1.1 of it.)
inline double fwd_time(const ConvShape& s, int num_sms) {
    Params p = {};
    const int v = pick(&p, s.Qout, s.M, 1, num_sms);
    const double blocks = static_cast<double>(jtiles(p, s.M)) * p.itiles / num_sms;
    const double waves = blocks < 1 ? 1 : blocks < 4 ? static_cast<int>(blocks + 0.999) : blocks;
    const double slices = (static_cast<double>(s.kh) * s.kw * s.Qin + KC - 1) / KC;
    return 1.8 + waves * (static_cast<long long>(slices) * (v == 0 ? 3.7 : v == 1 ? 2.1 : 1.1) +
                          (v == 0 ? 3.7 : v == 1 ? 2.5 : 1.5));
}

template <typename T, int OP, bool SEP>
cudaError_t launch(Params p, int I, long long J, long long outer, int num_sms,
                   cudaStream_t stream) {
    const int v = pick(&p, I, J, outer, num_sms);
    p.jt = jtiles(p, J);
    const long long blocks = p.jt * p.itiles * (OP == DGRAD ? outer : 1);
    const long long chunks = OP == DGRAD ? 1 : outer;
    if (blocks > 0x7fffffffLL || chunks > 65535) return cudaErrorInvalidConfiguration;
    const dim3 grid(static_cast<unsigned>(blocks), static_cast<unsigned>(chunks));
    auto k24 = qgemm_kernel<T, OP, SEP, 2, 4>;
    auto k22 = qgemm_kernel<T, OP, SEP, 2, 2>;
    auto k11 = qgemm_kernel<T, OP, SEP, 1, 1>;
    return launch_pdl(v == 0 ? k24 : v == 1 ? k22 : k11, grid, dim3(THREADS), 0, stream, p);
}

}  // namespace qg
}  // namespace quan
