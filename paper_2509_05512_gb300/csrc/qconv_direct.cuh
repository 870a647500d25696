// qconv_direct.cuh -- the quaternion convolution and its input gradient with a thread per output
// quaternion, straight from global memory: for layers of few products, where the tiles of
// qgemm_simt.cuh and the block weight and gathered rows of qconv_mma.cuh take longer to set up
// than the products.  Included by qconv_simt.cu and qconv_bwd.cu.
//
// What bounds it: the latency of a thread's chain of loads, then the load instructions (a warp's
// lanes hold different output channels, so a letter is a line per lane).  Measured against those
// kernels: 1x1 layers, fp32, 4 -> 80 channels, 50 images of 78 x 30: 33 and 165 us; bf16, 36 ->
// 244, 4 pixels: 3.7 and 15.8; 3x3 of 64 -> 64, fp32, 8 images of 32 x 32: 97 and 23.
// direct_time is the estimate that decides.
#pragma once
#include <cuda_bf16.h>

#include "internal.h"
#include "qgemm_simt.cuh"

namespace quan {
namespace qd {

// y for one (pixel, output quaternion channel).  Two partial sums per component, by the parity of
// the input channel.
template <typename T, bool SEP>
__global__ void __launch_bounds__(256) fwd_kernel(ConvShape s, const T* __restrict__ x,
                                                  const T* __restrict__ wr,
                                                  const T* __restrict__ wi,
                                                  const T* __restrict__ wj,
                                                  const T* __restrict__ wk, EpilogueArgs ep,
                                                  T* __restrict__ out) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");  // inputs from the previous kernel
    const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= s.M * s.Qout) return;
    const int co = static_cast<int>(idx % s.Qout);
    const long long m = idx / s.Qout;
    const int hw = s.Ho * s.Wo;
    const int n = static_cast<int>(m / hw);
    const int rem = static_cast<int>(m % hw);
    const int ho = rem / s.Wo, wo = rem % s.Wo;
    float4 a[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    for (int dh = 0; dh < s.kh; ++dh) {
        const int h = ho * s.stride - s.pad + dh;
        if (h < 0 || h >= s.H) continue;
        for (int dw = 0; dw < s.kw; ++dw) {
            const int w = wo * s.stride - s.pad + dw;
            if (w < 0 || w >= s.W) continue;
            const T* xp = x + ((static_cast<long long>(n) * s.H + h) * s.W + w) * s.Cin;
            const long long o = ((static_cast<long long>(co) * s.kh + dh) * s.kw + dw) * s.Qin;
            auto letters = [&](int ci) {
                return make_float4(qg::to_f32(__ldg(wr + o + ci)), qg::to_f32(__ldg(wi + o + ci)),
                                   qg::to_f32(__ldg(wj + o + ci)), qg::to_f32(__ldg(wk + o + ci)));
            };
            int ci = 0;
#pragma unroll 1
            for (; ci + 3 < s.Qin; ci += 4) {  // (the loads of four channels before their products)
                float4 q[4], v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    q[i] = letters(ci + i);
                    v[i] = qg::quat(xp + ci + i, s.Qin);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) qg::product<SEP>(a[i & 1], q[i], v[i]);
            }
#pragma unroll 1
            for (; ci < s.Qin; ++ci)
                qg::product<SEP>(a[0], letters(ci), qg::quat(xp + ci, s.Qin));
        }
    }
    const float4 v =
        make_float4(a[0].x + a[1].x, a[0].y + a[1].y, a[0].z + a[1].z, a[0].w + a[1].w);
    float bi[4], sc[4], sh[4];
    qg::vectors(ep, s.Qout, co, bi, sc, sh);
    qg::finish<T, SEP>(s, ep, out, v, bi, sc, sh, m * s.Cout + co);
}

// dx for one (pixel, input quaternion channel), any stride and padding: the sum over taps
// and output channels of conj(W) (x) dy (full form), or of W_p g_p per component p
// (separable form, g = M dy).
template <bool SEP>
__global__ void __launch_bounds__(256) dx_kernel(
    ConvShape s, const __nv_bfloat16* __restrict__ dy, const __nv_bfloat16* __restrict__ wr,
    const __nv_bfloat16* __restrict__ wi, const __nv_bfloat16* __restrict__ wj,
    const __nv_bfloat16* __restrict__ wk, __nv_bfloat16* __restrict__ dx) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= static_cast<long long>(s.N) * s.H * s.W * s.Qin) return;
    const int ci = static_cast<int>(idx % s.Qin);
    const long long pix = idx / s.Qin;
    const int w = static_cast<int>(pix % s.W);
    const int h = static_cast<int>((pix / s.W) % s.H);
    const int n = static_cast<int>(pix / (static_cast<long long>(s.W) * s.H));
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int dh = 0; dh < s.kh; ++dh) {
        const int th = h + s.pad - dh;  // ho * stride
        if (th < 0 || th % s.stride != 0) continue;
        const int ho = th / s.stride;
        if (ho >= s.Ho) continue;
        for (int dw = 0; dw < s.kw; ++dw) {
            const int tw = w + s.pad - dw;
            if (tw < 0 || tw % s.stride != 0) continue;
            const int wo = tw / s.stride;
            if (wo >= s.Wo) continue;
            const __nv_bfloat16* g =
                dy + ((static_cast<long long>(n) * s.Ho + ho) * s.Wo + wo) * s.Cout;
#pragma unroll 2
            for (int co = 0; co < s.Qout; ++co) {
                const long long o =
                    ((static_cast<long long>(co) * s.kh + dh) * s.kw + dw) * s.Qin + ci;
                const float4 q = make_float4(qg::to_f32(__ldg(wr + o)), qg::to_f32(__ldg(wi + o)),
                                             qg::to_f32(__ldg(wj + o)), qg::to_f32(__ldg(wk + o)));
                const float4 d = qg::quat(g + co, s.Qout);
                qg::product<SEP>(a, SEP ? q : qg::conj(q), SEP ? qg::mix_eq9(d) : d);
            }
        }
    }
    qg::store4(dx + pix * s.Cin + ci, s.Qin, a);
}

// Estimated time (us) of these kernels on num_sms SMs: Q channels (quaternions, consecutive
// threads) of px pixels in rows of `row`, Qs channels per tap.  A thread runs the taps that one
// pixel reads; lanes that hold several pixels run the taps of any of them.  Coefficients fitted
// to 1,850 layers of random sizes (80% of them between 0.8 and 1.35 of it).
struct Cost {
    double fixed, step, tap, load, warp;
};
constexpr Cost FWD_F32 = {3.2, 0.13, 0.056, 0.26, 1.7};
constexpr Cost FWD_BF16 = {3.3, 0.091, 0.091, 0.25, 1.4};
constexpr Cost DX = {2.9, 0.15, 0.20, 0.39, 4.4};

inline double time(const Cost& c, int Q, int Qs, long long px, int row, int taps, int one_h,
                   int any_h, int one_w, int any_w, double line, int num_sms) {
    const double h = static_cast<double>(Q) * row >= 32 ? one_h : any_h;
    const double w = Q % 32 == 0 ? one_w : any_w;
    const double warps = px * static_cast<double>(Q) / 32 / num_sms;  // per SM
    const double wsm = warps < 1 ? 1 : warps, occ = wsm < 64 ? 1 : wsm / 64;
    const double steps = Qs * h * w;
    const double lines = 4 * (Q < 32 ? Q : 32) * line < 4 ? 4 : 4 * (Q < 32 ? Q : 32) * line;
    const double loads = lines + 4 * (Q < 32 ? 32.0 / Q : 1.0) + 12;
    return c.fixed + steps * occ * c.step + taps * occ * c.tap +
           wsm * steps * loads / 1900 * c.load + wsm / 64 * c.warp;
}

inline int least(long long a, long long b) { return static_cast<int>(a < b ? a : b); }

// Forward: a letter is a line per channel of the warp, an input component a line per pixel; where
// the channels' rows (the pixels, for few channels) are a multiple of 64 or 128 bytes apart those
// lines evict one another (1.4 and 2.5 times the steps' estimate).
inline double fwd_time(const ConvShape& s, bool f32, int num_sms) {
    Cost c = f32 ? FWD_F32 : FWD_BF16;
    const long long pitch = static_cast<long long>(s.kh) * s.kw * s.Qin * (f32 ? 4 : 2);
    const bool pixels =
        s.Qout < 16 && static_cast<long long>(s.stride) * s.Cin * (f32 ? 4 : 2) % 128 == 0;
    const double evict = pixels || pitch % 128 == 0 ? 2.5 : pitch % 64 == 0 ? 1.4 : 1.0;
    c.step *= evict;
    c.load *= evict;
    return time(c, s.Qout, s.Qin, s.M, s.Wo, s.kh * s.kw, least(s.kh, s.H),
                least(s.kh, s.H + (s.Ho - 1LL) * s.stride), least(s.kw, s.W),
                least(s.kw, s.W + (s.Wo - 1LL) * s.stride), 1.0, num_sms);
}

// Input gradient: the channels of a letter are consecutive.
inline double dx_time(const ConvShape& s, int num_sms) {
    return time(DX, s.Qin, s.Qout, static_cast<long long>(s.N) * s.H * s.W, s.W, s.kh * s.kw,
                least((s.kh + s.stride - 1) / s.stride, s.Ho),
                least(s.kh, (s.Ho - 1LL) * s.stride + s.H),
                least((s.kw + s.stride - 1) / s.stride, s.Wo),
                least(s.kw, (s.Wo - 1LL) * s.stride + s.W), 2.0 / 128, num_sms);
}

template <typename K, typename... Args>
cudaError_t launch(K kern, long long outs, cudaStream_t stream, Args... args) {
    const long long blocks = (outs + 255) / 256;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    return launch_pdl(kern, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, stream, args...);
}

}  // namespace qd
}  // namespace quan
