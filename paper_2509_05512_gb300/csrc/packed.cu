// packed.cu -- the Python binding's way into the C ABI: the integer and pointer arguments of a
// hot entry point packed as 64-bit words.  A ctypes call converts every argument by itself,
// about 6 us for the 20 of a convolution; packing them with one struct.pack and passing one
// pointer takes about 2.  Not part of the public header.
#include <cstring>

#include "quan.h"

namespace {

struct Args {
    const long long* a;
    int i = 0;
    long long next() {
        long long v;
        memcpy(&v, a + i++, sizeof(v));
        return v;
    }
    void* ptr() { return reinterpret_cast<void*>(next()); }
    float* f32() { return static_cast<float*>(ptr()); }
    quan_stream_t stream() { return static_cast<quan_stream_t>(ptr()); }
    int num() { return static_cast<int>(next()); }
    float real() {
        double d;
        memcpy(&d, a + i++, sizeof(d));
        return static_cast<float>(d);
    }
};

// The arguments every convolution call starts with, in order.
struct Conv {
    void *x, *w[4];
    float *bias, *scale, *shift;
    int v[11];  // N, H, W, Cin, Cout, kh, kw, stride, pad, act (Cin absent for RGB)
    Conv(Args& g, int ints) {
        x = g.ptr();
        for (auto& p : w) p = g.ptr();
        bias = g.f32();
        scale = g.f32();
        shift = g.f32();
        for (int i = 0; i < ints; ++i) v[i] = g.num();
    }
};

#define QUAN_CONV_ARGS                                                                      \
    c.x, c.w[0], c.w[1], c.w[2], c.w[3], c.bias, c.scale, c.shift, c.v[0], c.v[1], c.v[2],  \
        c.v[3], c.v[4], c.v[5], c.v[6], c.v[7], c.v[8], c.v[9]

}  // namespace

extern "C" int quan_packed_call(int op, const long long* words) {
    Args g{words};
    switch (op) {
        case 0: {
            Conv c(g, 10);
            void* out = g.ptr();
            return quan_qconv2d_fwd(QUAN_CONV_ARGS, out, g.stream());
        }
        case 1: {
            Conv c(g, 10);
            float* out = g.f32();
            return quan_qconv2d_fwd_f32(
                static_cast<float*>(c.x), static_cast<float*>(c.w[0]), static_cast<float*>(c.w[1]),
                static_cast<float*>(c.w[2]), static_cast<float*>(c.w[3]), c.bias, c.scale, c.shift,
                c.v[0], c.v[1], c.v[2], c.v[3], c.v[4], c.v[5], c.v[6], c.v[7], c.v[8], c.v[9],
                out, g.stream());
        }
        case 2: {
            Conv c(g, 10);
            void* res = g.ptr();
            void* out = g.ptr();
            return quan_qconv2d_fwd_res(QUAN_CONV_ARGS, res, out, g.stream());
        }
        case 3: {
            Conv c(g, 10);
            void* res = g.ptr();
            void* ws = g.ptr();
            const size_t bytes = static_cast<size_t>(g.next());
            void* out = g.ptr();
            return quan_qconv2d_fwd_ex(QUAN_CONV_ARGS, res, ws, bytes, out, g.stream());
        }
        case 4: {
            Conv c(g, 10);
            void* out = g.ptr();
            return quan_qconv2d_sep_fwd(QUAN_CONV_ARGS, out, g.stream());
        }
        case 5:
        case 6: {
            void* dy = g.ptr();
            void* w[4];
            for (auto& p : w) p = g.ptr();
            int v[9];
            for (auto& i : v) i = g.num();
            void* ws = g.ptr();
            const size_t bytes = static_cast<size_t>(g.next());
            void* dx = g.ptr();
            auto f = op == 5 ? quan_qconv2d_bwd_data : quan_qconv2d_sep_bwd_data;
            return f(dy, w[0], w[1], w[2], w[3], v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7],
                     v[8], ws, bytes, dx, g.stream());
        }
        case 7:
        case 8: {
            void* x = g.ptr();
            void* dy = g.ptr();
            int v[9];
            for (auto& i : v) i = g.num();
            float* d[4];
            for (auto& p : d) p = g.f32();
            auto f = op == 7 ? quan_qconv2d_bwd_weight : quan_qconv2d_sep_bwd_weight;
            return f(x, dy, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], d[0], d[1], d[2],
                     d[3], g.stream());
        }
        case 9: {
            void* x = g.ptr();
            const long long npix = g.next();
            const int C = g.num();
            void* ws = g.ptr();
            const size_t bytes = static_cast<size_t>(g.next());
            float* mean = g.f32();
            float* var = g.f32();
            return quan_iqbn_batch_stats(x, npix, C, ws, bytes, mean, var, g.stream());
        }
        case 10: {
            void* x = g.ptr();
            const long long npix = g.next();
            const int C = g.num();
            float* mean = g.f32();
            float* var = g.f32();
            float* gamma = g.f32();
            float* beta = g.f32();
            const float eps = g.real();
            const int act = g.num();
            void* out = g.ptr();
            return quan_iqbn_train_fwd(x, npix, C, mean, var, gamma, beta, eps, act, out,
                                       g.stream());
        }
        case 11: {
            Conv c(g, 9);
            void* out = g.ptr();
            return quan_qconv2d_maxpool_rgb_fwd(
                static_cast<float*>(c.x), c.w[0], c.w[1], c.w[2], c.w[3], c.bias, c.scale, c.shift,
                c.v[0], c.v[1], c.v[2], c.v[3], c.v[4], c.v[5], c.v[6], c.v[7], c.v[8], out,
                g.stream());
        }
        case 12: {
            Conv c(g, 10);
            void* ws = g.ptr();
            const size_t bytes = static_cast<size_t>(g.next());
            void* out = g.ptr();
            return quan_qconv2d_maxpool_fwd(QUAN_CONV_ARGS, ws, bytes, out, g.stream());
        }
        default:
            return QUAN_ERR_INVALID_ARG;
    }
}

// quan_qconv2d_bwd_data_workspace_size_ex of nine packed integers.
extern "C" size_t quan_packed_bwd_workspace(const long long* words) {
    Args g{words};
    int v[9];
    for (auto& i : v) i = g.num();
    return quan_qconv2d_bwd_data_workspace_size_ex(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7],
                                                   v[8]);
}
