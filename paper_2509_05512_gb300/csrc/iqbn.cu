// iqbn.cu -- Independent Quaternion Batch Normalization in training mode (Eq. 11-12,
// Sec. III-C): the batch statistics of every real channel (one component of one
// quaternion channel) over N, H, W, and the normalisation with them.
//
// x is bf16 [npix][C] (NHWC flattened).  Both kernels are HBM-bound streams; every thread
// keeps one fixed group of channels (8 or 4 channels read as one 16- or 8-byte vector, or a
// single channel when C is not a multiple of 4) and walks the pixels with a grid-wide stride, so
// its per-channel state stays in registers.
//
// Statistics: each thread sums d = x - K_c and d^2 in fp32 over its pixels, with the shift
// K_c = x[0][c] (the first pixel's value, read by every thread) keeping E[d^2] - E[d]^2 free
// of cancellation when the mean is large; the block reduces in shared memory and writes its
// partial sums to its own row of a caller workspace; a second kernel adds the rows in a
// fixed order with compensated fp32 sums (no atomics: the result does not depend on
// timing) and forms
// mean = K + S1 / n and the biased variance S2 / n - (S1 / n)^2 of Eq. 11.
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"

namespace quan {
namespace {

// W channels of one pixel in one access: 16, 8 or 2 bytes.
template <int W>
struct Vec;
template <>
struct Vec<8> {
    using T = uint4;
};
template <>
struct Vec<4> {
    using T = uint2;
};
template <>
struct Vec<1> {
    using T = unsigned short;
};

template <int W>
__device__ __forceinline__ void unpack(const typename Vec<W>::T& v, float (&f)[W]) {
    if constexpr (W == 1) {
        f[0] = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(&v));
    } else {
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int i = 0; i < W / 2; ++i) {
            const float2 t = __bfloat1622float2(h[i]);
            f[2 * i] = t.x;
            f[2 * i + 1] = t.y;
        }
    }
}

template <int W>
__device__ __forceinline__ typename Vec<W>::T pack(const float (&f)[W]) {
    typename Vec<W>::T v;
    if constexpr (W == 1) {
        const __nv_bfloat16 t = __float2bfloat16_rn(f[0]);
        v = *reinterpret_cast<const unsigned short*>(&t);
    } else {
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
        for (int i = 0; i < W / 2; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    }
    return v;
}

// W channels per thread (one 16- or 8-byte vector, or a scalar); G = C / W channel groups;
// blockDim.x = G * R, R pixel rows per block.
// Four blocks per SM, the grid's share: at 72 registers only three fit, and the rest ran as a
// second wave of a quarter of the work.
template <int W>
__global__ void __launch_bounds__(256, 4) iqbn_stats_kernel(const __nv_bfloat16* __restrict__ x,
                                                         long long npix, int C, int G,
                                                         float* __restrict__ part) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    extern __shared__ float red[];  // [2][blockDim.x][W]
    const int slot = threadIdx.x % G, row = threadIdx.x / G;
    const int R = blockDim.x / G;
    const int c0 = slot * W;
    using V = typename Vec<W>::T;
    float K[W], a1[W], a2[W];
    unpack<W>(__ldg(reinterpret_cast<const V*>(x + c0)), K);
#pragma unroll
    for (int i = 0; i < W; ++i) a1[i] = a2[i] = 0.f;
    const long long stride = static_cast<long long>(gridDim.x) * R;
    auto add = [&](const V& raw) {
        float v[W];
        unpack<W>(raw, v);
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const float d = v[i] - K[i];
            a1[i] += d;
            a2[i] = fmaf(d, d, a2[i]);
        }
    };
    long long p = static_cast<long long>(blockIdx.x) * R + row;
    // eight independent loads in flight per thread, then the remainder one at a time
    for (; p + 7 * stride < npix; p += 8 * stride) {
        V raw[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            raw[k] = __ldg(reinterpret_cast<const V*>(x + (p + k * stride) * C + c0));
#pragma unroll
        for (int k = 0; k < 8; ++k) add(raw[k]);
    }
    for (; p < npix; p += stride) add(__ldg(reinterpret_cast<const V*>(x + p * C + c0)));
    float* r1 = red;
    float* r2 = red + blockDim.x * W;
#pragma unroll
    for (int i = 0; i < W; ++i) {
        r1[threadIdx.x * W + i] = a1[i];
        r2[threadIdx.x * W + i] = a2[i];
    }
    __syncthreads();
    if (row == 0) {
        for (int r = 1; r < R; ++r) {
#pragma unroll
            for (int i = 0; i < W; ++i) {
                a1[i] += r1[(r * G + slot) * W + i];
                a2[i] += r2[(r * G + slot) * W + i];
            }
        }
        float* row1 = part + static_cast<size_t>(blockIdx.x) * 2 * C;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            row1[c0 + i] = a1[i];
            row1[C + c0 + i] = a2[i];
        }
    }
}

// Compensated (Kahan) fp32 addition: the running sum and its lost low-order part.
__device__ __forceinline__ void kahan_add(float& sum, float& comp, float v) {
    const float y = v - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// Sum of the partial rows per channel in a fixed order (row lane rl takes every 128th or
// 32nd, compensated fp32; then the lanes as a tree, also compensated), then
// mean = K + S1 / n and var = max(S2 / n - (S1 / n)^2, 0) (these last few operations per
// channel in fp64; the sums stay in fp32 pairs, the double-precision rate of this part being
// low: the tree in fp64 took 9 us, and these operations, with the division 1 / n on the device
// and by a warp for each of the block's channels, 1.2 us: one warp does them for all, and the
// host divides).
// Block: 8 channels x 128 row lanes, so a lane's chain is a few loads long (32 channels x 32
// lanes, 19 rows each and 32 lanes added one by one, took 8.4 us for 256 channels); x 32 lanes
// for up to 64 rows (small tensors).
constexpr int FIN_C = 8;
// (s, e) += (s2, e2): the sum's rounding error, exact by Knuth's two-sum, goes to e.
__device__ __forceinline__ void pair_add(float& s, float& e, float s2, float e2) {
    const float t = s + s2, b = t - s;
    e = e + e2 + ((s - (t - b)) + (s2 - b));
    s = t;
}
__global__ void __launch_bounds__(1024) iqbn_finalize_kernel(const __nv_bfloat16* __restrict__ x,
                                                             double inv_n, int C, int rows,
                                                             const float* __restrict__ part,
                                                             float* __restrict__ mean,
                                                             float* __restrict__ var) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __shared__ float2 red[2][FIN_C][32], total[2][FIN_C];
    const int cl = threadIdx.x % FIN_C, rl = threadIdx.x / FIN_C;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int c = blockIdx.x * FIN_C + cl;
    float t1 = 0.f, t2 = 0.f, e1 = 0.f, e2 = 0.f;
    if (c < C) {
#pragma unroll 4
        for (int r = rl; r < rows; r += blockDim.x / FIN_C) {
            kahan_add(t1, e1, part[static_cast<size_t>(r) * 2 * C + c]);
            kahan_add(t2, e2, part[static_cast<size_t>(r) * 2 * C + C + c]);
        }
    }
    e1 = -e1;  // (the running compensation is what to subtract)
    e2 = -e2;
    auto merge = [&](int k) {
        const float u1 = __shfl_xor_sync(0xffffffffu, t1, k);
        const float f1 = __shfl_xor_sync(0xffffffffu, e1, k);
        const float u2 = __shfl_xor_sync(0xffffffffu, t2, k);
        const float f2 = __shfl_xor_sync(0xffffffffu, e2, k);
        pair_add(t1, e1, u1, f1);
        pair_add(t2, e2, u2, f2);
    };
    // the warp's four row lanes of each channel (lanes cl, cl + 8, ..)
#pragma unroll
    for (int k = FIN_C; k < 32; k *= 2) merge(k);
    if (lane < FIN_C) {
        red[0][cl][warp] = make_float2(t1, e1);
        red[1][cl][warp] = make_float2(t2, e2);
    }
    __syncthreads();
    if (warp < FIN_C) {  // warp w finishes channel w
        const bool in = lane < blockDim.x / 32;
        t1 = in ? red[0][warp][lane].x : 0.f;
        e1 = in ? red[0][warp][lane].y : 0.f;
        t2 = in ? red[1][warp][lane].x : 0.f;
        e2 = in ? red[1][warp][lane].y : 0.f;
#pragma unroll
        for (int k = 1; k < 32; k *= 2) merge(k);
        if (lane == 0) {
            total[0][warp] = make_float2(t1, e1);
            total[1][warp] = make_float2(t2, e2);
        }
    }
    __syncthreads();
    const int cw = blockIdx.x * FIN_C + threadIdx.x;
    if (threadIdx.x < FIN_C && cw < C) {
        const float2 s1 = total[0][threadIdx.x], s2 = total[1][threadIdx.x];
        const double m1 = (static_cast<double>(s1.x) + s1.y) * inv_n;
        const double m2 = (static_cast<double>(s2.x) + s2.y) * inv_n - m1 * m1;
        mean[cw] = static_cast<float>(static_cast<double>(__bfloat162float(x[cw])) + m1);
        var[cw] = m2 > 0.0 ? static_cast<float>(m2) : 0.0f;
    }
}

__device__ __forceinline__ float act_fn(float z, int act) {
    if (act == 1) return fmaxf(z, 0.0f);
    // SiLU z / (1 + e^-z), e^-z = 2^(-z log2 e), as (z / 16) (16 / (1 + 2^x)): the sixteenth of
    // the divisor stays below 2^126 for every finite 2^x, so its approximate reciprocal is no
    // subnormal, and a subnormal 2^x does not change 1 + 2^x: both may flush subnormals.  With
    // an exact division SiLU took the pass over its memory time: 74 us for the statistics
    // and this kernel at 64 x 56 x 56 x 256, now 61 (ReLU: 57).
    if (act == 2)
        return (z * 0.0625f) *
               rcp_approx_ftz(fmaf(ex2_approx_ftz(z * -1.44269504f), 0.0625f, 0.0625f));
    return z;
}

// Read for the last time: the line is the first to leave L2.
__device__ __forceinline__ uint4 ld_last(const uint4* p, uint64_t policy) {
    uint4 v;
    asm volatile("ld.global.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(policy)
                 : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_last(const uint2* p, uint64_t policy) {
    uint2 v;
    asm volatile("ld.global.L2::cache_hint.v2.b32 {%0, %1}, [%2], %3;"
                 : "=r"(v.x), "=r"(v.y)
                 : "l"(p), "l"(policy)
                 : "memory");
    return v;
}
__device__ __forceinline__ unsigned short ld_last(const unsigned short* p, uint64_t) { return *p; }

// out = act(gamma (x - mean) / sqrt(var + eps) + beta) (Eq. 11-12), as scale * x + shift.
// The pixels are walked from the last to the first: the statistics, which usually ran just
// before, read x from first to last, so its end is what L2 still holds.
template <int W>
__global__ void __launch_bounds__(256) iqbn_apply_kernel(
    const __nv_bfloat16* x, long long npix, int C, int G, const float* __restrict__ mean,
    const float* __restrict__ var, const float* __restrict__ gamma,
    const float* __restrict__ beta, float eps, int act, __nv_bfloat16* out) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int slot = threadIdx.x % G, row = threadIdx.x / G;
    const int R = blockDim.x / G;
    const int c0 = slot * W;
    float sc[W], sh[W];
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const int c = c0 + i;
        const float g = gamma ? gamma[c] : 1.0f;
        const float b = beta ? beta[c] : 0.0f;
        sc[i] = g / sqrtf(var[c] + eps);
        sh[i] = fmaf(-mean[c], sc[i], b);
    }
    const long long stride = static_cast<long long>(gridDim.x) * R;
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    const long long end = npix - 1;  // pixel end - p in place of p
    using V = typename Vec<W>::T;
    auto load = [&](long long q) {
        return ld_last(reinterpret_cast<const V*>(x + (end - q) * C + c0), policy);
    };
    auto finish = [&](long long q, const V& raw) {
        float v[W];
        unpack<W>(raw, v);
#pragma unroll
        for (int i = 0; i < W; ++i) v[i] = act_fn(fmaf(v[i], sc[i], sh[i]), act);
        *reinterpret_cast<V*>(out + (end - q) * C + c0) = pack<W>(v);
    };
    long long p = static_cast<long long>(blockIdx.x) * R + row;
    // four loads in flight before the first store (each thread reads only the elements it
    // writes, so an in-place call is still safe)
    for (; p + 3 * stride < npix; p += 4 * stride) {
        V raw[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) raw[k] = load(p + k * stride);
#pragma unroll
        for (int k = 0; k < 4; ++k) finish(p + k * stride, raw[k]);
    }
    for (; p < npix; p += stride) finish(p, load(p));
}

// Channel groups, block size and grid of one launch; false if C has no layout.
bool iqbn_layout(int C, int W, long long npix, int num_sms, int per_sm, int* G, int* block,
                 int* grid) {
    const int g = C / W;
    if (g < 1 || g > 256) return false;
    const int R = 256 / g;
    *G = g;
    *block = g * R;
    long long blocks = (npix + R - 1) / R;
    const long long cap = static_cast<long long>(num_sms) * per_sm;
    if (blocks > cap) blocks = cap;
    *grid = static_cast<int>(blocks);
    return true;
}

// Channels per access: 8 (16 bytes), 4 (8 bytes: the quaternion channel counts that are no
// multiple of 8; a scalar access each instead took 135 us, now 50 us, for the statistics and
// the normalisation of 40 M elements in 44 channels), or 1.  Small tensors keep the scalar
// accesses: with four channels a thread a block spans more pixels, and its last additions, row
// after row, take longer than the loads (1024 pixels of 12 channels, statistics and normalisation:
// 7.5 us with 8-byte accesses, 5.5 with scalar ones; 16,384: 8.4 and 10.2).
int iqbn_width(int C, long long npix, const void* a, const void* b) {
    if (iqbn_vec_ok(C, a, b)) return 8;
    const uintptr_t bits = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b);
    return C % 4 == 0 && bits % 8 == 0 && (C > 256 || npix * C >= 131072) ? 4 : 1;
}

}  // namespace

bool iqbn_vec_ok(int C, const void* a, const void* b) {
    return C % 8 == 0 && C / 8 <= 256 && reinterpret_cast<uintptr_t>(a) % 16 == 0 &&
           reinterpret_cast<uintptr_t>(b) % 16 == 0;
}

bool iqbn_supported(int C, const void* a, const void* b) {
    return iqbn_vec_ok(C, a, b) || (C >= 1 && C <= 256);
}

size_t iqbn_stats_workspace_bytes(int C) {
    return C < 1 ? 0 : static_cast<size_t>(IQBN_MAX_PARTIALS) * 2 * C * sizeof(float);
}

cudaError_t launch_iqbn_stats(const void* x, long long npix, int C, void* workspace,
                              float* mean, float* var, int num_sms, cudaStream_t stream) {
    const int W = iqbn_width(C, npix, x, x);
    int G = 0, block = 0, grid = 0;
    if (!iqbn_layout(C, W, npix, num_sms, 4, &G, &block, &grid)) return cudaErrorInvalidValue;
    if (grid > IQBN_MAX_PARTIALS) grid = IQBN_MAX_PARTIALS;
    const auto* xb = static_cast<const __nv_bfloat16*>(x);
    auto* part = static_cast<float*>(workspace);
    const size_t smem = static_cast<size_t>(2) * block * W * sizeof(float);
    auto kern = W == 8   ? iqbn_stats_kernel<8>
                : W == 4 ? iqbn_stats_kernel<4>
                         : iqbn_stats_kernel<1>;
    cudaError_t e = launch_pdl(kern, dim3(grid), dim3(block), smem, stream, xb, npix, C, G, part);
    if (e != cudaSuccess) return e;
    return launch_pdl(iqbn_finalize_kernel, dim3((C + FIN_C - 1) / FIN_C),
                      dim3(grid <= 64 ? 256 : 1024), 0, stream, xb,
                      1.0 / static_cast<double>(npix), C, grid, static_cast<const float*>(part),
                      mean, var);
}

cudaError_t launch_iqbn_apply(const void* x, long long npix, int C, const float* mean,
                              const float* var, const float* gamma, const float* beta, float eps,
                              int act, void* out, int num_sms, cudaStream_t stream) {
    const int W = iqbn_width(C, npix, x, out);
    int G = 0, block = 0, grid = 0;
    if (!iqbn_layout(C, W, npix, num_sms, 8, &G, &block, &grid)) return cudaErrorInvalidValue;
    const auto* xb = static_cast<const __nv_bfloat16*>(x);
    auto* ob = static_cast<__nv_bfloat16*>(out);
    auto kern = W == 8 ? iqbn_apply_kernel<8> : W == 4 ? iqbn_apply_kernel<4> : iqbn_apply_kernel<1>;
    return launch_pdl(kern, dim3(grid), dim3(block), 0, stream, xb, npix, C, G, mean, var, gamma,
                      beta, eps, act, ob);
}

}  // namespace quan
