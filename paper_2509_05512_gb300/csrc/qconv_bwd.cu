// qconv_bwd.cu -- gradients of the quaternion convolution before its epilogue, given
// dy = dL/dy for y = the convolution's accumulator (bias, IQBN and activation excluded).
//
// Full Hamilton form (Eq. 5): the Jacobians of the Hamilton product (Eq. 3) give, for
// every tap and channel pair,
//   dL/dX = conj(W) (x) dy,     dL/dW = dy (x) conj(X),
// conj(W) = (W_r, -W_i, -W_j, -W_k).  So
//   * the input gradient is itself a quaternion convolution: of dy, with the letters
//     conjugated, their channel axes swapped and the filter rotated by 180 degrees, padding
//     kh - 1 - pad, stride 1 (for a stride-1 forward).  bwd_transform_kernel writes those
//     letters into a caller workspace and the forward tensor-core kernels run the rest.
//     A stride-2 forward's input gradient runs by the parity classes of its pixels
//     (qconv_tc.cu), and one of any other stride as the same stride-1 convolution of dy with
//     s - 1 zero rows and columns inserted between its pixels (bwd_upsample_kernel, into
//     the workspace after the letters), when the caller's workspace would hold that tensor;
//     otherwise a kernel without tcgen05 runs;
//   * the weight gradient is a reduction over output pixels: on the tensor cores
//     (qconv_dw.cuh), or without tcgen05 chunk by chunk of pixels, fp32 partial sums added to
//     the zeroed output with atomicAdd.
// Without tcgen05 both run on warp-level MMAs (qconv_mma.cuh), or, where those do not apply, as
// the tiled CUDA-core products of qgemm_simt.cuh; an input gradient of few products takes a thread
// per quaternion (qconv_direct.cuh), by the estimated times.
// Separable form (Eq. 7): Eq. 8-10 -- the output gradients are first mixed by the matrix M
// of Eq. 9 (g_p = sum_m M[p][m] dy_m, M transposed equal to Eq. 7's sign table), then
// dL/dx_p is the transposed convolution of g_p with W_p alone and dL/dW_p the correlation
// of g_p with x_p alone.  On the tensor cores (stride 1) the input gradient is one
// convolution of dy whose block (q, p) is M[q][p] W'_q (W' the letters transposed and
// rotated, not conjugated): the forward kernel's transposed-separable mode.
#include <cuda_bf16.h>

#include "internal.h"
#include "qconv_direct.cuh"
#include "qgemm_simt.cuh"

namespace quan {
namespace {

// out_L[ci][dh][dw][co] = s_L * W_L[co][kh-1-dh][kw-1-dw][ci], s = (+1, -1, -1, -1) when
// conj, else +1.  Its output is the next kernel's weight operand, which the forward
// tensor-core kernels read before their dependency wait: this kernel does not trigger its
// dependents early, so the next one starts only once it has completed.
__global__ void __launch_bounds__(256) bwd_transform_kernel(
    int Qin, int Qout, int kh, int kw, int conj, const __nv_bfloat16* __restrict__ wr,
    const __nv_bfloat16* __restrict__ wi, const __nv_bfloat16* __restrict__ wj,
    const __nv_bfloat16* __restrict__ wk, __nv_bfloat16* __restrict__ out) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long per = static_cast<long long>(Qin) * kh * kw * Qout;
    const __nv_bfloat16* w[4] = {wr, wi, wj, wk};
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
         i < 4 * per; i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int L = static_cast<int>(i / per);
        long long r = i - L * per;
        const int co = static_cast<int>(r % Qout);
        r /= Qout;
        const int dw = static_cast<int>(r % kw);
        r /= kw;
        const int dh = static_cast<int>(r % kh);
        const int ci = static_cast<int>(r / kh);
        const long long src =
            ((static_cast<long long>(co) * kh + (kh - 1 - dh)) * kw + (kw - 1 - dw)) * Qin + ci;
        const __nv_bfloat16 v = w[L][src];
        out[i] = (L == 0 || !conj) ? v : __hneg(v);
    }
}

// Scratch of quan_qconv2d_bwd_data_static, the entry point for callers that cannot
// allocate device memory: the transformed letters of one call live here instead of in a
// caller workspace.  Every call writes all of the region it then reads, so nothing in it
// has to start at zero; calls that overlap on the GPU share it and race.  Host code must
// not pass this name to a kernel: on the host it is a stand-in, not a device address.
static __device__ __align__(256) unsigned char g_bwd_static_scratch[BWD_STATIC_SCRATCH_BYTES];

// u[n][y][x] = dy[n][y / s][x / s] where s divides y and x (and y / s < Ho, x / s < Wo),
// else 0: dy with s - 1 zeros between its pixels, [N][Hu][Wu][C], 16 bytes per thread.
__global__ void __launch_bounds__(256) bwd_upsample_kernel(const uint4* __restrict__ dy, int N,
                                                           int Ho, int Wo, int cv, int s, int Hu,
                                                           int Wu, uint4* __restrict__ u) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long total = static_cast<long long>(N) * Hu * Wu * cv;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int c = static_cast<int>(i % cv);
        const long long pix = i / cv;
        const int x = static_cast<int>(pix % Wu);
        const int y = static_cast<int>((pix / Wu) % Hu);
        const int n = static_cast<int>(pix / (static_cast<long long>(Wu) * Hu));
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (y % s == 0 && x % s == 0 && y / s < Ho && x / s < Wo)
            v = __ldg(dy + ((static_cast<long long>(n) * Ho + y / s) * Wo + x / s) * cv + c);
        u[i] = v;
    }
}

// The four weight gradients set to zero before a kernel adds to them: one launch that takes
// part in the dependent-launch chain (four memset nodes cost four launches and end it).
__global__ void __launch_bounds__(256) zero4_kernel(float* __restrict__ a, float* __restrict__ b,
                                                    float* __restrict__ c, float* __restrict__ d,
                                                    long long n) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        a[i] = 0.f;
        b[i] = 0.f;
        c[i] = 0.f;
        d[i] = 0.f;
    }
}

}  // namespace

cudaError_t launch_zero4(float* const t[4], long long n, int num_sms, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    long long blocks = (n + 255) / 256;
    if (blocks > num_sms * 8LL) blocks = num_sms * 8LL;
    return launch_pdl(zero4_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, stream,
                      t[0], t[1], t[2], t[3], n);
}

cudaError_t launch_bwd_upsample(const void* dy, int N, int Ho, int Wo, int C, int s, int Hu,
                                int Wu, void* u, int num_sms, cudaStream_t stream) {
    if (C % 8 != 0) return cudaErrorInvalidValue;
    const long long total = static_cast<long long>(N) * Hu * Wu * (C / 8);
    if (total == 0) return cudaSuccess;
    long long blocks = (total + 255) / 256;
    if (blocks > num_sms * 16LL) blocks = num_sms * 16LL;
    return launch_pdl(bwd_upsample_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0,
                      stream, static_cast<const uint4*>(dy), N, Ho, Wo, C / 8, s, Hu, Wu,
                      static_cast<uint4*>(u));
}

// Device address of the scratch on the current device (called once per device, with
// that device current, by the entry point's first call there).
cudaError_t bwd_static_scratch_address(void** ptr) {
    return cudaGetSymbolAddress(ptr, g_bwd_static_scratch);
}

size_t bwd_data_workspace_bytes(int Cin, int Cout, int kh, int kw) {
    return static_cast<size_t>(4) * (Cin / 4) * kh * kw * (Cout / 4) * 2;
}

cudaError_t launch_bwd_transform(int Cin, int Cout, int kh, int kw, const void* const w[4],
                                 bool conj, void* out, int num_sms, cudaStream_t stream) {
    const long long n = 4LL * (Cin / 4) * kh * kw * (Cout / 4);
    if (n == 0) return cudaSuccess;
    long long blocks = (n + 255) / 256;
    if (blocks > num_sms * 8LL) blocks = num_sms * 8LL;
    return launch_pdl(bwd_transform_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0,
                      stream, Cin / 4, Cout / 4, kh, kw, conj ? 1 : 0,
                      static_cast<const __nv_bfloat16*>(w[0]),
                      static_cast<const __nv_bfloat16*>(w[1]),
                      static_cast<const __nv_bfloat16*>(w[2]),
                      static_cast<const __nv_bfloat16*>(w[3]),
                      static_cast<__nv_bfloat16*>(out));
}

cudaError_t launch_bwd_data_simt(const ConvShape& s, const void* dy, const void* const w[4],
                                 void* dx, int num_sms, cudaStream_t stream) {
    if (mma_bwd_data_supported(s, dy, dx)) {
        if (qd::dx_time(s, num_sms) >= mma_bwd_data_time(s, num_sms))
            return launch_mma_bwd_data(s, dy, w, dx, num_sms, stream);
        last_variant = "direct";
        using T = __nv_bfloat16;
        return qd::launch(s.sep ? qd::dx_kernel<true> : qd::dx_kernel<false>,
                          static_cast<long long>(s.N) * s.H * s.W * s.Qin, stream, s,
                          static_cast<const T*>(dy), static_cast<const T*>(w[0]),
                          static_cast<const T*>(w[1]), static_cast<const T*>(w[2]),
                          static_cast<const T*>(w[3]), static_cast<T*>(dx));
    }
    last_variant = "tiles";
    qg::Params p = {};
    p.s = s;
    for (int l = 0; l < 4; ++l) p.a[l] = w[l];
    p.b = dy;
    p.out = dx;
    // pixel classes: rows and columns modulo the stride (at most the image's); the largest
    // is rows and columns 0, stride, 2 stride, ..
    p.cw = s.W < s.stride ? s.W : s.stride;
    const long long classes = static_cast<long long>(s.H < s.stride ? s.H : s.stride) * p.cw;
    const long long J = static_cast<long long>(s.N) * ((s.H + s.stride - 1) / s.stride) *
                        ((s.W + s.stride - 1) / s.stride);
    return s.sep ? qg::launch<__nv_bfloat16, qg::DGRAD, true>(p, s.Qin, J, classes, num_sms, stream)
                 : qg::launch<__nv_bfloat16, qg::DGRAD, false>(p, s.Qin, J, classes, num_sms,
                                                               stream);
}

cudaError_t launch_bwd_weight_simt(const ConvShape& s, const void* x, const void* dy,
                                   float* const dw[4], int num_sms, cudaStream_t stream) {
    if (mma_bwd_weight_supported(s, x, dy))
        return launch_mma_bwd_weight(s, x, dy, dw, num_sms, stream);
    last_variant = "tiles";
    const long long J = static_cast<long long>(s.kh) * s.kw * s.Qin;
    const cudaError_t e = launch_zero4(dw, J * s.Qout, num_sms, stream);
    if (e != cudaSuccess) return e;
    if (J == 0 || s.M == 0) return cudaSuccess;
    qg::Params p = {};
    p.s = s;
    p.a[0] = dy;
    p.b = x;
    for (int l = 0; l < 4; ++l) p.dw[l] = dw[l];
    // pixel chunks that give every SM about four blocks; more only adds atomics
    qg::Params t = p;
    qg::layout(&t, s.Qout, J, 2, 4);
    const long long tiles = qg::jtiles(t, J) * t.itiles;
    long long chunks = (4LL * num_sms + tiles - 1) / tiles;
    if (chunks > (s.M + qg::KC - 1) / qg::KC) chunks = (s.M + qg::KC - 1) / qg::KC;
    if (chunks < (s.M >> 30) + 1) chunks = (s.M >> 30) + 1;  // a chunk's pixels fit an int
    if (chunks > 65535) chunks = 65535;
    p.chunk = ((s.M + chunks - 1) / chunks + qg::KC - 1) / qg::KC * qg::KC;
    chunks = (s.M + p.chunk - 1) / p.chunk;
    return s.sep ? qg::launch<__nv_bfloat16, qg::WGRAD, true>(p, s.Qout, J, chunks, num_sms, stream)
                 : qg::launch<__nv_bfloat16, qg::WGRAD, false>(p, s.Qout, J, chunks, num_sms,
                                                               stream);
}

}  // namespace quan
