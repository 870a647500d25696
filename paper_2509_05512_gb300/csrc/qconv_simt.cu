// qconv_simt.cu -- quaternion convolution without tcgen05 (fp32 accumulation).
//
// Handles every shape the tensor-core path does not: fp32 tensors, quaternion channel
// counts that are not multiples of 16, unaligned pointers and the 4-channel stem.  Three forms,
// chosen by their estimated times: a thread per output (qconv_direct.cuh) for few products,
// warp-level MMAs (bf16; qconv_mma.cuh) where the tensors are aligned and a filter's channels fit
// shared memory, else a tiled product of quaternions on CUDA cores (qgemm_simt.cuh).  All of
// the Hamilton-product expansion of Eq. 5 (Sec. III-B):
//   y_r = W_r x_r - W_i x_i - W_j x_j - W_k x_k
//   y_i = W_r x_i + W_i x_r + W_j x_k - W_k x_j
//   y_j = W_r x_j - W_i x_k + W_j x_r + W_k x_i
//   y_k = W_r x_k + W_i x_j - W_j x_i + W_k x_r
// summed over taps and input quaternion channels, followed by the fused epilogue
// act(scale * (acc + bias) + shift + residual) (IQBN inference form of Eq. 11-12).
// The separable form of Eq. 7 (s.sep) keeps only the diagonal convolutions
// c_p = W_p x_p and mixes them with that equation's signs:
//   y_r = c_r - c_i - c_j - c_k,  y_i = c_r + c_i + c_j - c_k,
//   y_j = c_r - c_i + c_j + c_k,  y_k = c_r + c_i - c_j + c_k.
#include <cuda_bf16.h>

#include "internal.h"
#include "qconv_direct.cuh"
#include "qgemm_simt.cuh"

namespace quan {
namespace {

template <typename T>
cudaError_t launch_direct(const ConvShape& s, const void* x, const void* const w[4],
                          const EpilogueArgs& ep, void* out, cudaStream_t stream) {
    last_variant = "direct";
    auto kern = s.sep ? qd::fwd_kernel<T, true> : qd::fwd_kernel<T, false>;
    return qd::launch(kern, s.M * s.Qout, stream, s, static_cast<const T*>(x),
                      static_cast<const T*>(w[0]), static_cast<const T*>(w[1]),
                      static_cast<const T*>(w[2]), static_cast<const T*>(w[3]), ep,
                      static_cast<T*>(out));
}

template <typename T>
cudaError_t launch_fwd(const ConvShape& s, const void* x, const void* const w[4],
                       const EpilogueArgs& ep, void* out, int num_sms, cudaStream_t stream) {
    if (s.M == 0 || s.Qout == 0) return cudaSuccess;
    last_variant = "tiles";
    qg::Params p = {};
    p.s = s;
    for (int l = 0; l < 4; ++l) p.a[l] = w[l];
    p.b = x;
    p.ep = ep;
    p.out = out;
    return s.sep ? qg::launch<T, qg::FWD, true>(p, s.Qout, s.M, 1, num_sms, stream)
                 : qg::launch<T, qg::FWD, false>(p, s.Qout, s.M, 1, num_sms, stream);
}

}  // namespace

cudaError_t launch_qconv_simt_bf16(const ConvShape& s, const void* x, const void* const w[4],
                                   const EpilogueArgs& ep, void* out, int num_sms,
                                   cudaStream_t stream) {
    const bool mma = mma_fwd_supported(s, x, out, ep.residual);
    if (qd::fwd_time(s, false, num_sms) <
        (mma ? mma_fwd_time(s, num_sms) : qg::fwd_time(s, num_sms)))
        return launch_direct<__nv_bfloat16>(s, x, w, ep, out, stream);
    if (mma) return launch_mma_fwd(s, x, w, ep, out, num_sms, stream);
    return launch_fwd<__nv_bfloat16>(s, x, w, ep, out, num_sms, stream);
}

cudaError_t launch_qconv_simt_f32(const ConvShape& s, const void* x, const void* const w[4],
                                  const EpilogueArgs& ep, void* out, int num_sms,
                                  cudaStream_t stream) {
    if (qd::fwd_time(s, true, num_sms) < qg::fwd_time(s, num_sms))
        return launch_direct<float>(s, x, w, ep, out, stream);
    return launch_fwd<float>(s, x, w, ep, out, num_sms, stream);
}

}  // namespace quan
