// qconv_mma.cu -- launches of the warp-level tensor-core kernels (qconv_mma.cuh): bf16 layers
// whose quaternion channel counts are not multiples of 16.
#include <cuda_bf16.h>

#include <atomic>

#include "internal.h"
#include "ptx.cuh"
#include "qconv_mma.cuh"

namespace quan {
namespace {

bool al(const void* p, unsigned n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; }

template <typename K>
cudaError_t allow_smem(K kern, int bytes, std::atomic<unsigned long long>& done) {
    if (bytes <= 47 * 1024) return cudaSuccess;  // (48 KB less the kernels' static part)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done.load() & bit)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, qm::SMEM_MAX);
        if (e != cudaSuccess) return e;
        done.fetch_or(bit);
    }
    return cudaSuccess;
}

int fwd_smem(int kmax, int stages) {
    return (qm::MAX_N + stages * qm::PX) * (kmax + 8) * 2 + kmax;
}

// Blocks of `smem` bytes and 256 threads (at most 96 registers each) that fit one SM.
int per_sm(int smem) {
    int n = (227 * 1024) / (smem + 1024);
    return n > 2 ? 2 : (n < 1 ? 1 : n);
}

// Shared-memory and index limits of FWD and DGRAD: K = taps * C gathered channels per pixel
// (tap and channel fit the piece table's fields).
bool fits(int kh, int kw, int C) {
    if (kh > 120 || kw > 120 || C > 32764) return false;
    const long long k = (static_cast<long long>(kh) * kw * C + 15) / 16 * 16;
    return k <= 2048 && fwd_smem(static_cast<int>(k), 1) <= qm::SMEM_MAX;
}

// Estimated time (us) of FWD and DGRAD: the block weight of each class that a block runs, 256
// columns at a time (read from global memory where the letters do not fit the pixel buffers), the
// letters, then the tiles.  Fitted to 1,120 layers of random sizes (80% between 0.8 and 1.2 of it).
struct Cost {
    double fixed, columns, unstaged, letters, product, tile;
};
constexpr Cost FWD_COST = {1.2, 2.4, 12.0, 0.24, 0.0039, 4.4};
constexpr Cost DX_COST = {2.3, 2.1, 4.6, 0.13, 0.0049, 3.5};

double op_time(const Cost& c, int Cd, long long K, int classes, long long px, double per,
               int num_sms) {
    const int kmax = static_cast<int>((K + 15) / 16 * 16);
    const int stages = fwd_smem(kmax, 2) <= qm::SMEM_MAX ? 2 : 1;
    const bool staged = 4 * per <= static_cast<double>(stages) * qm::PX * (kmax + 8);
    const int ntiles = (Cd + qm::MAX_N - 1) / qm::MAX_N;
    const double tiles = static_cast<double>((px + qm::PX - 1) / qm::PX) + classes - 1;
    double runs = num_sms * per_sm(fwd_smem(kmax, stages)) / ntiles;
    if (runs < 1) runs = 1;
    if (runs > tiles) runs = tiles;
    const double each = static_cast<double>(static_cast<long long>((tiles + runs - 1) / runs));
    const double columns = static_cast<double>((K + 255) / 256) * (classes < each ? classes : each);
    return c.fixed + columns * (c.columns + (staged ? 0.0 : c.unstaged)) +
           (staged ? 4 * per / 512 * c.letters : 0.0) + each * (kmax * c.product + c.tile);
}

template <int OP, bool SEP>
cudaError_t launch_op(qm::Params& p, int num_sms, cudaStream_t stream) {
    p.stages = fwd_smem(p.kmax, 2) <= qm::SMEM_MAX ? 2 : 1;
    const int smem = fwd_smem(p.kmax, p.stages);
    const long long per = static_cast<long long>(p.s.Qout) * p.s.kh * p.s.kw * p.s.Qin;
    p.stage_letters = per % 2 == 0 && al(p.w[0], 4) && al(p.w[1], 4) && al(p.w[2], 4) &&
                      al(p.w[3], 4) && 4 * per <= static_cast<long long>(p.stages) * qm::PX * (p.kmax + 8);
    last_variant = "mma";
    auto kern = qm::qconv_mma_kernel<OP, SEP>;
    static std::atomic<unsigned long long> done{0};
    const cudaError_t e = allow_smem(kern, smem, done);
    if (e != cudaSuccess) return e;
    p.ntiles = (p.Cd + qm::MAX_N - 1) / qm::MAX_N;
    long long runs = static_cast<long long>(num_sms) * per_sm(smem) / p.ntiles;
    if (runs < 1) runs = 1;
    if (runs > p.tiles) runs = p.tiles;
    return launch_pdl(kern, dim3(static_cast<unsigned>(runs * p.ntiles)), dim3(qm::THREADS),
                      static_cast<size_t>(smem), stream, p);
}

}  // namespace

bool mma_fwd_supported(const ConvShape& s, const void* x, const void* out, const void* residual) {
    return al(x, 8) && al(out, 4) && al(residual, 2) && s.M < (1LL << 31) &&
           fits(s.kh, s.kw, s.Cin) && s.Cout <= 64 * 64;  // (letter offsets fit an int)
}

cudaError_t launch_mma_fwd(const ConvShape& s, const void* x, const void* const w[4],
                           const EpilogueArgs& ep, void* out, int num_sms, cudaStream_t stream) {
    qm::Params p = {};
    p.s = s;
    for (int l = 0; l < 4; ++l) p.w[l] = static_cast<const __nv_bfloat16*>(w[l]);
    p.src = static_cast<const __nv_bfloat16*>(x);
    p.ep = ep;
    p.out = static_cast<__nv_bfloat16*>(out);
    p.C = s.Cin; p.Hs = s.H; p.Ws = s.W;
    p.Cd = s.Cout; p.Hd = s.Ho; p.Wd = s.Wo;
    p.istep = s.stride; p.tdir = 1; p.tstep = 1; p.ostep = 1;
    p.kmax = (s.kh * s.kw * s.Cin + 15) / 16 * 16;
    p.ncls = 1;
    p.tiles = static_cast<int>((s.M + qm::PX - 1) / qm::PX);
    qm::Class& c = p.cls[0];
    c.Hc = s.Ho; c.Wc = s.Wo; c.th = s.kh; c.tw = s.kw;
    c.h0 = c.w0 = -s.pad;
    c.M = s.M;
    return s.sep ? launch_op<qm::FWD, true>(p, num_sms, stream)
                 : launch_op<qm::FWD, false>(p, num_sms, stream);
}

double mma_fwd_time(const ConvShape& s, int num_sms) {
    return op_time(FWD_COST, s.Cout, static_cast<long long>(s.kh) * s.kw * s.Cin, 1, s.M,
                   static_cast<double>(s.Qout) * s.kh * s.kw * s.Qin, num_sms);
}

double mma_bwd_data_time(const ConvShape& s, int num_sms) {
    const int h = s.H < s.stride ? s.H : s.stride, w = s.W < s.stride ? s.W : s.stride;
    const long long taps = static_cast<long long>((s.kh + s.stride - 1) / s.stride) *
                           ((s.kw + s.stride - 1) / s.stride);
    return op_time(DX_COST, s.Cin, taps * s.Cout, h * w, static_cast<long long>(s.N) * s.H * s.W,
                   static_cast<double>(s.Qout) * s.kh * s.kw * s.Qin, num_sms);
}

bool mma_bwd_data_supported(const ConvShape& s, const void* dy, const void* dx) {
    return al(dy, 8) && al(dx, 4) && s.stride <= 4 &&
           static_cast<long long>(s.N) * s.H * s.W < (1LL << 31) && fits(s.kh, s.kw, s.Cout) &&
           s.Cin <= 64 * 64;
}

cudaError_t launch_mma_bwd_data(const ConvShape& s, const void* dy, const void* const w[4],
                                void* dx, int num_sms, cudaStream_t stream) {
    qm::Params p = {};
    p.s = s;
    for (int l = 0; l < 4; ++l) p.w[l] = static_cast<const __nv_bfloat16*>(w[l]);
    p.src = static_cast<const __nv_bfloat16*>(dy);
    p.out = static_cast<__nv_bfloat16*>(dx);
    p.C = s.Cout; p.Hs = s.Ho; p.Ws = s.Wo;
    p.Cd = s.Cin; p.Hd = s.H; p.Wd = s.W;
    p.istep = 1; p.tdir = -1; p.tstep = p.ostep = s.stride;
    for (int a = 0; a < s.stride; ++a)
        for (int b = 0; b < s.stride; ++b) {
            qm::Class& c = p.cls[p.ncls];
            c.Hc = (s.H - a + s.stride - 1) / s.stride;
            c.Wc = (s.W - b + s.stride - 1) / s.stride;
            if (a >= s.H || b >= s.W) continue;
            c.eh = (a + s.pad) % s.stride;
            c.ew = (b + s.pad) % s.stride;
            c.th = c.eh < s.kh ? (s.kh - c.eh + s.stride - 1) / s.stride : 0;
            c.tw = c.ew < s.kw ? (s.kw - c.ew + s.stride - 1) / s.stride : 0;
            c.h0 = (a + s.pad - c.eh) / s.stride;
            c.w0 = (b + s.pad - c.ew) / s.stride;
            c.oh = a;
            c.ow = b;
            c.M = static_cast<long long>(s.N) * c.Hc * c.Wc;
            c.tile0 = p.tiles;
            p.tiles += static_cast<int>((c.M + qm::PX - 1) / qm::PX);
            const int k = (c.th * c.tw * s.Cout + 15) / 16 * 16;
            if (k > p.kmax) p.kmax = k;
            ++p.ncls;
        }
    if (p.kmax < 16) p.kmax = 16;
    return s.sep ? launch_op<qm::DGRAD, true>(p, num_sms, stream)
                 : launch_op<qm::DGRAD, false>(p, num_sms, stream);
}

bool mma_bwd_weight_supported(const ConvShape& s, const void* x, const void* dy) {
    return al(x, 8) && al(dy, 8) && s.Cin <= qm::WG_COLS && s.kh <= 120 && s.kw <= 120 &&
           s.M < (1LL << 31) && s.Cout <= 1024 && static_cast<long long>(s.kh) * s.kw <= 4096;
}

cudaError_t launch_mma_bwd_weight(const ConvShape& s, const void* x, const void* dy,
                                  float* const dw[4], int num_sms, cudaStream_t stream) {
    last_variant = "mma";
    const int taps = s.kh * s.kw;
    const cudaError_t e0 =
        launch_zero4(dw, static_cast<long long>(s.Qout) * taps * s.Qin, num_sms, stream);
    if (e0 != cudaSuccess || s.M == 0) return e0;
    qm::WParams p = {};
    p.s = s;
    p.x = static_cast<const __nv_bfloat16*>(x);
    p.dy = static_cast<const __nv_bfloat16*>(dy);
    for (int l = 0; l < 4; ++l) p.dw[l] = dw[l];
    p.tg = qm::WG_COLS / s.Cin;
    if (p.tg > taps) p.tg = taps;
    p.groups = (taps + p.tg - 1) / p.tg;
    p.tg = (taps + p.groups - 1) / p.groups;  // equal groups
    p.groups = (taps + p.tg - 1) / p.tg;
    p.cols = (p.tg * s.Cin + 15) / 16 * 16;
    p.mt = (s.Cout + qm::MAX_N - 1) / qm::MAX_N;
    p.rows = p.mt > 1 ? qm::MAX_N : (s.Cout + 15) / 16 * 16;
    int smem = 2 * qm::PX * (p.cols + 8 + p.rows + 8) * 2;
    const int fold = p.rows * (p.cols + 1) * 4;
    if (fold > smem) smem = fold;
    // pixel chunks: one block per SM (its registers) over the groups and row tiles
    const long long y = static_cast<long long>(p.groups) * p.mt;
    long long chunks = num_sms / y < 1 ? 1 : num_sms / y;
    const long long tiles = (s.M + qm::PX - 1) / qm::PX;
    if (chunks > tiles) chunks = tiles;
    p.chunk = (tiles + chunks - 1) / chunks * qm::PX;
    p.chunks = static_cast<int>((s.M + p.chunk - 1) / p.chunk);
    auto kern = s.sep ? qm::qconv_mma_dw_kernel<true> : qm::qconv_mma_dw_kernel<false>;
    static std::atomic<unsigned long long> done[2];
    const cudaError_t e = allow_smem(kern, smem, done[s.sep ? 1 : 0]);
    if (e != cudaSuccess) return e;
    // (at most 4096 taps x 16 row tiles: a line of blocks, as they pass a grid's second dimension)
    return launch_pdl(kern, dim3(static_cast<unsigned>(p.chunks * y)), dim3(qm::THREADS),
                      static_cast<size_t>(smem), stream, p);
}

}  // namespace quan
