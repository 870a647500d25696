// qconv_mma.cuh -- bf16 quaternion convolution and its two gradients for channel counts off
// the tcgen05 kernels' grid (quaternion channels that are not multiples of 16), on warp-level
// tensor-core instructions (mma.sync m16n8k16, bf16 in, fp32 out).  Included by qconv_mma.cu.
//
// Such layers are narrow (a few dozen real channels), so they are bound by memory and by the
// work around the products, not by the tensor pipe: 16 x 45 x 37 pixels, 24 -> 40 channels,
// 3x3 is 0.46 GFLOP on 3.4 MB.  What this form saves is that work: a tap's input channels are
// copied as 8-byte pieces (cp.async, zero-filled outside the image; C is a multiple of 4),
// where the CUDA-core form (qgemm_simt.cuh) loads and converts every bf16 by itself.
// Measured on that layer (forward, input gradient, weight gradient, caches cold): 18, 23 and
// 19 us, against 24, 37 and 60 us on CUDA cores in the tiled form and 32, 43 and 97 us with a
// thread per output; layers of fewer products go to qconv_direct.cuh.  These kernels run a few thousand instructions per warp, so code size
// shows: unrolled gather loops inlined at three places made the weight gradient 43 us.
//
// As real contractions, with the signed block weight B[q][p] = sign(q, p) W_{q xor p} of Eq. 6
// (separable form: sign(q, p) W_p, Eq. 7):
//   FWD    y[px][(q, co)]  = sum over (tap, p, ci) x[px + tap][(p, ci)] B[q][p][co][tap][ci]
//   DGRAD  dx[px][(p, ci)] = sum over (tap, q, co) dy[px - tap][(q, co)] B[q][p][co][tap][ci]
//          (the pixels of a tile share their row and column modulo the stride, so only the
//          taps that reach them are summed)
//   WGRAD  G[(q, co)][(tap, p, ci)] = sum over px dy[px][(q, co)] x[px + tap][(p, ci)], whose
//          16 blocks are then folded into the letters: dW_{q xor p} += sign(q, p) G[q][p]
// FWD and DGRAD keep the block weight of their tile of at most 64 output channels in shared
// memory ([n][k], k contiguous) for a persistent run over tiles of 64 pixels, whose gathered
// rows ([pixel][k]) are double-buffered.  WGRAD runs over tiles of 64 pixels of a chunk with
// the gathered rows of a group of taps and dy's rows double-buffered, all of a 64 x 256 tile
// of G in registers.  Its MMA sums are of one tile each and added up in fp32: a block of a wide
// layer (few blocks along the pixels) otherwise chains thousands of MMA steps.  Relative error
// against 64 bits, normal inputs, 252 -> 252 channels, 8 images of 126 x 126, 3x3: 3.6e-5 in one
// chain, 4.1e-7 so (2.33 and 2.01 ms), 1.5e-6 with a thread per weight.
#pragma once

namespace quan {
namespace qm {

constexpr int THREADS = 256;
constexpr int WARPS = 8;
constexpr int PX = 64;         // pixels per tile
constexpr int MAX_N = 64;      // FWD, DGRAD: output channels per block; WGRAD: rows of G
constexpr int WG_COLS = 256;   // WGRAD: columns of G per block
constexpr int SMEM_MAX = 220 * 1024;
enum Op { FWD = 0, DGRAD = 1 };

// The taps and pixels of one launch: FWD, or one parity-like class of DGRAD's pixels.
struct Class {
    int Hc, Wc;        // pixel grid per image
    int th, tw;        // taps
    int h0, w0;        // source row / column of pixel (0, 0)'s first tap
    int oh, ow;        // output row / column of pixel (0, 0)
    int eh, ew;        // filter tap of (u, v): (eh + u tstep, ew + v tstep)
    int tile0;         // first tile
    long long M;
};
constexpr int MAX_CLASSES = 16;

struct Params {
    ConvShape s;
    const __nv_bfloat16* w[4];
    const __nv_bfloat16* src;     // x or dy, [N][Hs][Ws][C]
    EpilogueArgs ep;
    __nv_bfloat16* out;           // [N][Hd][Wd][Cd]
    int C, Hs, Ws, Cd, Hd, Wd;
    int istep;                    // source step per pixel (FWD: stride), per tap +1 or -1
    int tdir;
    int tstep, ostep;             // DGRAD: stride
    int kmax;                     // largest K of a class, rounded up to 16
    int stages;                   // pixel buffers: 2, or 1 where two do not fit
    int stage_letters;            // the four letters fit the pixel buffers and are 4-byte aligned
    int ntiles, tiles, ncls;      // channel tiles; pixel tiles of all classes
    Class cls[MAX_CLASSES];
};

struct WParams {
    ConvShape s;
    const __nv_bfloat16* x;
    const __nv_bfloat16* dy;
    float* dw[4];
    int tg, groups;               // taps per group, groups
    int mt;                       // row tiles of 64
    int cols, rows;               // tg * Cin rounded up to 16; rows of a row tile rounded up
    int chunks;                   // blocks along the pixels
    long long chunk;              // pixels of each (a multiple of PX)
};

__device__ __forceinline__ void cp8(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src),
                 "r"(ok ? 8 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                    uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
        "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Signs of Eq. 5 (component q from component p) and of Eq. 7.
template <bool SEP>
__device__ __forceinline__ bool negative(int q, int p) {
    constexpr uint32_t FULL = (1u << 1) | (1u << 2) | (1u << 3) | (1u << 6) | (1u << 11) |
                              (1u << 13);
    constexpr uint32_t EQ7 = (1u << 1) | (1u << 2) | (1u << 3) | (1u << 7) | (1u << 9) |
                             (1u << 14);
    return ((SEP ? EQ7 : FULL) >> (4 * q + p)) & 1u;
}

__device__ __forceinline__ float activate(float z, int act) {
    if (act == 1) return fmaxf(z, 0.0f);
    if (act == 2) return z / (1.0f + __expf(-z));
    return z;
}

__device__ __forceinline__ bool not_finite(float v) { return !(fabsf(v) <= 3.402823466e+38f); }

// The taps of a pixel inside the source only: the MMAs multiply the zeros that stand for the
// padding as well, which makes NaN of an infinite or NaN weight.  False where no tap is
// outside (the MMAs' sum stands), else the sum without them.  m: the pixel's index in its
// class; brow: its channel's row of the block weight.
__device__ __forceinline__ bool sum_inside(const Params& p, const Class& c,
                                           const __nv_bfloat16* brow, unsigned m, float& sum) {
    const unsigned row = m / static_cast<unsigned>(c.Wc), n = row / static_cast<unsigned>(c.Hc);
    const int hb = static_cast<int>(row - n * c.Hc) * p.istep + c.h0;
    const int wb = static_cast<int>(m - row * c.Wc) * p.istep + c.w0;
    const __nv_bfloat16* img = p.src + static_cast<long long>(n) * p.Hs * p.Ws * p.C;
    bool outside = false;
    sum = 0.f;
#pragma unroll 1
    for (int t = 0; t < c.th * c.tw; ++t) {
        const int u = t / c.tw, h = hb + p.tdir * u, w = wb + p.tdir * (t - u * c.tw);
        if (h < 0 || h >= p.Hs || w < 0 || w >= p.Ws) {
            outside = true;
            continue;
        }
        const __nv_bfloat16* g = img + (static_cast<long long>(h) * p.Ws + w) * p.C;
#pragma unroll 1
        for (int k = 0; k < p.C; ++k)
            sum = fmaf(__bfloat162float(brow[t * p.C + k]), __bfloat162float(g[k]), sum);
    }
    return outside;
}

template <int OP, bool SEP>
__global__ void __launch_bounds__(THREADS) qconv_mma_kernel(const __grid_constant__ Params p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const ConvShape& s = p.s;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int ld = p.kmax + 8;  // row pitch in elements: an odd number of 16-byte units
    __nv_bfloat16* sB = reinterpret_cast<__nv_bfloat16*>(smem);            // [MAX_N][ld]
    __nv_bfloat16* sA = sB + MAX_N * ld;                                   // [stages][PX][ld]
    int* tab = reinterpret_cast<int*>(sA + p.stages * PX * ld);            // [kmax / 4]
    const int nt = static_cast<int>(blockIdx.x) % p.ntiles;
    const int me = static_cast<int>(blockIdx.x) / p.ntiles;
    const int nblk = static_cast<int>(gridDim.x) / p.ntiles;
    const int n0 = nt * MAX_N;
    const int nn = p.Cd - n0 < MAX_N ? p.Cd - n0 : MAX_N;  // output channels of this block
    const int Q = OP == FWD ? s.Qout : s.Qin;              // per output component
    const int Qs = OP == FWD ? s.Qin : s.Qout;             // per source component
    const int taps_all = s.kh * s.kw;
    const uint32_t aB = smem_u32(sB), aA = smem_u32(sA);
    __shared__ float2 affine[MAX_N];  // y = scale (acc + bias) + shift as (scale, offset)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (OP == FWD && tid < nn) {
        const int ch = n0 + tid;
        const float sc = p.ep.scale ? __ldg(p.ep.scale + ch) : 1.f;
        const float sh = p.ep.scale ? __ldg(p.ep.shift + ch) : 0.f;
        affine[tid] = make_float2(sc, p.ep.bias ? fmaf(sc, __ldg(p.ep.bias + ch), sh) : sh);
    }

    int tile = me;
    for (int ci = 0; ci < p.ncls; ++ci) {
        const Class& c = p.cls[ci];
        const int tend = c.tile0 + static_cast<int>((c.M + PX - 1) / PX);
        if (tile >= tend) continue;
        const int taps = c.th * c.tw, K = taps * p.C, K16 = (K + 15) & ~15;
        const int chunks = K / 4;  // 8-byte pieces per pixel
        __syncthreads();           // the previous class's last products have read sA and sB
        // the letters as they are, into the pixel buffers' space (one round trip to memory;
        // read element by element where they do not fit or are not 4-byte aligned)
        const __nv_bfloat16* raw = nullptr;
        const int per = s.Qout * taps_all * s.Qin;
        if (p.stage_letters) {
#pragma unroll 1
            for (int l = 0; l < 4; ++l)
                for (int i = tid; i < per / 2; i += THREADS)
                    cp4(aA + static_cast<uint32_t>(l * per * 2 + 4 * i), p.w[l] + 2 * i);
            cp_commit();
            raw = sA;
        }
        // the class's pieces: tap (u, v) and channel of each
        for (int i = tid; i < chunks; i += THREADS) {
            const int t = i / (p.C / 4), c4 = i - t * (p.C / 4);
            const int u = t / c.tw, v = t - u * c.tw;
            tab[i] = (u << 24) | (v << 16) | (4 * c4);
        }
        cp_wait<0>();
        __syncthreads();
        // the block weight's rows n0 .. n0 + nn - 1, rows past them zero.  A thread keeps its
        // k (tap, source component and channel) and walks the rows without divisions
        for (int k = tid; k < K; k += THREADS) {
            const int t = k / p.C, kc = k - t * p.C;
            const int u = t / c.tw, w = t - u * c.tw;
            const int tap = (c.eh + u * p.tstep) * s.kw + c.ew + w * p.tstep;
            const int a = kc / Qs, ca = kc - a * Qs;
            int b = n0 / Q, cb = n0 - b * Q;  // output component and channel of row r
#pragma unroll 1
            for (int r0 = 0; r0 < MAX_N; r0 += 8) {
                __nv_bfloat16 v[8];  // eight loads in flight
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    v[r] = __float2bfloat16_rn(0.f);
                    if (r0 + r < nn) {
                        const int q = OP == FWD ? b : a, pc = OP == FWD ? a : b;
                        const int co = OP == FWD ? cb : ca, cin = OP == FWD ? ca : cb;
                        const int L = SEP ? pc : (q ^ pc);
                        const int e = (co * taps_all + tap) * s.Qin + cin;
                        v[r] = raw ? raw[L * per + e] : __ldg(p.w[L] + e);
                        if (negative<SEP>(q, pc)) v[r] = __hneg(v[r]);
                    }
                    if (++cb == Q) {
                        cb = 0;
                        ++b;
                    }
                }
#pragma unroll
                for (int r = 0; r < 8; ++r) sB[(r0 + r) * ld + k] = v[r];
            }
        }
        __syncthreads();
        // columns past K: zero in both operands
        for (int i = tid; i < (K16 - K) * (MAX_N + p.stages * PX); i += THREADS) {
            const int r = i / (K16 - K), k = K + i - r * (K16 - K);
            sB[r * ld + k] = __float2bfloat16_rn(0.f);  // (sA's rows follow sB's)
        }
        __syncthreads();

        // gather of a tile: warp w copies pixels w, w + 8, .., lane l locating pixel w + 8 l
        auto gather = [&](int t, int buf) {
            int pn, ph, pw;
            {
                const unsigned m = static_cast<unsigned>(t - c.tile0) * PX + warp + WARPS * (lane & 7);
                const bool in = m < static_cast<unsigned>(c.M);
                const unsigned mm = in ? m : 0u;
                const unsigned row = mm / static_cast<unsigned>(c.Wc);
                const unsigned n = row / static_cast<unsigned>(c.Hc);
                pn = in ? static_cast<int>(n) : -1;
                ph = static_cast<int>(row - n * c.Hc) * p.istep + c.h0;
                pw = static_cast<int>(mm - row * c.Wc) * p.istep + c.w0;
            }
#pragma unroll 1
            for (int x = 0; x < PX / WARPS; ++x) {
                const int r = warp + WARPS * x;
                const int n = __shfl_sync(0xffffffffu, pn, x);
                const int hb = __shfl_sync(0xffffffffu, ph, x);
                const int wb = __shfl_sync(0xffffffffu, pw, x);
                const bool in = n >= 0;
                const __nv_bfloat16* img =
                    p.src + static_cast<long long>(n) * p.Hs * p.Ws * p.C;
                const uint32_t dst = aA + static_cast<uint32_t>((buf * PX + r) * ld * 2);
#pragma unroll 1
                for (int q = lane; q < chunks; q += 32) {
                    const int e = tab[q];
                    const int h = hb + p.tdir * (e >> 24), w = wb + p.tdir * ((e >> 16) & 255);
                    const bool ok = in && h >= 0 && h < p.Hs && w >= 0 && w < p.Ws;
                    const __nv_bfloat16* g =
                        ok ? img + (static_cast<long long>(h) * p.Ws + w) * p.C + (e & 0xffff)
                           : p.src;
                    cp8(dst + 8u * q, g, ok);
                }
            }
        };
        // warp: pixels 16 (warp & 3) .., channel tiles of 8: (warp >> 2) * 4 ..
        const int m0 = 16 * (warp & 3), nb = 32 * (warp >> 2);
        const uint32_t fa = aA + static_cast<uint32_t>(((m0 + (lane & 15)) * ld +
                                                        8 * (lane >> 4)) * 2);
        const uint32_t fb = aB + static_cast<uint32_t>(
                                     ((nb + (lane & 7) + 8 * (lane >> 4)) * ld +
                                      8 * ((lane >> 3) & 1)) * 2);
        const bool hi = nb + 16 < nn;  // channel tiles 2 and 3 in use
        int buf = 0, ahead = 0, lt = tile;  // tiles requested ahead, the next to request
        for (; tile < tend; tile += nblk) {
            // (one place that gathers: short kernels pay for every line of code they fetch)
#pragma unroll 1
            for (; ahead < p.stages; ++ahead, lt += nblk) {
                if (lt < tend) gather(lt, (buf + ahead) & (p.stages - 1));
                cp_commit();
            }
            if (p.stages == 2) cp_wait<1>();
            else cp_wait<0>();
            __syncthreads();
            float acc[4][4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[t][e] = 0.f;
            if (nb < nn) {
                const uint32_t a0 = fa + static_cast<uint32_t>(buf * PX * ld * 2);
#pragma unroll 2
                for (int k = 0; k < K16; k += 16) {
                    uint32_t a[4], b[4];
                    ldsm4(a, a0 + 2u * k);
                    ldsm4(b, fb + 2u * k);
                    mma(acc[0], a, b[0], b[1]);
                    mma(acc[1], a, b[2], b[3]);
                    if (hi) {
                        ldsm4(b, fb + 2u * k + static_cast<uint32_t>(16 * ld * 2));
                        mma(acc[2], a, b[0], b[1]);
                        mma(acc[3], a, b[2], b[3]);
                    }
                }
                // output pixel of the class's pixel m
                auto pixel = [&](long long m) {
                    if constexpr (OP == FWD) return m;
                    const unsigned mm = static_cast<unsigned>(m);
                    const unsigned row = mm / static_cast<unsigned>(c.Wc);
                    const int j = static_cast<int>(mm - row * c.Wc);
                    const unsigned n = row / static_cast<unsigned>(c.Hc);
                    const int i = static_cast<int>(row - n * c.Hc);
                    return (static_cast<long long>(n) * p.Hd + i * p.ostep + c.oh) * p.Wd +
                           j * p.ostep + c.ow;
                };
                // rows m0 + lane / 4 (+ 8), channels nb + 8 t + 2 (lane % 4), + 1
                const long long mrow = static_cast<long long>(tile - c.tile0) * PX + m0 + lane / 4;
                float check = 0.f;  // NaN when one of the sums is not finite
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const long long m = mrow + 8 * h;
                    if (m >= c.M) continue;
                    const long long o = pixel(m);
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int ch = n0 + nb + 8 * t + 2 * (lane & 3);
                        if (ch >= n0 + nn) continue;  // (nn is even)
                        float z[2] = {acc[t][2 * h], acc[t][2 * h + 1]};
                        check = fmaf(z[0], 0.f, fmaf(z[1], 0.f, check));
                        if constexpr (OP == FWD) {
                            const float2 f0 = affine[ch - n0], f1 = affine[ch - n0 + 1];
                            z[0] = fmaf(f0.x, z[0], f0.y);
                            z[1] = fmaf(f1.x, z[1], f1.y);
                            if (p.ep.residual) {
                                const auto* rp = static_cast<const __nv_bfloat16*>(p.ep.residual) +
                                                 o * p.Cd + ch;
                                z[0] += __bfloat162float(rp[0]);
                                z[1] += __bfloat162float(rp[1]);
                            }
                            if (s.act != 0) {
                                z[0] = activate(z[0], s.act);
                                z[1] = activate(z[1], s.act);
                            }
                        }
                        *reinterpret_cast<__nv_bfloat162*>(p.out + o * p.Cd + ch) =
                            __floats2bfloat162_rn(z[0], z[1]);
                    }
                }
                if (check != 0.f) {  // rare: the thread's sixteen sums once more
#pragma unroll 1
                    for (int e = 0; e < 16; ++e) {
                        const long long m = mrow + 8 * (e & 1);
                        const int row = nb + 8 * (e >> 2) + 2 * (lane & 3) + ((e >> 1) & 1);
                        float z;
                        if (m >= c.M || row >= nn ||
                            !sum_inside(p, c, sB + row * ld, static_cast<unsigned>(m), z))
                            continue;
                        const long long o = pixel(m);
                        const long long at = o * p.Cd + n0 + row;
                        if constexpr (OP == FWD) {
                            z = fmaf(affine[row].x, z, affine[row].y);
                            if (p.ep.residual)
                                z += __bfloat162float(
                                    static_cast<const __nv_bfloat16*>(p.ep.residual)[at]);
                            z = activate(z, s.act);
                        }
                        p.out[at] = __float2bfloat16_rn(z);
                    }
                }
            }
            __syncthreads();  // every warp has read this buffer
            buf = (buf + 1) & (p.stages - 1);
            --ahead;
        }
        cp_wait<0>();
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <bool SEP>
__global__ void __launch_bounds__(THREADS, 1) qconv_mma_dw_kernel(const __grid_constant__ WParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const ConvShape& s = p.s;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int ldx = p.cols + 8, ldy = p.rows + 8;  // pitches: odd numbers of 16-byte units
    __nv_bfloat16* sX = reinterpret_cast<__nv_bfloat16*>(smem);  // [2][PX][ldx]
    __nv_bfloat16* sY = sX + 2 * PX * ldx;                       // [2][PX][ldy]
    __shared__ int tab[WG_COLS / 4];
    const int by = static_cast<int>(blockIdx.x) / p.chunks;
    const int grp = by % p.groups, mt = by / p.groups;
    const int tap0 = grp * p.tg, taps_all = s.kh * s.kw;
    const int tn = taps_all - tap0 < p.tg ? taps_all - tap0 : p.tg;
    const int r0 = mt * MAX_N;
    const int rn = s.Cout - r0 < MAX_N ? s.Cout - r0 : MAX_N;  // dy channels of this block
    const int cn = tn * s.Cin;
    const int xch = cn / 4, ych = rn / 4;  // 8-byte pieces per pixel
    for (int i = tid; i < xch; i += THREADS) {
        const int t = i / (s.Cin / 4), c4 = i - t * (s.Cin / 4);
        const int dh = (tap0 + t) / s.kw, dw = tap0 + t - dh * s.kw;
        tab[i] = (dh << 24) | (dw << 16) | (4 * c4);
    }
    // columns past the data: zero (their products are not stored, but must not be NaN: they
    // share no accumulator with stored ones; zeroed so that no uninitialised value is read)
    for (int i = tid; i < 2 * PX * (ldx - cn); i += THREADS) {
        const int r = i / (ldx - cn);
        sX[r * ldx + cn + i - r * (ldx - cn)] = __float2bfloat16_rn(0.f);
    }
    for (int i = tid; i < 2 * PX * (ldy - rn); i += THREADS) {
        const int r = i / (ldy - rn);
        sY[r * ldy + rn + i - r * (ldy - rn)] = __float2bfloat16_rn(0.f);
    }
    const long long beg = (static_cast<int>(blockIdx.x) - by * p.chunks) * p.chunk;
    long long end = beg + p.chunk;
    if (end > s.M) end = s.M;
    const uint32_t aX = smem_u32(sX), aY = smem_u32(sY);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    auto gather = [&](long long m0, int buf) {
        int pn, ph, pw;  // lane l locates pixel warp + 8 l
        {
            const long long m = m0 + warp + WARPS * (lane & 7);
            const bool in = m < end;
            const unsigned mm = static_cast<unsigned>(in ? m : beg);
            const unsigned row = mm / static_cast<unsigned>(s.Wo);
            const unsigned n = row / static_cast<unsigned>(s.Ho);
            pn = in ? static_cast<int>(n) : -1;
            ph = static_cast<int>(row - n * s.Ho) * s.stride - s.pad;
            pw = static_cast<int>(mm - row * s.Wo) * s.stride - s.pad;
        }
#pragma unroll 1
        for (int t = 0; t < PX / WARPS; ++t) {
            const int r = warp + WARPS * t;
            const long long m = m0 + r;
            const int n = __shfl_sync(0xffffffffu, pn, t);
            const int hb = __shfl_sync(0xffffffffu, ph, t);
            const int wb = __shfl_sync(0xffffffffu, pw, t);
            const bool in = n >= 0;
            const __nv_bfloat16* img = p.x + static_cast<long long>(n) * s.H * s.W * s.Cin;
            const uint32_t dx = aX + static_cast<uint32_t>((buf * PX + r) * ldx * 2);
#pragma unroll 1
            for (int q = lane; q < xch; q += 32) {
                const int e = tab[q];
                const int h = hb + (e >> 24), w = wb + ((e >> 16) & 255);
                const bool ok = in && h >= 0 && h < s.H && w >= 0 && w < s.W;
                cp8(dx + 8u * q,
                    ok ? img + (static_cast<long long>(h) * s.W + w) * s.Cin + (e & 0xffff) : p.x,
                    ok);
            }
            const uint32_t dd = aY + static_cast<uint32_t>((buf * PX + r) * ldy * 2);
#pragma unroll 1
            for (int q = lane; q < ych; q += 32)
                cp8(dd + 8u * q, in ? p.dy + m * s.Cout + r0 + 4 * q : p.dy, in);
        }
    };

    // warp: column tiles of 16 at 16 (warp + 8 t), t = 0, 1; all row tiles of 16
    float acc[4][4][4];  // [row tile][column tile of 8][..]: the sums of one pixel tile
    float sum[4][4][4];  // of all tiles
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[a][b][e] = sum[a][b][e] = 0.f;
    int buf = 0;
    long long lm = beg;  // the next tile to request
    for (long long m0 = beg; m0 < end; m0 += PX) {
        // (one place that gathers: short kernels pay for every line of code they fetch)
#pragma unroll 1
        for (; lm <= m0 + PX; lm += PX) {
            if (lm < end) gather(lm, lm == m0 ? buf : buf ^ 1);
            cp_commit();
        }
        cp_wait<1>();
        __syncthreads();
#pragma unroll 1
        for (int k = 0; k < PX; k += 16) {
            // x rows k + .., columns: [k][n] storage, transposed fragments
            uint32_t b[2][4];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int n = 16 * (warp + 8 * t);
                if (n < p.cols)
                    ldsm4t(b[t], aX + static_cast<uint32_t>(
                                          ((buf * PX + k + (lane & 7) + 8 * ((lane >> 3) & 1)) *
                                               ldx + n + 8 * (lane >> 4)) * 2));
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                if (16 * a >= p.rows) break;
                // dy: [k][m] storage, transposed fragments
                uint32_t f[4];
                ldsm4t(f, aY + static_cast<uint32_t>(
                                   ((buf * PX + k + (lane & 7) + 8 * (lane >> 4)) * ldy +
                                    16 * a + 8 * ((lane >> 3) & 1)) * 2));
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (16 * (warp + 8 * t) >= p.cols) continue;
                    mma(acc[a][2 * t], f, b[t][0], b[t][1]);
                    mma(acc[a][2 * t + 1], f, b[t][2], b[t][3]);
                }
            }
        }
        // The MMAs round each step towards zero, so a chain of them loses accuracy with its
        // length: fp32 additions, rounded to nearest, take over after every tile's four.
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    sum[a][t][e] += acc[a][t][e];
                    acc[a][t][e] = 0.f;
                }
        __syncthreads();
        buf ^= 1;
    }
    cp_wait<0>();
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // G to shared memory, then every letter element adds its four blocks and goes out once
    float* sG = reinterpret_cast<float*>(smem);
    const int ldg = p.cols + 1;
    float check = 0.f;  // NaN when one of the sums is not finite
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        if (16 * a >= p.rows) break;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int n = 16 * (warp + 8 * (t >> 1)) + 8 * (t & 1) + 2 * (lane & 3);
            if (n >= p.cols) continue;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                sG[(16 * a + lane / 4 + 8 * (e >> 1)) * ldg + n + (e & 1)] = sum[a][t][e];
                check = fmaf(sum[a][t][e], 0.f, check);
            }
        }
    }
    // Rare: the thread's sums that are not finite once more, over the pixels whose tap is inside
    // the image (the MMAs multiply dy by the zeros that stand for the padding).
    if (check != 0.f) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i) {
            const int r = 16 * (i >> 4) + lane / 4 + 8 * ((i >> 1) & 1);
            const int n = 16 * (warp + 8 * ((i >> 3) & 1)) + 8 * ((i >> 2) & 1) + 2 * (lane & 3) + (i & 1);
            if (r >= rn || n >= cn || !not_finite(sG[r * ldg + n])) continue;
            const int t = n / s.Cin, dh = (tap0 + t) / s.kw, dw = tap0 + t - dh * s.kw;
            float g = 0.f;
#pragma unroll 1
            for (long long m = beg; m < end; ++m) {
                const unsigned row = static_cast<unsigned>(m) / static_cast<unsigned>(s.Wo);
                const unsigned img = row / static_cast<unsigned>(s.Ho);
                const int h = static_cast<int>(row - img * s.Ho) * s.stride - s.pad + dh;
                const int w = static_cast<int>(static_cast<unsigned>(m) - row * s.Wo) * s.stride -
                              s.pad + dw;
                if (h < 0 || h >= s.H || w < 0 || w >= s.W) continue;
                const long long px = (static_cast<long long>(img) * s.H + h) * s.W + w;
                g = fmaf(__bfloat162float(p.dy[m * s.Cout + r0 + r]),
                         __bfloat162float(p.x[px * s.Cin + n - t * s.Cin]), g);
            }
            sG[r * ldg + n] = g;
        }
    }
    __syncthreads();
    const int per = tn * s.Qin;  // (tap, ci) of this group
#pragma unroll 1
    for (int i = tid; i < 4 * s.Qout * per; i += THREADS) {
        const int L = i / (s.Qout * per), rem = i - L * (s.Qout * per);
        const int co = rem / per, tc = rem - co * per;
        const int t = tc / s.Qin, cin = tc - t * s.Qin;
        float v = 0.f;
        bool any = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int pc = SEP ? L : (q ^ L);
            const int r = q * s.Qout + co - r0;
            if (r < 0 || r >= rn) continue;
            const float g = sG[r * ldg + t * s.Cin + pc * s.Qin + cin];
            v = negative<SEP>(q, pc) ? v - g : v + g;
            any = true;
        }
        if (any)
            atomicAdd(p.dw[L] + (static_cast<long long>(co) * taps_all + tap0 + t) * s.Qin + cin, v);
    }
}

}  // namespace qm
}  // namespace quan
