// qconv_dw.cuh -- weight gradient of the full-form quaternion convolution (Eq. 5) on the
// tensor cores, stride 1 or 2.  Included by qconv_tc.cu only.
//
// As a real contraction the forward convolution is y[px][m Qout + co] = sum over taps and
// real input channels of B[m][p] x[px + tap][p Qin + ci], with the signed block weight
// B[m][p] = sign(m, p) W_{m xor p} of Eq. 6.  Its real weight gradient for one tap is the
// plain product over output pixels
//     G_tap[c][d] = sum_px x[px + tap][c] dy[px][d]        (c: input, d: output channel),
// and each letter gathers its four signed blocks:
//     dW_L[co][tap][ci] = sum over (m, p) with m xor p = L of sign(m, p) G_tap[p Qin + ci][m Qout + co].
//
// Both MMA operands come straight from the NHWC tensors: a TMA im2col box of 64 channels x P
// pixels lands as P rows of 128 bytes, the MN-major SWIZZLE_128B layout (channels along M or N,
// pixels along K).
//
// Pixels (K).  The output pixels are walked in rows of Wp = Wo + ext columns, dy being zero
// (out of its bounds) in the ext extra ones, and x in rows of the same pitch (its im2col walk
// starts pad columns early and runs Wp wide).  Filter tap (dh, dw) of the pixel at position m
// then reads x's position m + dw of the walk shifted by dh rows, so ONE box of P + ext
// positions serves every dw of a tap row: the taps are row offsets of the MMA's A descriptor
// (the swizzle applies to absolute addresses, so any 128-byte row may start an operand).
// Boxes of any P tile the walk without regard to image rows; the padding is ext columns of
// Wp.  A box per tap instead reads x once per tap, and the L2-to-SM traffic, about 35 bytes
// per clock and SM, set the pace (37 us, now 31 us, for 64 -> 64 channels, 128 images of
// 32 x 32; 25 and 17 us for 128 -> 128, 32 of 28 x 28; 199 and 183 us for 256 -> 256, 64 of
// 56 x 56).
// Stride 2: x is seen as four tensors, one per parity (a, b) of the input row and column, each
// with its own map; tap dh reads row ho + floor((dh - pad) / 2) of the maps with
// a = (dh - pad) mod 2, so the dw of one parity share a box (slot), two slots per tap row.
//
// M, N.  A "unit" is one tap's window of one 64-channel chunk of x; A stacks two units to
// M = 128 (leading byte offset = the distance between their windows), B holds ncols / 64 boxes
// of dy, N = ncols.  A CTA owns nch chunks x ndh tap rows x ndw taps of a row, an accumulator
// of ncols fp32 TMEM columns per pair of units, one ncols-wide group of output channels and a
// contiguous range of pixel blocks (split K); its epilogue folds the 16 blocks into the
// letters and adds them to the fp32 outputs with atomics (zeroed before the launch).
// Separable form (Eq. 7, gradient Eq. 10): y_m = sum_p S[m][p] W_p conv x_p, so block
// (m, p) goes to letter p with Eq. 7's sign S[m][p] instead (the same 16 blocks: the
// product computes the 12 cross-component blocks the separable form does not use).

namespace dwk {

constexpr int THREADS = 256;  // warp 1 MMA issuer, warp 2 TMEM owner,
constexpr int EPI_WARP0 = 4;  // warps 4-7 epilogue (TMEM lane quarters 0-3)
// Every warp but the issuer produces: box k of a stage is loaded by producer k mod 7.  A TMA
// instruction costs its thread 0.1-0.25 us, so one producing thread set the pace (92 us
// for both gradients of the 64 -> 64 layer, 56 with seven).
constexpr int PRODUCERS = 7;
constexpr int MAX_STAGES = 4;
constexpr int MAX_PAIRS = 8;  // 512 TMEM columns at ncols = 64
constexpr int BOX_ROW = 128;  // bytes of one pixel's 64 channels
constexpr int BAR_BYTES = 256;

// Tensor maps of x: [0] for stride 1; [2 a + b] for stride 2, parity (a, b) of the input row
// and column.
struct DwMaps {
    CUtensorMap x[4];
};

struct DwParams {
    int N, Ho, Wo, Qin, Qout, kh, kw, pad, taps;
    int stride;              // 1 or 2 (four parity maps of x)
    int lone;                // stride 2: bit 0 (1) set when x has one row (column), so that
                             // the odd parity's map is empty and its boxes are zero
    int Wp;                  // columns of the pixel walk: Wo + ext
    int P;                   // pixels per block, a multiple of 16
    int org;                 // floor(-pad / stride): first row and column of x's walk
    long long kblocks;       // ceil(N Ho Wp / P)
    int nxc;                 // 64-channel chunks of x
    int nch, ndh, ndw;       // chunks, tap rows and taps of a row per CTA
    int slots;               // boxes per chunk and tap row: min(stride, ndw)
    int n0;                  // taps in slot 0: ceil(ndw / slots)
    int units, npairs;       // nch ndh ndw, and its half rounded up
    int gch, gdh, gdw;       // groups of each
    int nx;                  // x boxes per stage: nch ndh slots
    int ncols, nyb;          // output channels per CTA (N of each MMA); dy boxes per stage
    int groups, splits, stages;
    int sep;                 // 1: fold for the separable form
    int producers;           // TMA-issuing threads: min(PRODUCERS, nx + nyb)
    uint32_t tmem_cols;
    uint32_t xbox_bytes, xbox_stride;  // (P + n0 - 1) rows; from box to box, 1 KB multiples
    uint32_t ybox_bytes;
    uint32_t stage_bytes;
    unsigned long long wait_limit_ns;
    float* dwr;
    float* dwi;
    float* dwj;
    float* dwk;
};

// Tap t of a CTA's tap-row share starting at w0: its filter column, box slot and box row.  The
// taps of one column parity come first (stride 2), so windows of successive t lie at
// increasing addresses.
__device__ __forceinline__ void dw_tap(const DwParams& p, int w0, int t, int& dw, int& slot,
                                       int& row) {
    slot = t >= p.n0 ? 1 : 0;
    row = t - slot * p.n0;
    dw = w0 + slot + p.slots * row;
}

// Shared-memory descriptor, low word, with a leading byte offset: for MN-major swizzled
// tiles it is the distance between successive 64-element (128-byte) groups along M or N.
__device__ __forceinline__ uint32_t desc_lo_lbo(uint32_t saddr, uint32_t lbo_bytes) {
    return ((saddr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16);
}

// kind::f16 instruction descriptor with both operands MN-major (transpose bits 15, 16).
__host__ __device__ constexpr uint32_t make_idesc_mn(int M, int N) {
    return make_idesc(M, N, 0) | (1u << 15) | (1u << 16);
}

__device__ __forceinline__ float* letter_ptr(const DwParams& p, int L) {
    return L == 0 ? p.dwr : (L == 1 ? p.dwi : (L == 2 ? p.dwj : p.dwk));
}

__global__ void __launch_bounds__(THREADS, 1)
    qconv_dw_kernel(const __grid_constant__ DwMaps tmaps,
                    const __grid_constant__ CUtensorMap tmap_dy, const DwParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const uint32_t sbase = smem_u32(smem);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.stages * p.stage_bytes);
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (MAX_STAGES + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * MAX_STAGES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_STAGES + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint64_t limit = p.wait_limit_ns;
    // CTA -> (unit-pair group, output-channel group, K split); CTAs of one split are
    // adjacent in launch order, so they read the same pixel rows at about the same time
    int g = static_cast<int>(blockIdx.x) % p.groups;
    const int split = static_cast<int>(blockIdx.x) / p.groups;
    const int ch0 = g % p.gch * p.nch;  // first chunk, tap row, tap of the row
    g /= p.gch;
    const int dh0 = g % p.gdh * p.ndh;
    g /= p.gdh;
    const int dw0 = g % p.gdw * p.ndw;
    const int cg = g / p.gdw;           // output-channel group
    const long long kb_begin = p.kblocks * split / p.splits;
    const long long kb_end = p.kblocks * (split + 1) / p.splits;

    griddep_launch_dependents();
    if (threadIdx.x == 0) {
        for (int i = 0; i < p.stages; ++i) {
            mbar_init(full_bar(i), p.producers);
            mbar_init(empty_bar(i), 1);
        }
        mbar_init(done_bar, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0 && lane == 0) {
        for (int i = 0; i < (p.stride == 1 ? 1 : 4); ++i) tma_prefetch_desc(&tmaps.x[i]);
        tma_prefetch_desc(&tmap_dy);
    }
    if (warp == 2) {
        tmem_alloc(smem_u32(tmem_slot), p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    griddep_wait();  // x and dy complete, the zeroed outputs visible

    if (warp != 1) {
        // ---------------------------------------------------------------- TMA producers
        const int me = warp == 0 ? 0 : warp - 1;  // 0 .. PRODUCERS - 1
        if (lane == 0 && me < p.producers) {
            const uint64_t pol = l2_policy_evict_normal();
            const int boxes = p.nx + p.nyb;
            uint32_t tx = 0;
            for (int k = me; k < boxes; k += p.producers)
                tx += k < p.nx ? p.xbox_bytes : p.ybox_bytes;
            const int hw = p.Ho * p.Wp;
            uint32_t filled = 0, fill_parity = 0;
            bool ok = true;
            int stage = 0;
            uint32_t phase = 0;
            for (long long kb = kb_begin; kb < kb_end; ++kb) {
                if (!wait_or_abort(empty_bar(stage), phase ^ 1u, limit, abort_flag,
                                   STATUS_TIMEOUT_PRODUCER)) {
                    ok = false;
                    break;
                }
                const long long m0 = kb * p.P;
                const int n = static_cast<int>(m0 / hw);
                const int rem = static_cast<int>(m0 - static_cast<long long>(n) * hw);
                const int h = rem / p.Wp, w = rem - h * p.Wp;
                const uint32_t fb = full_bar(stage);
                mbar_arrive_expect_tx(fb, tx);
                filled |= 1u << stage;
                fill_parity = (fill_parity & ~(1u << stage)) | (phase << stage);
                const uint32_t dst = sbase + stage * p.stage_bytes;
                for (int k = me; k < boxes; k += p.producers) {
                    if (k >= p.nx) {  // dy
                        const int c = k - p.nx;
                        tma_load_im2col_4d(dst + p.nx * p.xbox_stride + c * p.ybox_bytes, &tmap_dy,
                                           fb, cg * p.ncols + c * 64, w, h, n, 0, 0, pol);
                        continue;
                    }
                    // box (chunk, tap row, slot); past the last of each: the last once more
                    const int slot = k % p.slots, cd = k / p.slots;
                    int dh = dh0 + cd % p.ndh, xc = ch0 + cd / p.ndh, dw = dw0 + slot;
                    if (dh >= p.kh) dh = p.kh - 1;
                    if (xc >= p.nxc) xc = p.nxc - 1;
                    if (dw >= p.kw) dw = p.kw - 1;
                    int oh = dh, ow = dw, map = 0, img = n;
                    if (p.stride == 2) {
                        const int th = dh - p.pad, tw = dw - p.pad;
                        map = 2 * (th & 1) + (tw & 1);
                        oh = (th >> 1) - p.org;
                        ow = (tw >> 1) - p.org;
                        // an empty parity class: a box past the last image, zero-filled
                        if (((th & 1) && (p.lone & 1)) || ((tw & 1) && (p.lone & 2))) img = p.N;
                    }
                    tma_load_im2col_4d(dst + k * p.xbox_stride, &tmaps.x[map], fb, xc * 64,
                                       w + p.org, h + p.org, img, static_cast<uint16_t>(ow),
                                       static_cast<uint16_t>(oh), pol);
                }
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (!ok || *abort_flag)
                drain_fills(full_bar(0), p.stages, filled, fill_parity, limit);
        }
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = make_idesc_mn(128, p.ncols);
            const uint32_t hi = desc_hi(1024, 2);  // 8-pixel groups 1024 bytes apart, SW128
            const uint32_t ksteps = static_cast<uint32_t>(p.P) / 16;
            // descriptor low words, relative to a stage, of every unit pair's first K step
            uint32_t a_off[MAX_PAIRS];
#pragma unroll
            for (int a = 0; a < MAX_PAIRS; ++a) {
                uint32_t at[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    int u = 2 * a + i;
                    if (u >= p.units) u = p.units - 1;  // odd unit count: repeat the last
                    const int cd = u / p.ndw;
                    int dw, slot, row;
                    dw_tap(p, dw0, u - cd * p.ndw, dw, slot, row);
                    at[i] = static_cast<uint32_t>(cd * p.slots + slot) * p.xbox_stride +
                            static_cast<uint32_t>(row) * BOX_ROW;
                }
                a_off[a] = (at[0] >> 4) | ((at[1] - at[0]) >> 4 << 16);
            }
            int stage = 0;
            uint32_t phase = 0;
            bool first = true;
            for (long long kb = kb_begin; kb < kb_end; ++kb) {
                if (!wait_or_abort(full_bar(stage), phase, limit, abort_flag, STATUS_TIMEOUT_MMA))
                    break;
                tc_fence_after();
                const uint32_t a0 = (sbase + stage * p.stage_bytes) >> 4;
                const uint32_t b0 = sbase + stage * p.stage_bytes + p.nx * p.xbox_stride;
                for (uint32_t j = 0; j < ksteps; ++j) {
                    const uint32_t b_lo = desc_lo_lbo(b0 + j * 2048u, p.ybox_bytes);
#pragma unroll
                    for (int a = 0; a < MAX_PAIRS; ++a) {
                        if (a >= p.npairs) break;
                        umma_f16_w(tmem_base + static_cast<uint32_t>(a * p.ncols),
                                   a_off[a] + a0 + j * 128u, hi, b_lo, hi, idesc, first ? 0u : 1u);
                    }
                    first = false;
                }
                umma_commit(empty_bar(stage));
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            // arrives once every MMA issued above has completed (also after an abort, so
            // the teardown can wait for them before TMEM is released)
            umma_commit(done_bar);
        }
    }
    if (warp >= EPI_WARP0) {
        // ---------------------------------------------------------------- epilogue
        const int q = warp - EPI_WARP0;  // TMEM lane quarter
        const bool ok = wait_or_abort(done_bar, 0, limit, abort_flag, STATUS_TIMEOUT_EPILOGUE);
        tc_fence_after();
        if (ok && !*abort_flag) {
            const int row = 32 * q + lane;  // x channel within the unit pair
            const long long wstride = static_cast<long long>(p.taps) * p.Qin;  // one co step
            for (int a = 0; a < p.npairs; ++a) {
                const int u = 2 * a + row / 64;
                const int cd = u / p.ndw;
                int dw, slot, trow;
                dw_tap(p, dw0, u - cd * p.ndw, dw, slot, trow);
                const int dh = dh0 + cd % p.ndh, xc = ch0 + cd / p.ndh;
                // (a repeated unit or one past the filter or the channels is not written)
                const bool live = u < p.units && dh < p.kh && dw < p.kw && xc < p.nxc;
                const int tap = dh * p.kw + dw;
                const int c = (live ? xc : 0) * 64 + row % 64;
                const int pc = c / p.Qin, ci = c - pc * p.Qin;
                const long long row_off = static_cast<long long>(tap) * p.Qin + ci;
                for (int j0 = 0; j0 < p.ncols; j0 += 32) {
                    uint32_t v[32];
                    tmem_ld_32x32b_x32(
                        tmem_base + (static_cast<uint32_t>(32 * q) << 16) +
                            static_cast<uint32_t>(a * p.ncols + j0),
                        v);
                    tmem_ld_wait();
                    if (!live) continue;
                    // 16 columns never straddle two output components (Qout is a multiple
                    // of 16): letter, sign and base address are fixed per half
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int d0 = cg * p.ncols + j0 + 16 * h;
                        const int m = d0 / p.Qout, co0 = d0 - m * p.Qout;
                        const bool neg = ((p.sep ? SEP_NEG : NEG_MASK) >> (4 * m + pc)) & 1u;
                        float* dst = letter_ptr(p, p.sep ? pc : (m ^ pc)) + co0 * wstride + row_off;
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) {
                            const float val = __uint_as_float(v[16 * h + jj]);
                            atomicAdd(dst + jj * wstride, neg ? -val : val);
                        }
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        // the issuer's last commit covers every MMA it issued: wait for it (bounded) so no
        // MMA still writes the accumulators when they are released
        if (lane == 0) {
            const uint64_t t0 = global_timer_ns();
            while (!mbar_try_wait(done_bar, 0u)) {
                if (global_timer_ns() - t0 > limit) {
                    atomicOr(&g_status, STATUS_TIMEOUT_DRAIN);
                    break;
                }
            }
        }
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, p.tmem_cols);
    }
}

}  // namespace dwk
