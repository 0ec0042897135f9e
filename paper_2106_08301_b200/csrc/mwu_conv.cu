// mwu_conv_implicit_ws and mwu_conv_dense: the convolution over operands laid out once per call in the
// caller's workspace.
//
//   conv_prep_kernel      one launch, two jobs side by side.  The image becomes a line of pixels, 64 channels of
//                         a pixel to a 128-byte row, with enough zero pixels between image rows and images that
//                         a tap never reaches into a neighbour.  The weights (packed records, or a plain matrix)
//                         get a tap-major reduction axis: column (i*kw + j) * cin + c instead of c * kh*kw + i*kw + j.
//   mwu_conv_line_kernel  for every tap the activation operand of 128 consecutive pixels of the line is 128 rows
//                         of it, shifted by a constant.  So a CTA fetches a tile's rows with their halo once per 64
//                         channels (plain TMA boxes), and every tap's MMAs read them through a descriptor that
//                         starts the tap's shift further on; the weights arrive as one 128 x 64 box per tap.
//                         Fetching a box per tap instead (the image nine times) bound the kernel: 576 KB from L2
//                         for a tile of 112 pixels and 18 taps x chunks, against 360 KB for 256 pixels.
// Roles (11 warps): warp 0 fetches halo rows, warp 10 weights, warp 1 owns tensor memory and issues the MMAs
// (128 x 128 x 16; a tile of 256 pixels is two accumulators that share every weight box), warps 2-9 store NCHW
// output (a tensor-memory lane is a pixel).  Accumulators are double-buffered.
// Every wait on an mbarrier is bounded; when one runs out the kernel raises MWU_DEV_TIMEOUT, waits
// for the loads it has in flight, frees its tensor memory and returns.
#include "mwu_gemm_dev.cuh"

namespace mwu {
namespace gemm {

EncodeTiledFn get_encode_fn();          // mwu_gemm.cu

constexpr int L_THREADS = 32 * 11;
constexpr int L_B_WARP = 10;
constexpr int L_MAX_STAGES = 8;         // weight boxes in flight
constexpr int L_SMEM = 227 * 1024;

struct ConvParams {
    Params g;                           // packed weights, N = filters, K = cin*kh*kw, Y, y_fp32, dev_status
    int C, H, W, KH, KW, pad, OH, OW, NIMG;
    int Hp, Wp, shift;                  // the line of pixels: image rows, pitch, and how far the taps start before a pixel
    long long M;                        // its pixels: NIMG * Hp * Wp
    unsigned img_magic, row_magic;
    int tm;                             // pixels of a tile: 128 or 256
    int fetches;                        // fetches of a tile and 64 channels: one for all taps, one per kernel row, or one per tap
    int a_rows, a_bufs, box_rows;       // rows of a fetch, buffers, rows of a TMA box
    int b_stages;
    int n_ntiles;                       // 128-filter tiles
    long long wait_limit;               // cycles a wait may take
    long long withhold;                 // testing aid: running number of a weight box that is left out (-1: none)
};

struct ConvSmem {
    unsigned long long a_full[2], a_empty[2], b_full[L_MAX_STAGES], b_empty[L_MAX_STAGES], tfull[2], tempty[2], drain;
    unsigned tmem_base;
    int abort;
    int no_abort;
};

// Bounded wait with this kernel's own limit.  The producers and the MMA issuer poll for a while (a waiter
// suspended in try_wait wakes a few hundred cycles late, once per 64 x 128 step), the others sleep at once.
template <bool POLL>
__device__ __forceinline__ bool mbar_wait_lim(unsigned bar, unsigned parity, volatile int *abort, long long limit) {
#pragma unroll 1
    for (int i = 0; i < (POLL ? 4096 : 1); ++i)
        if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
#pragma unroll 1
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort) return false;
        if (clock64() - t0 > limit) { *abort = 1; return false; }
    }
}

// n / d for n < 2^31, with m = floor(2^32 / d) + 1: the product's high word is the quotient or one too many
__device__ __forceinline__ unsigned line_divide(unsigned n, unsigned d, unsigned m, unsigned *rem) {
    unsigned q = d == 1u ? n : __umulhi(n, m);
    unsigned r = n - q * d;
    if ((int)r < 0) { --q; r += d; }
    *rem = r;
    return q;
}
// (image, row, column) of a pixel of the line
__device__ __forceinline__ void line_pixel(const ConvParams &p, unsigned P, int *img, int *y, int *x) {
    unsigned rem, col;
    *img = (int)line_divide(P, (unsigned)p.Hp * (unsigned)p.Wp, p.img_magic, &rem);
    *y = (int)line_divide(rem, (unsigned)p.Wp, p.row_magic, &col);
    *x = (int)col;
}

// ------------------------------------------------------------------------------------------
// preparation
// ------------------------------------------------------------------------------------------
constexpr int PREP_THREADS = 256;

// a warp: 32 pixels x 16 channels, read along the image rows, written as 32 bytes of each pixel's row
__device__ __forceinline__ void image_to_line(const ConvParams &p, const unsigned short *x, unsigned short *xt, long long task) {
    const int lane = threadIdx.x & 31;
    const unsigned n_c = (unsigned)p.C / 16u;
    const long long pix0 = (task / n_c) * 32;
    const int c0 = (int)(task % n_c) * 16;
    const long long P = pix0 + lane;
    if (P >= p.M) return;
    int img, y, xx;
    line_pixel(p, (unsigned)P, &img, &y, &xx);
    y -= p.pad - p.shift;                                   // shift: zero pixels follow an image row, else they surround it
    xx -= p.pad - p.shift;
    const bool in = (unsigned)y < (unsigned)p.H && (unsigned)xx < (unsigned)p.W;
    const long long plane = (long long)p.H * p.W;
    const unsigned short *src = x + ((long long)img * p.C + c0) * plane + (in ? y * p.W + xx : 0);
    unsigned v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = in ? (unsigned)__ldg(src + e * plane) : 0u;
    uint4 *dst = reinterpret_cast<uint4 *>(xt + P * p.C + c0);
    dst[0] = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
    dst[1] = make_uint4(v[8] | (v[9] << 16), v[10] | (v[11] << 16), v[12] | (v[13] << 16), v[14] | (v[15] << 16));
}

// a packed 128 x 64 record -> tap-major rows; `part` of `parts` CTAs that decode it alike and write its share of rows
// (the 2-byte stores take longer than the decoding)
template <int BW>
__device__ __forceinline__ void record_to_taps(const Params &p, unsigned short *Wd, int taps, int C, long long rec, int part, int parts) {
    __shared__ __align__(1024) unsigned char tile[REC_BYTES];
    constexpr int ENT = DecodeCfg<BW, PREP_THREADS>::ENT;
    const PackedRec *recs = reinterpret_cast<const PackedRec *>(p.packed + p.off_rec);
    const long long rt = rec / p.n_stages, ks = rec % p.n_stages;
    const int tid = threadIdx.x;
    PackedRec r0, r1;
    {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(&recs[rec]));
        const uint4 b = __ldg(reinterpret_cast<const uint4 *>(&recs[rec + 1]));
        r0.ubase = a.x; r0.dbase = a.y; r0.pbase = a.z; r0.live = a.w;
        r1.ubase = b.x; r1.dbase = b.y; r1.pbase = b.z; r1.live = b.w;
    }
    unsigned m0[ENT], m1[ENT];
    fetch_entries<BW, PREP_THREADS>(r0, r1, p, tid, m0, m1);
    write_entries<BW, PREP_THREADS>(tile, r0, r1, p, tid, m0, m1);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // A lane writes the same two of the 64 columns in every row; the columns are dealt out by tap first, so that
    // neighbouring lanes store neighbouring channels.  (A thread writing 8 columns as they stand meets 8 taps:
    // 32 sectors a store instead of about 32 * taps / 64 + 1; 512 x 256 x 7 x 7, 3x3, n 8, b 16: 28.3 us a call, so 18.6,
    // 384 x 192 x 14 x 14, 5x5: 46.1, so 37.2.)
    const int per = BK / taps, more = BK % taps;            // the first `more` of the taps met have one channel more
    const int k0 = (int)ks * BK, lane = tid & 31, rows = kTileRows / parts;
    int src[2];
    unsigned short *dst[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int q = lane + 32 * h, q1 = q - more * (per + 1);
        const int met = q1 < 0 ? q / (per + 1) : more + q1 / per, nth = q1 < 0 ? q - met * (per + 1) : q1 % per;
        const int e = met + nth * taps, c = (k0 + e) / taps, tap = k0 + e - c * taps;
        src[h] = e;
        dst[h] = Wd + (long long)tap * C + c;
    }
#pragma unroll 4
    for (int i = tid >> 5; i < rows; i += PREP_THREADS / 32) {
        const int r = part * rows + i;
        const long long at = (rt * kTileRows + r) * p.K;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            dst[h][at] = *reinterpret_cast<const unsigned short *>(tile + r * 128 + (((src[h] >> 3) ^ (r & 7)) << 4) + (src[h] & 7) * 2);
    }
}

// CTAs [0, n_w): weights; the rest: image.  BW 0: a plain weight matrix [rows][ldw] in [c][tap] column order
template <int BW>
__global__ void __launch_bounds__(PREP_THREADS) conv_prep_kernel(const __grid_constant__ ConvParams p, const unsigned short *Wd,
                                                                 long long ldw, long long n_pad, unsigned short *wt, unsigned n_w,
                                                                 int parts, const unsigned short *x, unsigned short *xt) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the tensor-core kernel may set itself up meanwhile
    const int taps = p.KH * p.KW;
    if (blockIdx.x < n_w) {
        if constexpr (BW == 0) {
            const long long K = p.g.K, total = n_pad * K;
            for (long long i = (long long)blockIdx.x * PREP_THREADS + threadIdx.x; i < total; i += (long long)n_w * PREP_THREADS) {
                const long long row = i / K;
                const int kk = (int)(i - row * K), tap = kk / p.C, c = kk - tap * p.C;
                wt[i] = row < p.g.N ? Wd[row * ldw + (long long)c * taps + tap] : (unsigned short)0;     // rows past the last: zeros
            }
        } else {
            MWU_CHECK_HEADER(p.g);
            record_to_taps<BW>(p.g, wt, taps, p.C, blockIdx.x / (unsigned)parts, (int)(blockIdx.x % (unsigned)parts), parts);
        }
    } else {
        image_to_line(p, x, xt, (long long)(blockIdx.x - n_w) * (PREP_THREADS / 32) + (threadIdx.x >> 5));
    }
}

// ------------------------------------------------------------------------------------------
// the tensor-core kernel
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(L_THREADS, 1)
mwu_conv_line_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                     const __grid_constant__ ConvParams p) {
    if (!p.g.all_live) MWU_CHECK_HEADER(p.g);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sA = smem_raw + smem_pad_1024(smem_raw);
    const unsigned a_bytes = (unsigned)p.a_rows * 128u;
    unsigned char *sB = sA + (size_t)p.a_bufs * a_bytes;
    __shared__ ConvSmem sm_;
    ConvSmem *sm = &sm_;
    volatile int *abort = &sm->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int chunks = p.C / BK;                            // of 64 channels
    const int fetches = p.fetches, taps_per = p.KH * p.KW / fetches;
    const int m_tiles = (int)((p.M + p.tm - 1) / p.tm);
    const long long total_tiles = (long long)m_tiles * p.n_ntiles;
    const long long limit = p.wait_limit;
    const int halves = p.tm / 128;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sm->a_full[b]), 1);
            mbar_init(smem_u32(&sm->a_empty[b]), 1);
            mbar_init(smem_u32(&sm->tfull[b]), 1);
            mbar_init(smem_u32(&sm->tempty[b]), 8);
        }
        for (int s = 0; s < L_MAX_STAGES; ++s) {
            mbar_init(smem_u32(&sm->b_full[s]), 1);
            mbar_init(smem_u32(&sm->b_empty[s]), 1);
        }
        mbar_init(smem_u32(&sm->drain), 1);
        sm->abort = 0;
        sm->no_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) tmem_alloc(smem_u32(&sm->tmem_base), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // launched with programmatic stream serialization: the set-up above ran while the kernel that
    // prepares the operands was still finishing; its memory is complete from here on
    // No trigger for the kernel behind: its small CTAs would crowd, eight to an SM, on the SMs that have no tile, and
    // run there while the others stand idle (384 x 192 x 14 x 14, 5x5, n 16, call after call: 82 us with it, 48 without).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const unsigned tmem_base = *reinterpret_cast<volatile unsigned *>(&sm->tmem_base);

    // The three roles below are one thread each: a step then holds no warp vote or barrier (a quarter of a 128 x 128
    // step's time), and a wait that runs out leaves no other lane behind.
    if (warp == 0) {
        // ---------------- halo rows ----------------
        if (elect_one()) {
            unsigned buf = 0, phase = 0, issued = 0, last_phase = 0;
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < total_tiles; t += gridDim.x) {
                const int p0 = (int)(t / p.n_ntiles) * p.tm;
                for (int f = 0; f < chunks * fetches; ++f) {
                    const int chunk = f / fetches, part = f - chunk * fetches;
                    ok = mbar_wait_lim<true>(smem_u32(&sm->a_empty[buf]), phase ^ 1u, abort, limit);
                    if (!ok) break;
                    const unsigned bar = smem_u32(&sm->a_full[buf]);
                    mbar_expect_tx(bar, a_bytes);
                    // a box may start before the first pixel or end after the last: zeros there
                    const int first = fetches > p.KH ? part / p.KW * p.Wp + part % p.KW : part * p.Wp;      // its first tap's shift
                    const int row = p0 - p.shift * (p.Wp + 1) + first;
                    for (int b = 0; b * p.box_rows < p.a_rows; ++b)
                        tma_load_2d(smem_u32(sA + buf * a_bytes + (unsigned)(b * p.box_rows) * 128u), &tmap_x, bar, chunk * BK,
                                    row + b * p.box_rows);
                    issued |= 1u << buf;
                    last_phase = (last_phase & ~(1u << buf)) | (phase << buf);
                    if (++buf == (unsigned)p.a_bufs) { buf = 0; phase ^= 1u; }
                }
            }
            // leaving early: the loads already issued must have landed before the CTA goes away.  Their
            // barriers need nothing but the loads' own bytes, so these waits end (and are bounded anyway).
            if (!ok)
                for (int b = 0; b < 2; ++b)
                    if ((issued >> b) & 1u) mbar_wait_lim<true>(smem_u32(&sm->a_full[b]), (last_phase >> b) & 1u, &sm->no_abort, limit);
        }
        __syncwarp();
    } else if (warp == L_B_WARP) {
        // ---------------- weights ----------------
        if (elect_one()) {
            unsigned stage = 0, phase = 0, issued = 0, last_phase = 0;
            long long seq = 0;                              // boxes so far
            bool ok = true;
            for (long long t = blockIdx.x; ok && t < total_tiles; t += gridDim.x) {
                const int nt = (int)(t % p.n_ntiles);
                for (int f = 0; ok && f < chunks * fetches; ++f) {
                    const int chunk = f / fetches, tap0 = (f - chunk * fetches) * taps_per;
                    for (int q = 0; q < taps_per; ++q) {
                        ok = mbar_wait_lim<true>(smem_u32(&sm->b_empty[stage]), phase ^ 1u, abort, limit);
                        if (!ok) break;
                        if (seq++ != p.withhold) {
                            const unsigned bar = smem_u32(&sm->b_full[stage]);
                            mbar_expect_tx(bar, REC_BYTES);
                            tma_load_2d(smem_u32(sB + stage * REC_BYTES), &tmap_w, bar, (tap0 + q) * p.C + chunk * BK, nt * kTileRows);
                            issued |= 1u << stage;
                            last_phase = (last_phase & ~(1u << stage)) | (phase << stage);
                        }
                        if (++stage == (unsigned)p.b_stages) { stage = 0; phase ^= 1u; }
                    }
                }
            }
            if (!ok)
                for (int s = 0; s < p.b_stages; ++s)
                    if ((issued >> s) & 1u) mbar_wait_lim<true>(smem_u32(&sm->b_full[s]), (last_phase >> s) & 1u, &sm->no_abort, limit);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (elect_one()) {
            unsigned buf = 0, a_phase = 0, stage = 0, b_phase = 0;
            bool ok = true, issued_any = false;
            const unsigned idesc = make_idesc(128);
            long long k = 0;
            for (long long t = blockIdx.x; ok && t < total_tiles; t += gridDim.x, ++k) {
                const unsigned acc = (unsigned)(k & 1), use_phase = (unsigned)((k >> 1) & 1);
                ok = mbar_wait_lim<true>(smem_u32(&sm->tempty[acc]), use_phase ^ 1u, abort, limit);
                if (!ok) break;
                tc_fence_after();
                const unsigned d = tmem_base + acc * 256u;
                for (int f = 0; f < chunks * fetches; ++f) {
                    ok = mbar_wait_lim<true>(smem_u32(&sm->a_full[buf]), a_phase, abort, limit);
                    if (!ok) break;
                    const unsigned a_s = smem_u32(sA + buf * a_bytes);
                    int i = 0, j = 0;
                    for (int q = 0; q < taps_per; ++q) {
                        ok = mbar_wait_lim<true>(smem_u32(&sm->b_full[stage]), b_phase, abort, limit);
                        if (!ok) break;
                        tc_fence_after();
                        const unsigned long long bdesc = make_desc(smem_u32(sB + stage * REC_BYTES));
                        const unsigned long long adesc = make_desc(a_s + (unsigned)(i * p.Wp + j) * 128u);
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4)
                            umma_bf16(d, adesc + (unsigned long long)(k4 * 2), bdesc + (unsigned long long)(k4 * 2), idesc,
                                      (f | q | k4) ? 1u : 0u);
                        if (halves == 2) {
#pragma unroll
                            for (int k4 = 0; k4 < 4; ++k4)
                                umma_bf16(d + 128u, adesc + (unsigned long long)((128 * 128 >> 4) + k4 * 2),
                                          bdesc + (unsigned long long)(k4 * 2), idesc, (f | q | k4) ? 1u : 0u);
                        }
                        umma_commit(smem_u32(&sm->b_empty[stage]));
                        issued_any = true;
                        if (++j == p.KW) { j = 0; ++i; }
                        if (++stage == (unsigned)p.b_stages) { stage = 0; b_phase ^= 1u; }
                    }
                    if (!ok) break;
                    umma_commit(smem_u32(&sm->a_empty[buf]));
                    if (++buf == (unsigned)p.a_bufs) { buf = 0; a_phase ^= 1u; }
                }
                if (ok) umma_commit(smem_u32(&sm->tfull[acc]));
            }
            // everything issued must have retired before tensor memory is freed
            if (issued_any) {
                umma_commit(smem_u32(&sm->drain));
                mbar_wait_lim<true>(smem_u32(&sm->drain), 0, &sm->no_abort, limit);
            }
        }
        __syncwarp();
    } else {
        // ---------------- output: tensor-memory lanes are pixels, columns are filters ----------------
        const int quarter = warp & 3, second = (warp - 2) >> 2;
        // two warps to a quarter: a half of the pixels each, or of the filters
        const int half = halves == 2 ? second : 0, c_from = halves == 2 ? 0 : second * 64, c_to = halves == 2 ? 128 : c_from + 64;
        bool ok = true;
        long long k = 0;
        const long long plane = (long long)p.OH * p.OW;
        for (long long t = blockIdx.x; ok && t < total_tiles; t += gridDim.x, ++k) {
            const long long nt = t % p.n_ntiles, P = (t / p.n_ntiles) * p.tm + half * 128 + quarter * 32 + lane;
            const unsigned acc = (unsigned)(k & 1), use_phase = (unsigned)((k >> 1) & 1);
            int img = 0, oh = 0, ow = 0;
            bool px = P < p.M;
            if (px) {
                line_pixel(p, (unsigned)P, &img, &oh, &ow);
                px = oh < p.OH && ow < p.OW;                // the others are zero pixels
            }
            if (!mbar_wait_lim<false>(smem_u32(&sm->tfull[acc]), use_phase, abort, limit)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const unsigned trow = tmem_base + ((unsigned)(quarter * 32) << 16) + acc * 256u + (unsigned)half * 128u;
#pragma unroll 1
            for (int c0 = c_from; c0 < c_to; c0 += 32) {
                const long long o0 = nt * kTileRows + c0;
                if (o0 >= p.g.N) break;
                unsigned v[32];
                tmem_ld32(trow + (unsigned)c0, v);
                const long long at = (img * p.g.N + o0) * plane + (long long)oh * p.OW + ow;
                if (px) {
                    if (p.g.y_fp32) {
                        float *dst = reinterpret_cast<float *>(p.g.Y) + at;
#pragma unroll
                        for (int j = 0; j < 32; ++j, dst += plane)
                            if (o0 + j < p.g.N) *dst = __uint_as_float(v[j]);
                    } else {
                        __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(p.g.Y) + at;
#pragma unroll
                        for (int j = 0; j < 32; ++j, dst += plane)
                            if (o0 + j < p.g.N) *dst = __float2bfloat16_rn(__uint_as_float(v[j]));
                    }
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sm->tempty[acc]));
        }
    }

    // teardown
    tc_fence_before();
    __syncthreads();
    // after the barrier: a role that finished its own work early must still see a flag raised later
    if (*abort && threadIdx.x == 0) atomicOr(p.g.dev_status, (unsigned)MWU_DEV_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------
// testing aid (see mwu.h): limit of the bounded waits and a weight box to leave out
static long long g_wait_limit = WAIT_LIMIT_CYCLES;
static long long g_withhold = -1;

// shapes this path serves: stride 1, channels in chunks of 64, at most 128 output pixels per row
static bool line_shape(int n, int c, int h, int w, int kh, int kw, int stride, int pad) {
    if (n <= 0 || c <= 0 || h <= 0 || w <= 0 || kh <= 0 || kw <= 0 || stride != 1 || pad < 0) return false;
    if (c % BK != 0 || h + 2 * pad < kh || w + 2 * pad < kw || pad > 32767) return false;
    return w + 2 * pad - kw + 1 <= 128 && w <= 65535 && h <= 65535;
}

// The line of pixels.  With pad < kernel a run of `pad` zero pixels after every image row and `pad` such rows after
// every image serve both neighbours; a wider padding is laid out in full.
static void line_of(int n, int h, int w, int kh, int kw, int pad, int *Hp, int *Wp, int *shift, long long *M) {
    const bool shared = pad < kh && pad < kw;
    *Hp = h + (shared ? pad : 2 * pad);
    *Wp = w + (shared ? pad : 2 * pad);
    *shift = shared ? pad : 0;
    *M = (long long)n * *Hp * *Wp;
}
static size_t line_bytes(int n, int c, int h, int w, int kh, int kw, int pad) {
    int Hp, Wp, shift;
    long long M;
    line_of(n, h, w, kh, kw, pad, &Hp, &Wp, &shift, &M);
    return align_up((size_t)M * c * 2, 1024);
}
static size_t conv_workspace(int64_t rows, int n, int c, int h, int w, int kh, int kw, int pad) {
    const int64_t n_pad = (rows + kTileRows - 1) / kTileRows * kTileRows;
    return line_bytes(n, c, h, w, kh, kw, pad) + (size_t)n_pad * (size_t)c * kh * kw * 2;
}

// p.g is filled; bw 0: plain weights Wd
static int run_line(ConvParams &p, int bw, const void *Wd, long long ldw, const void *X_nchw, int n, int c, int h, int w, int kh,
                    int kw, int pad, void *workspace, int sm_count, cudaStream_t st) {
    EncodeTiledFn encode = get_encode_fn();
    if (!encode) return MWU_ERR_CUDA;
    p.C = c; p.H = h; p.W = w; p.KH = kh; p.KW = kw; p.pad = pad; p.NIMG = n;
    p.OH = h + 2 * pad - kh + 1;
    p.OW = w + 2 * pad - kw + 1;
    line_of(n, h, w, kh, kw, pad, &p.Hp, &p.Wp, &p.shift, &p.M);
    if (p.M + 256 >= (1ll << 31)) return MWU_ERR_SHAPE;
    p.img_magic = (unsigned)((1ull << 32) / ((unsigned)p.Hp * (unsigned)p.Wp)) + 1u;
    p.row_magic = (unsigned)((1ull << 32) / (unsigned)p.Wp) + 1u;
    const int64_t n_pad = (p.g.N + kTileRows - 1) / kTileRows * kTileRows;
    p.n_ntiles = (int)(n_pad / kTileRows);
    p.wait_limit = g_wait_limit;
    p.withhold = g_withhold;
    // Tiles of 256 pixels share a weight box between two accumulators; of 128 where those would leave SMs idle.
    // All taps from one fetch where two buffers of it fit beside four weight boxes, else a fetch per kernel row, and for
    // kernels too wide for that (some 1300 columns) one per tap.
    const long long room = L_SMEM - 2048;
    p.tm = (p.M + 255) / 256 * p.n_ntiles * 10 >= 6ll * sm_count ? 256 : 128;
    for (const int fetches : {1, kh, kh * kw}) {
        const long long rows = p.tm + (fetches > 1 ? 0 : (long long)(kh - 1) * p.Wp) + (fetches > kh ? 0 : kw - 1);
        p.fetches = fetches;
        const long long boxes = (rows + 255) / 256;
        p.box_rows = (int)(((rows + boxes - 1) / boxes + 7) / 8 * 8);
        const long long a_rows = boxes * p.box_rows;
        p.a_bufs = a_rows * 256 + 4 * REC_BYTES <= room ? 2 : 1;
        const long long left = room - p.a_bufs * a_rows * 128;
        p.a_rows = (int)a_rows;
        p.b_stages = left / REC_BYTES > L_MAX_STAGES ? L_MAX_STAGES : (int)(left / REC_BYTES);
        if (left >= 2 * REC_BYTES) break;
    }
    unsigned short *xt = (unsigned short *)workspace;
    unsigned short *wt = (unsigned short *)((char *)workspace + line_bytes(n, c, h, w, kh, kw, pad));
    auto map_2d = [&](CUtensorMap *tm, void *ptr, long long inner, long long outer, int rows) {
        const cuuint64_t dim[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
        const cuuint64_t str[1] = {(cuuint64_t)inner * 2};
        const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)rows};
        const cuuint32_t est[2] = {1, 1};
        return encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, dim, str, box, est, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap tmap_x, tmap_w;
    if (!map_2d(&tmap_x, xt, c, p.M, p.box_rows) || !map_2d(&tmap_w, wt, p.g.K, n_pad, kTileRows)) return MWU_ERR_CUDA;
    // weights: a record to a CTA, or to four that share its rows while the records are few
    unsigned n_w;
    int parts = 1;
    if (bw == 0) {
        const long long want = (n_pad * p.g.K + 4 * PREP_THREADS - 1) / (4 * PREP_THREADS);
        n_w = (unsigned)(want < 16ll * sm_count ? want : 16ll * sm_count);
    } else {
        const long long n_rec = p.g.n_rec_tiles * p.g.n_stages;
        while (parts < 4 && n_rec * parts * 2 <= 2ll * sm_count) parts *= 2;
        if (n_rec * parts >= (1ll << 30)) return MWU_ERR_SHAPE;
        n_w = (unsigned)(n_rec * parts);
    }
    const long long tasks = (p.M + 31) / 32 * (c / 16), img_ctas = (tasks + PREP_THREADS / 32 - 1) / (PREP_THREADS / 32);
    if (img_ctas >= (1ll << 30)) return MWU_ERR_SHAPE;
    auto prep = bw == 0 ? conv_prep_kernel<0> : bw == 2 ? conv_prep_kernel<2> : bw == 4 ? conv_prep_kernel<4>
              : bw == 8 ? conv_prep_kernel<8> : conv_prep_kernel<16>;
    count_launch(2);
    if (launch_chained(prep, dim3(n_w + (unsigned)img_ctas), dim3(PREP_THREADS), 0, st, 1, p, (const unsigned short *)Wd, ldw,
                       (long long)n_pad, wt, n_w, parts, (const unsigned short *)X_nchw, xt) != cudaSuccess)
        return MWU_ERR_CUDA;
    const size_t smem = (size_t)p.a_bufs * p.a_rows * 128 + (size_t)p.b_stages * REC_BYTES + 1024;
    if (cudaFuncSetAttribute(mwu_conv_line_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, L_SMEM - 1024) != cudaSuccess)
        return MWU_ERR_CUDA;
    const long long tiles = (p.M + p.tm - 1) / p.tm * p.n_ntiles;
    const int grid = (int)(tiles < sm_count ? tiles : sm_count);
    return launch_chained(mwu_conv_line_kernel, dim3((unsigned)grid), dim3(L_THREADS), smem, st, 1, tmap_x, tmap_w, p) == cudaSuccess
               ? MWU_OK : MWU_ERR_CUDA;
}

}  // namespace gemm
}  // namespace mwu

extern "C" void mwu_debug_conv_wait(int64_t limit_cycles, int64_t withhold_stage) {
    mwu::gemm::g_wait_limit = limit_cycles > 0 ? limit_cycles : mwu::gemm::WAIT_LIMIT_CYCLES;
    mwu::gemm::g_withhold = withhold_stage;
}

extern "C" size_t mwu_conv_workspace_bytes(const mwu_proj_desc *desc, int32_t n, int32_t c, int32_t h,
                                           int32_t w, int32_t kh, int32_t kw, int32_t stride, int32_t pad) {
    using namespace mwu;
    if (validate_desc(desc, true) != MWU_OK || !gemm::line_shape(n, c, h, w, kh, kw, stride, pad)) return 0;
    if ((int64_t)c * kh * kw != desc->cols) return 0;
    return gemm::conv_workspace(desc->rows, n, c, h, w, kh, kw, pad);
}

extern "C" int mwu_conv_implicit_ws(const mwu_proj_desc *desc, const void *packed, const void *X_nchw,
                                    int32_t n, int32_t c, int32_t h, int32_t w, int32_t kh, int32_t kw,
                                    int32_t stride, int32_t pad, void *Y_nchw, int32_t y_dtype,
                                    void *workspace, size_t workspace_bytes, uint32_t *dev_status,
                                    void *cuda_stream) {
    using namespace mwu;
    using namespace mwu::gemm;
    const size_t need = mwu_conv_workspace_bytes(desc, n, c, h, w, kh, kw, stride, pad);
    if (!workspace || need == 0 || workspace_bytes < need)
        return mwu_conv_implicit(desc, packed, X_nchw, n, c, h, w, kh, kw, stride, pad, Y_nchw, y_dtype,
                                 dev_status, cuda_stream);
    if (!packed || !X_nchw || !Y_nchw || !dev_status) return MWU_ERR_INVALID_ARG;
    if (y_dtype != 0 && y_dtype != 1) return MWU_ERR_INVALID_ARG;
    if (!aligned_to(packed, 256) || !aligned_to(X_nchw, 16) || !aligned_to(Y_nchw, 16) ||
        !aligned_to(dev_status, 4) || !aligned_to(workspace, 256))
        return MWU_ERR_ALIGNMENT;
    int sm_count = 0;
    int rc = check_device(&sm_count);
    if (rc != MWU_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;

    ConvParams p = {};
    const PackedLayout L = packed_layout(desc);
    p.g.packed = (const unsigned char *)packed;
    p.g.off_rec = L.off_rec; p.g.off_ulist = L.off_ulist; p.g.off_dpos = L.off_dpos;
    p.g.off_dpay = L.off_dpay; p.g.off_ppos = L.off_ppos;
    p.g.n_unified = (unsigned)L.n_unified; p.g.n_dense = (unsigned)L.n_dense; p.g.n_plist = (unsigned)L.n_plist;
    p.g.n_rec_tiles = L.n_tiles;
    p.g.n_stages = L.n_stages;
    p.g.N = desc->rows;
    p.g.K = desc->cols;
    p.g.bw = desc->block;
    p.g.Y = Y_nchw;
    p.g.y_fp32 = y_dtype;
    p.g.dev_status = dev_status;
    return run_line(p, desc->block, nullptr, 0, X_nchw, n, c, h, w, kh, kw, pad, workspace, sm_count, st);
}

extern "C" size_t mwu_conv_dense_workspace_bytes(int64_t rows, int32_t n, int32_t c, int32_t h, int32_t w,
                                                 int32_t kh, int32_t kw, int32_t stride, int32_t pad) {
    using namespace mwu;
    if (rows <= 0 || !gemm::line_shape(n, c, h, w, kh, kw, stride, pad)) return 0;
    return gemm::conv_workspace(rows, n, c, h, w, kh, kw, pad);
}

extern "C" int mwu_conv_dense(int64_t rows, const void *Wd, int64_t ldw, const void *X_nchw, int32_t n, int32_t c,
                              int32_t h, int32_t w, int32_t kh, int32_t kw, int32_t stride, int32_t pad,
                              void *Y_nchw, int32_t y_dtype, void *workspace, size_t workspace_bytes,
                              uint32_t *dev_status, void *cuda_stream) {
    using namespace mwu;
    using namespace mwu::gemm;
    if (!Wd || !X_nchw || !Y_nchw || !dev_status || !workspace) return MWU_ERR_INVALID_ARG;
    if (y_dtype != 0 && y_dtype != 1) return MWU_ERR_INVALID_ARG;
    const size_t need = mwu_conv_dense_workspace_bytes(rows, n, c, h, w, kh, kw, stride, pad);
    if (need == 0 || ldw < (int64_t)c * kh * kw) return MWU_ERR_SHAPE;
    if (workspace_bytes < need) return MWU_ERR_WORKSPACE;
    if (!aligned_to(Wd, 2) || !aligned_to(X_nchw, 16) || !aligned_to(Y_nchw, 16) || !aligned_to(dev_status, 4) ||
        !aligned_to(workspace, 256))
        return MWU_ERR_ALIGNMENT;
    int sm_count = 0;
    const int rc = check_device(&sm_count);
    if (rc != MWU_OK) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    ConvParams p = {};
    p.g.all_live = 1;                                   // plain weights: no packed header to compare with
    p.g.N = rows;
    p.g.K = (long long)c * kh * kw;
    p.g.Y = Y_nchw;
    p.g.y_fp32 = y_dtype;
    p.g.dev_status = dev_status;
    return run_line(p, 0, Wd, ldw, X_nchw, n, c, h, w, kh, kw, pad, workspace, sm_count, st);
}
