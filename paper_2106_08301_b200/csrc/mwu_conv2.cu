// mwu_conv_implicit for kernels of up to nine taps: one kernel from NCHW image and packed weights to NCHW
// output, any stride and padding, no scratch memory.
//
// The k x k taps of a convolution are shifts of one image.  Lay the image out as rows of 64 channels, one
// row per pixel, the pixels of all images in one line with enough zero pixels between image rows and
// between images that no tap reaches into a neighbour; then for every tap the activation operand of 128
// output pixels is 128 consecutive rows, shifted by a constant.  So a CTA brings the rows of a tile and
// its halo into shared memory once (128 + (kh-1) * row pitch + kw-1 rows, swizzled) and every tap's MMAs
// read them through a descriptor that starts the tap's shift further on.  A stride s splits the padded
// image into s x s planes, each with its own taps, halo and shifts.  No im2col row is built and the image
// is fetched about 1.5 times instead of once per tap.  (The junk rows at the zero pixels are multiplied and
// dropped: 7 % of the work at 28 x 28, 31 % at 7 x 7.)
//
// The packed records are 64 columns in [channel][tap] order, so `taps` consecutive records hold 64 channels
// of every tap.  They are decoded into as many tiles as the other kernels do, and then every row is permuted
// in place (a warp holds the whole row in registers in between) into one 128 x 64 tile per tap; once per CTA
// and chunk of 64 channels, for up to four output tiles (one accumulator each in tensor memory).
//
// Roles (17 warps): warps 0-15 decode the weights, gather the halo rows from NCHW (a lane is a pixel, eight
// channels make a 16-byte store) and store the output; warp 16 owns tensor memory and issues the MMAs.  With
// few tiles the chunks of a tile are split over a cluster, whose partial sums meet in distributed shared memory.
//
// What bounds it: latency of the gathers and the decode; the MMAs of a tile take 0.6 us.
// Every wait on an mbarrier is bounded; when one runs out the kernel raises MWU_DEV_TIMEOUT, frees its
// tensor memory and returns (its only asynchronous copies are waited for by the threads that made them).
#include "mwu_gemm_dev.cuh"

namespace mwu {
namespace gemm {

constexpr int CV_WORKERS = 16;          // warps that decode, gather and store
constexpr int CV_MMA_WARP = CV_WORKERS;
constexpr int CV_THREADS = 32 * (CV_WORKERS + 1);
constexpr int CV_WORK_THREADS = 32 * CV_WORKERS;
constexpr int CV_TILE = 128;            // output pixels of a tile
constexpr int CV_BATCH = 4;             // tiles that share one pass over the weights: accumulators of 128 columns
constexpr int CV_TAPS = 9;              // most taps: their weight tiles are all in shared memory
constexpr int CV_SMEM = 227 * 1024;

struct HaloParams {
    Params g;                           // packed weights, N = filters, K = cin*kh*kw, Y, y_fp32, dev_status
    const unsigned short *X;
    int C, H, W, KH, KW, stride, pad, OH, OW, NIMG;
    int Hp, Wp;                         // the image in the line of pixels: rows and pitch, zero pixels included
    int shared_pad;                     // zero pixels are shared by neighbouring rows and images (see halo_geometry)
    long long M;                        // pixels of the line: NIMG * Hp * Wp
    int group_mode;                     // what one gather serves: 0 all taps of a plane, 1 those of one kernel row, 2 one tap
    int a_rows, a_bufs;                 // rows of a gather buffer, and how many there are
    int chunks;                         // of 64 channels
    unsigned tmem_cols, img_magic, row_magic;
    int n_ntiles, per_ntile, split;     // 128-filter tiles; CTA groups sharing one's pixel tiles; CTAs of a cluster
};

struct HaloSmem {
    unsigned long long a_full[2], a_empty[2], w_full, w_empty, t_full, t_empty;
    int4 group[CV_TAPS];                // of every gather: see TapGroup
    int4 group2[CV_TAPS];
    uint4 rec[CV_TAPS + 1];             // record table of the chunk being decoded
    unsigned tmem_base;
    int abort;
};

// barrier over NT threads; true when `pred` held in any of them
template <int NT>
__device__ __forceinline__ bool named_any(int id, bool pred) {
    unsigned r;
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred a, b;\n\t"
        "setp.ne.u32 a, %1, 0;\n\t"
        "bar.red.or.pred b, %2, %3, a;\n\t"
        "selp.u32 %0, 1, 0, b;\n\t}"
        : "=r"(r) : "r"(pred ? 1u : 0u), "r"(id), "n"(NT) : "memory");
    return r != 0u;
}

// One gather: the taps (di0 + s * i, dj0 + s * j), i < ni, j < nj, of one plane; tap (i, j) reads the rows
// i * Wp + j further on than the tile's own, counted from `base`.  A pixel (y, x) of the plane's line is the
// image's (y * s + dy, x * s + dx).
struct TapGroup {
    int di0, dj0, ni, nj, base, dy, dx;
};
__device__ __forceinline__ int tap_groups(const HaloParams &p) {
    const int pa = p.stride < p.KH ? p.stride : p.KH, pb = p.stride < p.KW ? p.stride : p.KW;
    return p.group_mode == 0 ? pa * pb : (p.group_mode == 1 ? p.KH * pb : p.KH * p.KW);
}
__device__ __forceinline__ TapGroup tap_group(const HaloParams &p, int g) {
    const int s = p.stride, pb = s < p.KW ? s : p.KW;
    TapGroup t;
    if (p.group_mode == 2) { t.di0 = g / p.KW; t.dj0 = g - t.di0 * p.KW; }
    else { t.di0 = g / pb; t.dj0 = g - t.di0 * pb; }
    t.ni = p.group_mode == 0 ? (p.KH - 1 - t.di0) / s + 1 : 1;
    t.nj = p.group_mode == 2 ? 1 : (p.KW - 1 - t.dj0) / s + 1;
    t.base = (t.di0 / s) * p.Wp + t.dj0 / s;
    if (p.shared_pad) t.base -= p.pad * p.Wp + p.pad;
    t.dy = p.shared_pad ? 0 : t.di0 % s - p.pad;
    t.dx = p.shared_pad ? 0 : t.dj0 % s - p.pad;
    return t;
}
// (their divisions take longer than a gather's loads: worked out once per CTA)
__device__ __forceinline__ TapGroup load_group(const int4 *a, const int4 *b, int g) {
    const int4 x = a[g], y = b[g];
    TapGroup t = {x.x, x.y, x.z, x.w, y.x, y.y, y.z};
    return t;
}

// n / d for n < 2^31, with m = floor(2^32 / d) + 1: the product's high word is the quotient or one too many
__device__ __forceinline__ unsigned divide(unsigned n, unsigned d, unsigned m, unsigned *rem) {
    unsigned q = d == 1u ? n : __umulhi(n, m);
    unsigned r = n - q * d;
    if ((int)r < 0) { --q; r += d; }
    *rem = r;
    return q;
}
// (image, row, column) of a pixel of the line
__device__ __forceinline__ void split_pixel(const HaloParams &p, long long P, int *img, int *y, int *x) {
    const unsigned per_img = (unsigned)p.Hp * (unsigned)p.Wp;
    unsigned rem, col;
    if (p.M < (1ll << 31)) *img = (int)divide((unsigned)P, per_img, p.img_magic, &rem);
    else { const long long q = P / per_img; *img = (int)q; rem = (unsigned)(P - q * per_img); }
    *y = (int)divide(rem, (unsigned)p.Wp, p.row_magic, &col);
    *x = (int)col;
}

// Entries of a record's lists that a thread holds while they travel, `round` by `round`.
template <int BW>
struct Entries {
    static constexpr int BATCH = BW == 16 ? 1 : (BW == 2 ? 4 : 2);
    uint2 u[BATCH];                     // x: spread signs, y: off | bf16(u) << 16
    unsigned off[BATCH];
    unsigned pay[BATCH][BW / 2];
};
template <int BW>
__device__ __forceinline__ void read_entries(const Params &g, const uint4 &a, const uint4 &b, unsigned first, Entries<BW> &x) {
    const uint2 *ul = reinterpret_cast<const uint2 *>(g.packed + g.off_ulist) + a.x;
    const unsigned short *dpos = reinterpret_cast<const unsigned short *>(g.packed + g.off_dpos) + a.y;
    const unsigned *pay = reinterpret_cast<const unsigned *>(g.packed + g.off_dpay) + (size_t)a.y * (BW / 2);
    const unsigned n_u = b.x - a.x, n_d = b.y - a.y;
#pragma unroll
    for (int k = 0; k < Entries<BW>::BATCH; ++k) {
        const unsigned e = first + (unsigned)k * CV_WORK_THREADS;
        if (e < n_u) x.u[k] = __ldg(ul + e);
        if (e < n_d) {
            x.off[k] = __ldg(dpos + e);
            const unsigned *src = pay + (size_t)e * (BW / 2);
            if (BW >= 8) {
#pragma unroll
                for (int h = 0; h < BW / 8; ++h) {
                    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src) + h);
                    x.pay[k][(4 * h) % (BW / 2)] = v.x; x.pay[k][(4 * h + 1) % (BW / 2)] = v.y;
                    x.pay[k][(4 * h + 2) % (BW / 2)] = v.z; x.pay[k][(4 * h + 3) % (BW / 2)] = v.w;
                }
            } else if (BW == 4) {
                const uint2 v = __ldg(reinterpret_cast<const uint2 *>(src));
                x.pay[k][0] = v.x; x.pay[k][1 % (BW / 2)] = v.y;
            } else x.pay[k][0] = __ldg(src);
        }
    }
}
template <int BW>
__device__ __forceinline__ void put_block(unsigned char *tile, unsigned off, const unsigned (&w)[BW / 2]) {
    if (BW >= 8) *reinterpret_cast<uint4 *>(tile + off) = make_uint4(w[0], w[1 % (BW / 2)], w[2 % (BW / 2)], w[3 % (BW / 2)]);
    if (BW == 16)
        *reinterpret_cast<uint4 *>(tile + (off ^ 16u)) = make_uint4(w[4 % (BW / 2)], w[5 % (BW / 2)], w[6 % (BW / 2)], w[7 % (BW / 2)]);
    if (BW == 4) *reinterpret_cast<uint2 *>(tile + off) = make_uint2(w[0], w[1 % (BW / 2)]);
    if (BW == 2) *reinterpret_cast<unsigned *>(tile + off) = w[0];
}
template <int BW>
__device__ __forceinline__ void write_blocks(unsigned char *tile, const uint4 &a, const uint4 &b, unsigned first, const Entries<BW> &x) {
    constexpr unsigned OFF_MASK = DecodeCfg<BW, CV_WORK_THREADS>::OFF_MASK;
    const unsigned n_u = b.x - a.x, n_d = b.y - a.y;
#pragma unroll
    for (int k = 0; k < Entries<BW>::BATCH; ++k) {
        const unsigned e = first + (unsigned)k * CV_WORK_THREADS;
        if (e < n_u) {
            const unsigned u2 = __byte_perm(x.u[k].y, 0u, 0x3232);
            unsigned w[BW / 2];
#pragma unroll
            for (int t = 0; t < BW / 2; ++t) w[t] = ((x.u[k].x << (15 - t)) & 0x80008000u) ^ u2;      // sign bits t and 16+t
            put_block<BW>(tile, x.u[k].y & OFF_MASK, w);
        }
        if (e < n_d) put_block<BW>(tile, x.off[k] & OFF_MASK, x.pay[k]);
    }
}

// Row r of the record tiles, laid end to end, is 64 * TAPS values in [channel][tap] order; afterwards tile t
// holds the 64 channels of tap t.  A warp holds a row in registers in between; lane l takes channels 2l and
// 2l + 1 of every tap.  A warp's rows have one r % 8, so the places in the swizzled rows are computed once.
template <int TAPS>
__device__ __noinline__ void permute_rows(unsigned w_s, int warp, int lane) {
    const int r8 = warp & 7;
    unsigned from[2][TAPS];
#pragma unroll
    for (int t = 0; t < TAPS; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned k = (unsigned)((2 * lane + h) * TAPS + t), col = k & 63u;
            from[h][t] = (k >> 6) * REC_BYTES + (((col >> 3) ^ (unsigned)r8) << 4) + (col & 7u) * 2u;
        }
    const unsigned to = (((unsigned)lane >> 2) ^ (unsigned)r8) * 16u + ((unsigned)lane & 3u) * 4u;
#pragma unroll 2
    for (int g8 = warp >> 3; g8 < kTileRows / 8; g8 += CV_WORKERS / 8) {
        const unsigned row = w_s + (unsigned)(g8 * 1024 + r8 * 128);
        unsigned short lo[TAPS], hi[TAPS];
#pragma unroll
        for (int t = 0; t < TAPS; ++t) {
            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(lo[t]) : "r"(row + from[0][t]));
            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(hi[t]) : "r"(row + from[1][t]));
        }
        __syncwarp();
#pragma unroll
        for (int t = 0; t < TAPS; ++t)
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(row + (unsigned)t * REC_BYTES + to), "r"((unsigned)lo[t] | ((unsigned)hi[t] << 16)) : "memory");
    }
}

// The records of one chunk of 64 channels -> one 128 x 64 tile per tap, by all workers.
template <int BW>
__device__ __forceinline__ void weights_to_taps(const HaloParams &p, unsigned char *w, uint4 *s_rec, int nt, int chunk, int taps, int tid) {
    const uint4 *recs = reinterpret_cast<const uint4 *>(p.g.packed + p.g.off_rec) + (long long)nt * p.g.n_stages;
    const int s0 = chunk * taps;
    const int n = s0 + taps < (int)p.g.n_stages ? taps : (int)p.g.n_stages - s0;        // at least one
    constexpr unsigned ROUND = Entries<BW>::BATCH * CV_WORK_THREADS;
    if (tid <= n) s_rec[tid] = __ldg(recs + s0 + tid);
    uint4 *z = reinterpret_cast<uint4 *>(w);
    for (int i = tid; i < taps * (REC_BYTES / 16); i += CV_WORK_THREADS) z[i] = make_uint4(0, 0, 0, 0);
    named_any<CV_WORK_THREADS>(1, false);
    // a record whose ranges do not lie inside the sections counts as empty
    auto ends = [&](int i, uint4 &a, uint4 &b) {
        a = s_rec[i];
        b = s_rec[i + 1];
        if (a.x > b.x || b.x > p.g.n_unified || a.y > b.y || b.y > p.g.n_dense) {
            if (tid == 0) atomicOr(p.g.dev_status, (unsigned)MWU_DEV_BOUNDS);
            b.x = a.x; b.y = a.y;
        }
    };
    // The CTAs of a launch mostly decode the same records at the same time; each starts with another one, so that
    // they do not all ask for the same lines of L2 at once.
    int cur_i = (int)(blockIdx.x % (unsigned)n);
    uint4 a, b, na, nb;
    ends(cur_i, a, b);
    Entries<BW> x;
    read_entries<BW>(p.g, a, b, (unsigned)tid, x);
    for (int i = 0; i < n; ++i) {
        const int next_i = cur_i + 1 == n ? 0 : cur_i + 1;
        if (i + 1 < n) ends(next_i, na, nb);
        const unsigned most = max(b.x - a.x, b.y - a.y);
        for (unsigned r0 = 0;; r0 += ROUND) {
            const bool last = r0 + ROUND >= most;
            const Entries<BW> cur = x;
            // the next round's entries travel while this one's are stored
            if (!last) read_entries<BW>(p.g, a, b, r0 + ROUND + (unsigned)tid, x);
            else if (i + 1 < n) read_entries<BW>(p.g, na, nb, (unsigned)tid, x);
            write_blocks<BW>(w + cur_i * REC_BYTES, a, b, r0 + (unsigned)tid, cur);
            if (last) break;
        }
        a = na; b = nb; cur_i = next_i;
    }
    named_any<CV_WORK_THREADS>(1, false);
    const int warp = tid >> 5, lane = tid & 31;
    const unsigned w_s = smem_u32(w);
    switch (taps) {
        case 2: permute_rows<2>(w_s, warp, lane); break;
        case 3: permute_rows<3>(w_s, warp, lane); break;
        case 4: permute_rows<4>(w_s, warp, lane); break;
        case 5: permute_rows<5>(w_s, warp, lane); break;
        case 6: permute_rows<6>(w_s, warp, lane); break;
        case 7: permute_rows<7>(w_s, warp, lane); break;
        case 8: permute_rows<8>(w_s, warp, lane); break;
        case 9: permute_rows<9>(w_s, warp, lane); break;
        default: break;                                     // one tap: the record tile is the tap tile
    }
}

// The rows of one gather.  A warp takes eight channels (a 16-byte piece of a row) of 32 pixels at a time, three
// times 32 pixels in flight together.
__device__ __forceinline__ void gather_rows(const HaloParams &p, unsigned char *dst, const TapGroup &tgp, long long p0, int chunk,
                                            int warp, int lane) {
    const int rows = CV_TILE + (tgp.ni - 1) * p.Wp + tgp.nj - 1;
    const long long plane = (long long)p.H * p.W;
    const int oct = warp & 7, c0 = chunk * BK + oct * 8, n_ch = p.C - c0 < 8 ? p.C - c0 : 8;
    const int sy = p.stride;                                // 1 where zero pixels are shared
    constexpr int U = 3, STEP = 32 * (CV_WORKERS / 8);
    for (int r0 = (warp >> 3) * 32 + lane; r0 - lane < rows; r0 += U * STEP) {
        const unsigned short *src[U];
        bool in[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int r = r0 + k * STEP;
            const long long P = p0 + tgp.base + r;
            int img = 0, y = 0, x = 0;
            in[k] = r < rows && P >= 0 && P < p.M && n_ch > 0;
            split_pixel(p, in[k] ? P : 0, &img, &y, &x);
            y = y * sy + tgp.dy;
            x = x * sy + tgp.dx;
            in[k] = in[k] && (unsigned)y < (unsigned)p.H && (unsigned)x < (unsigned)p.W;
            src[k] = in[k] ? p.X + ((long long)img * p.C + c0) * plane + (y * p.W + x) : p.X;
        }
        unsigned v[U][8];
#pragma unroll
        for (int k = 0; k < U; ++k)
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                v[k][e] = 0;
                if (in[k] && e < n_ch) v[k][e] = __ldg(src[k] + e * plane);
            }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int r = r0 + k * STEP;
            if (r < p.a_rows && r - lane < rows)
                *reinterpret_cast<uint4 *>(dst + swz((unsigned)r, (unsigned)oct)) =
                    make_uint4(v[k][0] | (v[k][1] << 16), v[k][2] | (v[k][3] << 16), v[k][4] | (v[k][5] << 16), v[k][6] | (v[k][7] << 16));
        }
    }
}

template <int BW>
__global__ void __launch_bounds__(CV_THREADS, 1) mwu_conv_halo_kernel(const __grid_constant__ HaloParams p) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    MWU_CHECK_HEADER(p.g);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_raw + smem_pad_1024(smem_raw);
    unsigned char *sW = base;
    unsigned char *sA = sW + (size_t)(p.KH * p.KW) * REC_BYTES;
    __shared__ HaloSmem sm_;
    HaloSmem *sm = &sm_;
    volatile int *abort = &sm->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int taps = p.KH * p.KW, n_groups = tap_groups(p);
    const int rank = (int)(blockIdx.x % (unsigned)p.split);
    const unsigned unit = blockIdx.x / (unsigned)p.split;
    const int nt = (int)(unit / (unsigned)p.per_ntile), first_tile = (int)(unit % (unsigned)p.per_ntile);
    const long long n_tiles = (p.M + CV_TILE - 1) / CV_TILE;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sm->a_full[b]), CV_WORKERS);
            mbar_init(smem_u32(&sm->a_empty[b]), 1);
        }
        mbar_init(smem_u32(&sm->w_full), CV_WORKERS);
        mbar_init(smem_u32(&sm->w_empty), 1);
        mbar_init(smem_u32(&sm->t_full), 1);
        mbar_init(smem_u32(&sm->t_empty), CV_WORKERS);
        sm->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1 && lane < n_groups) {
        const TapGroup t = tap_group(p, lane);
        sm->group[lane] = make_int4(t.di0, t.dj0, t.ni, t.nj);
        sm->group2[lane] = make_int4(t.base, t.dy, t.dx, 0);
    }
    __syncwarp();
    if (warp == CV_MMA_WARP) {
        tmem_alloc(smem_u32(&sm->tmem_base), p.tmem_cols);
        // by this warp, and only now: the kernel behind may take all of an SM's tensor memory before it waits for this one
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = *reinterpret_cast<volatile unsigned *>(&sm->tmem_base);
    const unsigned a_bytes = (unsigned)p.a_rows * 128u;
    const long long step = (long long)p.per_ntile;          // tiles first_tile, first_tile + step, ...

    if (warp < CV_WORKERS) {
        // ---------------- weights, halo rows, then the output ----------------
        unsigned ab = 0, a_phase = 0, t_phase = 0, w_phase = 0;
        bool ok = true;
        for (long long t0 = first_tile; t0 < n_tiles; t0 += CV_BATCH * step) {
            // A wait that runs out makes a worker skip its work, but not leave: all of them meet at every barrier
            // of the workers and leave together there.
            for (int chunk = rank; chunk < p.chunks; chunk += p.split) {
                if (ok && !mbar_wait(smem_u32(&sm->w_empty), w_phase ^ 1u, abort)) ok = false;
                if (named_any<CV_WORK_THREADS>(1, !ok)) { ok = false; break; }          // the same decision in every worker
                weights_to_taps<BW>(p, sW, sm->rec, nt, chunk, taps, (int)threadIdx.x);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sm->w_full));
                w_phase ^= 1u;
                for (int q = 0; q < CV_BATCH && t0 + q * step < n_tiles; ++q) {
                    const long long p0 = (t0 + q * step) * CV_TILE;
                    for (int g = 0; ok && g < n_groups; ++g) {
                        if (!mbar_wait(smem_u32(&sm->a_empty[ab]), a_phase ^ 1u, abort)) ok = false;
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                        gather_rows(p, sA + ab * a_bytes, load_group(sm->group, sm->group2, g), p0, chunk, warp, lane);
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&sm->a_full[ab]));
                        if (++ab == (unsigned)p.a_bufs) { ab = 0; a_phase ^= 1u; }
                    }
                }
            }
            if (ok && !mbar_wait(smem_u32(&sm->t_full), t_phase, abort)) ok = false;
            if (named_any<CV_WORK_THREADS>(1, !ok)) { ok = false; break; }
            t_phase ^= 1u;
            tc_fence_after();
            // tensor-memory lanes are pixels, columns are filters: 32 columns to a warp
            const int quarter = warp & 3, c0 = (warp >> 2) * 32;
            const long long out_plane = (long long)p.OH * p.OW;
            for (int q = 0; q < CV_BATCH && t0 + q * step < n_tiles; ++q) {
                const unsigned trow = tmem_base + ((unsigned)(quarter * 32) << 16) + (unsigned)(q * 128 + c0);
                if (p.split > 1) {
                    // partial sums [filter][pixel] for the cluster (one tile per CTA then); the tap tiles are free
                    float *part = reinterpret_cast<float *>(base);
                    unsigned v[32];
                    tmem_ld32(trow, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) part[(c0 + j) * CV_TILE + quarter * 32 + lane] = __uint_as_float(v[j]);
                    break;
                }
                const long long P = (t0 + q * step) * CV_TILE + quarter * 32 + lane;
                int img = 0, oh = 0, ow = 0;
                bool px = P < p.M;
                if (px) {
                    split_pixel(p, P, &img, &oh, &ow);
                    px = oh < p.OH && ow < p.OW;
                }
                const long long at = (long long)img * p.g.N * out_plane + (long long)oh * p.OW + ow;
                const long long o0 = (long long)nt * kTileRows + c0;
                unsigned v[32];
                tmem_ld32(trow, v);
                if (px) {
                    if (p.g.y_fp32) {
                        float *dst = reinterpret_cast<float *>(p.g.Y) + at + o0 * out_plane;
#pragma unroll
                        for (int j = 0; j < 32; ++j, dst += out_plane)
                            if (o0 + j < p.g.N) *dst = __uint_as_float(v[j]);
                    } else {
                        __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(p.g.Y) + at + o0 * out_plane;
#pragma unroll
                        for (int j = 0; j < 32; ++j, dst += out_plane)
                            if (o0 + j < p.g.N) *dst = __float2bfloat16_rn(__uint_as_float(v[j]));
                    }
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sm->t_empty));
        }
    } else {
        // ---------------- MMA issuer ----------------
        const unsigned idesc = make_idesc(128);
        unsigned ab = 0, a_phase = 0, w_phase = 0, t_phase = 0;
        bool ok = true, issued = false;
        for (long long t0 = first_tile; ok && t0 < n_tiles; t0 += CV_BATCH * step) {
            if (!mbar_wait_spin(smem_u32(&sm->t_empty), t_phase ^ 1u, abort)) ok = false;
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            tc_fence_after();
            for (int chunk = rank; ok && chunk < p.chunks; chunk += p.split) {
                if (!mbar_wait_spin(smem_u32(&sm->w_full), w_phase, abort)) ok = false;
                if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                for (int q = 0; ok && q < CV_BATCH && t0 + q * step < n_tiles; ++q) {
                    bool fresh = chunk == rank;          // the tile's first MMA overwrites
                    for (int g = 0; ok && g < n_groups; ++g) {
                        const TapGroup tgp = load_group(sm->group, sm->group2, g);
                        if (!mbar_wait_spin(smem_u32(&sm->a_full[ab]), a_phase, abort)) ok = false;
                        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                        tc_fence_after();
                        const unsigned a_s = smem_u32(sA + ab * a_bytes), w_s = smem_u32(sW);
                        if (elect_one()) {
                            for (int i = 0; i < tgp.ni; ++i)
                                for (int j = 0; j < tgp.nj; ++j) {
                                    const int tap = (tgp.di0 + i * p.stride) * p.KW + tgp.dj0 + j * p.stride;
                                    const unsigned long long adesc = make_desc(a_s + (unsigned)(i * p.Wp + j) * 128u);
                                    const unsigned long long bdesc = make_desc(w_s + (unsigned)tap * REC_BYTES);
#pragma unroll
                                    for (int k4 = 0; k4 < 4; ++k4) {
                                        umma_bf16(tmem_base + (unsigned)(q * 128), adesc + (unsigned long long)(k4 * 2),
                                                  bdesc + (unsigned long long)(k4 * 2), idesc, fresh ? 0u : 1u);
                                        fresh = false;
                                    }
                                }
                            umma_commit(smem_u32(&sm->a_empty[ab]));
                        }
                        fresh = false;
                        issued = true;
                        __syncwarp();
                        if (++ab == (unsigned)p.a_bufs) { ab = 0; a_phase ^= 1u; }
                    }
                }
                if (!ok) break;
                if (elect_one()) umma_commit(smem_u32(&sm->w_empty));
                __syncwarp();
                w_phase ^= 1u;
            }
            if (!ok) break;
            if (elect_one()) umma_commit(smem_u32(&sm->t_full));
            __syncwarp();
            t_phase ^= 1u;
        }
        // everything this warp issued must have retired before tensor memory is freed
        if (issued) {
            __shared__ unsigned long long drain;
            __shared__ int s_no_abort;
            if (lane == 0) {
                s_no_abort = 0;
                mbar_init(smem_u32(&drain), 1);
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            }
            __syncwarp();
            if (elect_one()) umma_commit(smem_u32(&drain));
            __syncwarp();
            mbar_wait(smem_u32(&drain), 0, &s_no_abort);
        }
        __syncwarp();
    }

    // teardown
    tc_fence_before();
    __syncthreads();
    // after the barrier: a role that finished its own work early must still see a flag raised later
    if (*abort && threadIdx.x == 0) atomicOr(p.g.dev_status, (unsigned)MWU_DEV_TIMEOUT);
    __syncwarp();
    if (warp == CV_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, p.tmem_cols);
    }
    if (p.split > 1) {
        // tensor memory is given back before the cluster barrier, so holding it never depends on another CTA
        cluster_sync_all();
        const float *part = reinterpret_cast<const float *>(base);
        const long long P0 = (long long)first_tile * CV_TILE, out_plane = (long long)p.OH * p.OW;
        // filters rank, rank + split, ...: a warp sums 32 pixels of one filter
        for (int w = warp; w < (kTileRows / p.split) * (CV_TILE / 32); w += CV_THREADS / 32) {
            const int f = (w >> 2) * p.split + rank, px0 = (w & 3) * 32 + lane;
            const long long P = P0 + px0, o = (long long)nt * kTileRows + f;
            float acc = 0.f;
            const unsigned at = smem_u32(part + f * CV_TILE + px0);
#pragma unroll 4
            for (int c = 0; c < p.split; ++c) {
                float v;
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(mbar_addr_in_cta(at, (unsigned)c)) : "memory");
                acc += v;
            }
            int img = 0, oh = 0, ow = 0;
            bool px = P < p.M && o < p.g.N && *abort == 0;
            if (px) {
                split_pixel(p, P, &img, &oh, &ow);
                px = oh < p.OH && ow < p.OW;
            }
            if (px) {
                const long long idx = ((long long)img * p.g.N + o) * out_plane + (long long)oh * p.OW + ow;
                if (p.g.y_fp32) reinterpret_cast<float *>(p.g.Y)[idx] = acc;
                else reinterpret_cast<__nv_bfloat16 *>(p.g.Y)[idx] = __float2bfloat16_rn(acc);
            }
        }
        __syncwarp();
        cluster_sync_all();                                 // nobody leaves while its sums are still being read
    }
}

// ------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------
// The line of pixels, the gather that fits beside the tap tiles, and the split of the work.  p.g.N, C .. NIMG
// are set.  Zero pixels: with stride 1 and pad < kernel one run of `pad` after every image row and `pad` rows
// after every image serve both neighbours; otherwise (strides, wider paddings) the padded image is laid out
// in full, one plane per residue of the stride.
static void halo_geometry(HaloParams &p, int sm_count) {
    const int s = p.stride;
    p.OH = (p.H + 2 * p.pad - p.KH) / s + 1;
    p.OW = (p.W + 2 * p.pad - p.KW) / s + 1;
    p.shared_pad = s == 1 && p.pad < p.KH && p.pad < p.KW;
    p.Hp = p.shared_pad ? p.H + p.pad : (p.H + 2 * p.pad + s - 1) / s;
    p.Wp = p.shared_pad ? p.W + p.pad : (p.W + 2 * p.pad + s - 1) / s;
    p.M = (long long)p.NIMG * p.Hp * p.Wp;
    p.img_magic = (unsigned)((1ull << 32) / ((unsigned)p.Hp * (unsigned)p.Wp)) + 1u;
    p.row_magic = (unsigned)((1ull << 32) / (unsigned)p.Wp) + 1u;
    p.chunks = (p.C + BK - 1) / BK;
    const long long room = CV_SMEM - 2048 - (long long)(p.KH * p.KW) * REC_BYTES;
    for (p.group_mode = 0; p.group_mode < 3; ++p.group_mode) {
        const long long ni = p.group_mode == 0 ? (p.KH - 1) / s + 1 : 1, nj = p.group_mode == 2 ? 1 : (p.KW - 1) / s + 1;
        const long long rows = (CV_TILE + (ni - 1) * p.Wp + nj - 1 + 7) / 8 * 8;
        if (rows * 128 <= room || p.group_mode == 2) {
            p.a_rows = (int)rows;
            p.a_bufs = rows * 256 <= room ? 2 : 1;
            break;
        }
    }
    const long long n_tiles = (p.M + CV_TILE - 1) / CV_TILE;
    long long per = sm_count / p.n_ntiles;
    if (per < 1) per = 1;
    if (per > n_tiles) per = n_tiles;
    p.per_ntile = (int)per;
    p.split = 1;
    if (per == n_tiles)
        while (p.split * 2 <= 8 && p.split * 2 <= p.chunks && n_tiles * p.n_ntiles * p.split * 2 <= sm_count) p.split *= 2;
    const long long mine = (n_tiles + per - 1) / per;
    p.tmem_cols = mine > 2 ? 512u : (mine > 1 ? 256u : 128u);
}

// Shapes this kernel serves: up to nine taps, and an image whose padded rows and columns can be counted in 32 bits (the
// paddings of an image of a few pixels may reach 32767).  The rest take the kernel for any number of taps.
bool halo_eligible(int h, int w, int kh, int kw, int stride, int pad) {
    const long long hp = (h + 2ll * pad + stride - 1) / stride, wp = (w + 2ll * pad + stride - 1) / stride;
    return (long long)kh * kw <= CV_TAPS && hp * wp < (1ll << 31);
}

// `g` carries the packed weights and the output; the image is X [n][c][h][w]
int run_conv_halo(const Params &g, const void *X, int n, int c, int h, int w, int kh, int kw, int stride, int pad, int sm_count,
                  cudaStream_t st) {
    HaloParams p = {};
    p.g = g;
    p.X = (const unsigned short *)X;
    p.C = c; p.H = h; p.W = w; p.KH = kh; p.KW = kw; p.stride = stride; p.pad = pad; p.NIMG = n;
    p.n_ntiles = (int)g.n_rec_tiles;
    halo_geometry(p, sm_count);
    auto kern = g.bw == 2 ? mwu_conv_halo_kernel<2> : g.bw == 4 ? mwu_conv_halo_kernel<4>
              : g.bw == 8 ? mwu_conv_halo_kernel<8> : mwu_conv_halo_kernel<16>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CV_SMEM - 1024) != cudaSuccess) return MWU_ERR_CUDA;
    const long long grid = (long long)p.n_ntiles * p.per_ntile * p.split;
    if (grid >= (1ll << 31)) return MWU_ERR_SHAPE;
    size_t smem = (size_t)(kh * kw) * REC_BYTES + (size_t)p.a_bufs * p.a_rows * 128;
    if (p.split > 1 && smem < (size_t)kTileRows * CV_TILE * 4) smem = (size_t)kTileRows * CV_TILE * 4;       // partial sums
    count_launch();
    return launch_chained(kern, dim3((unsigned)grid), dim3(CV_THREADS), smem + 1024, st, p.split, p) == cudaSuccess ? MWU_OK
                                                                                                                    : MWU_ERR_CUDA;
}

}  // namespace gemm
}  // namespace mwu
