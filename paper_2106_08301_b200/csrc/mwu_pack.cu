// mwu_pack: serialise a projection into the packed storage form (Section 3.1 / Table 1: one
// magnitude per unified block, nothing but its position for a pruned block, one sign bit per
// weight of a unified block, bf16 values for the rest), arranged per GEMM tile.
//
//   count_kernel  a CTA per tile of 128 rows and 32 records, a lane per record (128 rows x 64 columns)
//                 walking the rows: number of unified / dense / pruned blocks and the record's live-slice
//                 mask.  Only for weights of many records; a few are counted by scan_kernel itself.
//   scan_kernel   one cluster of eight CTAs: exclusive scan of the per-record counts (each CTA its eighth,
//                 totals through distributed shared memory), header.
//   fill_kernel   one CTA per record.  First one thread per row: class masks, then a scan over the
//                 rows of the number of blocks per (class, store slot), which gives every block its
//                 place in the round-robin order of its class list; the places go to shared memory.
//                 Then the lists leave in list order, consecutive threads writing consecutive
//                 entries; a dense block's values are read by the lanes that share its 64-byte run.
// The three are chained with programmatic stream serialization.  Weights of up to 655360 blocks need fill_kernel alone: its
// CTAs count what comes before their records themselves.
#include "mwu_common.cuh"

namespace mwu {
namespace pack {

struct Params {
    const float *W;
    const float *U;
    const float *u;
    const unsigned *pruned_bitmap;
    const unsigned *unified_bitmap;
    const unsigned *sign_bits;
    unsigned char *packed;
    unsigned *dev_status;
    long long rows, cols;
    int b;
    long long bpr;                  // blocks per row: cols / b
    unsigned n_stages;              // L.n_stages, for 32-bit record arithmetic (records < 2^31)
    PackedLayout L;
    unsigned long long gap[5][2];   // byte ranges between the sections (alignment padding), zeroed with the header
};

// class masks of row r of a record; padding rows are all-pruned
__device__ __forceinline__ void row_masks(const Params &p, int nb, long long tile, long long stage, int r,
                                          unsigned *P, unsigned *U, unsigned long long *sgn) {
    const unsigned mask = (nb >= 32) ? 0xffffffffu : ((1u << nb) - 1u);
    const long long n = tile * kTileRows + r;
    *P = mask;
    *U = 0;
    *sgn = 0;
    if (n < p.rows) {
        const long long j0 = n * p.bpr + stage * nb;
        *P = (p.pruned_bitmap[j0 >> 5] >> (j0 & 31)) & mask;
        *U = (p.unified_bitmap[j0 >> 5] >> (j0 & 31)) & mask & ~*P;
        const long long f = n * p.cols + stage * kStageK;
        *sgn = (unsigned long long)p.sign_bits[f >> 5] |
               ((unsigned long long)p.sign_bits[(f >> 5) + 1] << 32);
    }
}

// byte offset of block i of row r inside the record's decoded tile: rows of 128 bytes, the
// row's 16-byte chunks XOR-permuted by r % 8 (the layout the tensor-core instruction reads)
__device__ __forceinline__ unsigned tile_offset(unsigned r, unsigned i, int b) {
    const unsigned byte_in_row = i * 2u * (unsigned)b;
    const unsigned c = byte_in_row >> 4, within = byte_in_row & 15u;
    return (r >> 3) * 1024u + (r & 7u) * 128u + ((c ^ (r & 7u)) << 4) + within;
}

// sign bits of one block (bit l = weight l, at most 16 of them) -> bit l/2 + 16 * (l % 2): the even bits closed up in the
// low half, the odd bits in the high half
__device__ __forceinline__ unsigned spread_signs(unsigned x) {
    unsigned t = (x ^ (x >> 1)) & 0x2222u;
    x ^= t ^ (t << 1);
    t = (x ^ (x >> 2)) & 0x0c0cu;
    x ^= t ^ (t << 2);
    t = (x ^ (x >> 4)) & 0x00f0u;
    x ^= t ^ (t << 4);
    return __byte_perm(x, 0u, 0x4140);
}

__device__ __forceinline__ unsigned live_of(unsigned P, int b) {
    const int nb = kStageK / b;
    const unsigned mask = (nb >= 32) ? 0xffffffffu : ((1u << nb) - 1u);
    const unsigned notP = ~P & mask;
    const int bps = (16 / b) > 0 ? (16 / b) : 1;            // blocks per 16-column slice
    unsigned live = 0;
    for (int s = 0; s < 4; ++s) {
        const unsigned m = (b >= 16) ? (1u << s) : (((1u << bps) - 1u) << (s * bps));
        if (notP & m) live |= 1u << s;
    }
    return live;
}

constexpr int COUNT_WARPS = 16;                         // each takes 8 of the tile's 128 rows

struct CountSmem {
    unsigned cu[COUNT_WARPS][32], cp[COUNT_WARPS][32], live[COUNT_WARPS][32];
};

// Counts of one unit (a tile and 32 of its stages), by COUNT_WARPS warps (warp: 0 .. COUNT_WARPS-1) that all
// call it together; the first of them writes them to the record table.  `sync` joins these warps.
template <class Sync>
__device__ __forceinline__ void count_unit(const Params &p, unsigned unit, int warp, int lane, CountSmem &s, Sync sync) {
    const unsigned chunks = (p.n_stages + 31u) / 32u;       // 32 records of a tile at a time: lane = record (stage)
    const long long tile = unit / chunks;
    const long long stage = (long long)(unit % chunks) * 32 + lane;
    const int nb = kStageK / p.b;
    const unsigned mask = (nb >= 32) ? 0xffffffffu : ((1u << nb) - 1u);
    const long long bpr = p.bpr;                            // blocks per row
    constexpr int RPW = kTileRows / COUNT_WARPS;
    unsigned cu = 0, cp = 0, live = 0;
    if (stage < p.L.n_stages) {
        unsigned P[RPW], U[RPW];
#pragma unroll
        for (int rr = 0; rr < RPW; ++rr) {                  // all of the warp's loads are in flight together
            const long long n = tile * kTileRows + warp * RPW + rr;
            P[rr] = 0xffffffffu;                            // padding rows are all-pruned
            U[rr] = 0;
            if (n < p.rows) {
                const long long j0 = n * bpr + stage * nb;
                P[rr] = __ldg(p.pruned_bitmap + (j0 >> 5)) >> (j0 & 31);
                U[rr] = __ldg(p.unified_bitmap + (j0 >> 5)) >> (j0 & 31);
            }
        }
#pragma unroll
        for (int rr = 0; rr < RPW; ++rr) {
            const unsigned Pm = P[rr] & mask;
            cu += __popc(U[rr] & mask & ~Pm);
            cp += __popc(Pm);
            live |= live_of(Pm, p.b);
        }
    }
    s.cu[warp][lane] = cu; s.cp[warp][lane] = cp; s.live[warp][lane] = live;
    sync();
    if (warp == 0 && stage < p.L.n_stages) {
        unsigned tu = 0, tp = 0, tl = 0;
#pragma unroll
        for (int w = 0; w < COUNT_WARPS; ++w) { tu += s.cu[w][lane]; tp += s.cp[w][lane]; tl |= s.live[w][lane]; }
        // counts for now (ubase, dbase, pbase, live); scan_kernel makes bases
        uint4 *recs = reinterpret_cast<uint4 *>(p.packed + p.L.off_rec);
        recs[tile * p.L.n_stages + stage] = make_uint4(tu, (unsigned)(kTileRows * nb) - tu - tp, tp, tl);
    }
}

// launched with programmatic stream serialization: the projection may still be running
__global__ void __launch_bounds__(32 * COUNT_WARPS) count_kernel(Params p) {
    __shared__ CountSmem s;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    count_unit(p, blockIdx.x, threadIdx.x >> 5, threadIdx.x & 31, s, [] { __syncthreads(); });
}

constexpr int SCAN_CTAS = 8, SCAN_THREADS = 1024, SCAN_PER = 4;      // consecutive records a thread takes at a time

__device__ __forceinline__ void scan_cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// header and gaps, by the first six warps of a CTA
__device__ __forceinline__ void write_header(const Params &p) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the padding between the sections must read as zero (each gap is shorter than the alignment)
    {
        const int g = wid - 1;                              // a warp to a gap; the first warp writes the header
        if (g >= 0 && g < 5)
            for (unsigned long long a = p.gap[g][0] + lane; a < p.gap[g][1]; a += 32) p.packed[a] = 0;
    }
    if (threadIdx.x < 32) {
        unsigned long long *h = reinterpret_cast<unsigned long long *>(p.packed);
        unsigned long long v = 0;
        switch (threadIdx.x) {
            case 0: v = kMagic; break;
            case 1: v = 4; break;
            case 2: v = (unsigned long long)p.rows; break;
            case 3: v = (unsigned long long)p.cols; break;
            case 4: v = (unsigned long long)p.b; break;
            case 5: v = (unsigned long long)p.L.n_pad; break;
            case 6: v = (unsigned long long)p.L.n_tiles; break;
            case 7: v = (unsigned long long)p.L.n_stages; break;
            case 8: v = (unsigned long long)p.L.n_pruned; break;
            case 9: v = (unsigned long long)p.L.n_unified; break;
            case 10: v = (unsigned long long)p.L.n_dense; break;
            case 11: v = (unsigned long long)p.L.n_plist; break;
            case 12: v = (unsigned long long)p.L.off_rec; break;
            case 13: v = (unsigned long long)p.L.off_ulist; break;
            case 14: v = (unsigned long long)p.L.off_dpos; break;
            case 15: v = (unsigned long long)p.L.off_dpay; break;
            case 16: v = (unsigned long long)p.L.off_ppos; break;
            case 17: v = (unsigned long long)p.L.total; break;
            default: v = 0;
        }
        h[threadIdx.x] = v;
    }
}

// Bound by latency: a handful of dependent L2 round trips and cluster barriers (8192 records on one CTA, in
// two rounds, took 13 us).  Counts the records itself when count_kernel has not (`counted` == 0).
__global__ void __launch_bounds__(SCAN_THREADS) scan_kernel(Params p, int counted) {
    __shared__ CountSmem s_count[SCAN_THREADS / (32 * COUNT_WARPS)];
    __shared__ unsigned s_w[3][32];
    __shared__ unsigned long long s_tot[3];                 // this CTA's totals, read by all
    __shared__ unsigned long long s_before[2][3];           // totals of the CTAs before this one, and of all
    const unsigned n_rec = (unsigned)(p.L.n_tiles * p.L.n_stages);
    uint4 *recs = reinterpret_cast<uint4 *>(p.packed + p.L.off_rec);     // ubase, dbase, pbase, live
    const unsigned cta = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // fill_kernel reads the projection's outputs before it waits for this kernel, so it may start only once
    // the projection is complete: after count_kernel's own wait, or after this one
    if (!counted) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");      // the counts are complete and visible
    if (!counted) {
        constexpr int TEAMS = SCAN_THREADS / (32 * COUNT_WARPS);
        const int team = wid / COUNT_WARPS;
        const unsigned units = (unsigned)p.L.n_tiles * ((p.n_stages + 31u) / 32u);
        for (unsigned unit = cta * TEAMS + team; unit < units; unit += SCAN_CTAS * TEAMS) {
            auto join = [team] { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(32 * COUNT_WARPS) : "memory"); };
            count_unit(p, unit, wid % COUNT_WARPS, lane, s_count[team], join);
            join();                                         // the counts have been read
        }
        scan_cluster_sync();
    }
    const unsigned per = (n_rec + SCAN_CTAS - 1) / SCAN_CTAS;
    const unsigned r0 = min(cta * per, n_rec), r1 = min(r0 + per, n_rec);
    constexpr unsigned STEP = SCAN_PER * SCAN_THREADS;
    uint4 held[SCAN_PER];
    auto read = [&](unsigned i0) {
#pragma unroll
        for (int k = 0; k < SCAN_PER; ++k) held[k] = (i0 + k < r1) ? __ldcg(recs + i0 + k) : make_uint4(0, 0, 0, 0);
    };
    // totals of this CTA's records
    unsigned long long tot[3] = {0, 0, 0};
    for (unsigned g0 = r0; g0 < r1; g0 += STEP) {
        read(g0 + threadIdx.x * SCAN_PER);
#pragma unroll
        for (int k = 0; k < SCAN_PER; ++k) { tot[0] += held[k].x; tot[1] += held[k].y; tot[2] += held[k].z; }
    }
    if (threadIdx.x < 3) s_tot[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        // a thread's share fits 32 bits (counts of up to 4096 blocks); CTAs hold fewer than 2^31 blocks in all
        const unsigned t = __reduce_add_sync(0xffffffffu, (unsigned)tot[c]);
        if (lane == 0 && t) atomicAdd(&s_tot[c], (unsigned long long)t);
    }
    scan_cluster_sync();
    if (threadIdx.x < 3) {
        const unsigned at = (unsigned)__cvta_generic_to_shared(&s_tot[threadIdx.x]);
        unsigned long long before = 0, all = 0;
#pragma unroll
        for (unsigned c = 0; c < SCAN_CTAS; ++c) {
            unsigned long long t;
            unsigned remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(at), "r"(c));
            asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(t) : "r"(remote) : "memory");
            before += c < cta ? t : 0ull;
            all += t;
        }
        s_before[0][threadIdx.x] = before;
        s_before[1][threadIdx.x] = all;
    }
    __syncthreads();
    unsigned long long cu = s_before[0][0], cd = s_before[0][1], cp = s_before[0][2];
    for (unsigned g0 = r0; g0 < r1; g0 += STEP) {
        const unsigned i0 = g0 + threadIdx.x * SCAN_PER;
        if (per > STEP) read(i0);                           // else this thread still holds them
        unsigned su = 0, sd = 0, sp = 0;                    // a step's counts fit 32 bits
#pragma unroll
        for (int k = 0; k < SCAN_PER; ++k) { su += held[k].x; sd += held[k].y; sp += held[k].z; }
        // inclusive scan of the thread sums: inside a warp, then over the 32 warp totals
        unsigned iu = su, id = sd, ip = sp;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned au = __shfl_up_sync(0xffffffffu, iu, off);
            const unsigned ad = __shfl_up_sync(0xffffffffu, id, off);
            const unsigned ap = __shfl_up_sync(0xffffffffu, ip, off);
            if (lane >= off) { iu += au; id += ad; ip += ap; }
        }
        __syncthreads();                                    // the previous step's warp totals have been read
        if (lane == 31) { s_w[0][wid] = iu; s_w[1][wid] = id; s_w[2][wid] = ip; }
        __syncthreads();
        const unsigned wu = s_w[0][lane], wd = s_w[1][lane], wp = s_w[2][lane];
        const unsigned bu = __reduce_add_sync(0xffffffffu, lane < wid ? wu : 0u);      // totals of the warps before this one
        const unsigned bd = __reduce_add_sync(0xffffffffu, lane < wid ? wd : 0u);
        const unsigned bp = __reduce_add_sync(0xffffffffu, lane < wid ? wp : 0u);
        unsigned long long ru = cu + bu + (iu - su), rd = cd + bd + (id - sd), rp = cp + bp + (ip - sp);
#pragma unroll
        for (int k = 0; k < SCAN_PER; ++k) {
            if (i0 + k < r1) recs[i0 + k] = make_uint4((unsigned)ru, (unsigned)rd, (unsigned)rp, held[k].w);
            ru += held[k].x; rd += held[k].y; rp += held[k].z;
        }
        if (per > STEP) {                                   // the totals of this step, for the next one
            cu += __reduce_add_sync(0xffffffffu, wu);
            cd += __reduce_add_sync(0xffffffffu, wd);
            cp += __reduce_add_sync(0xffffffffu, wp);
        }
    }
    scan_cluster_sync();                                    // nobody leaves while its totals are still being read
    if (cta != 0) return;
    if (threadIdx.x == SCAN_THREADS - 1) {
        const unsigned long long au = s_before[1][0], ad = s_before[1][1], ap = s_before[1][2];
        if (au != (unsigned long long)p.L.n_unified || ad != (unsigned long long)p.L.n_dense ||
            ap != (unsigned long long)p.L.n_plist)
            atomicOr(p.dev_status, (unsigned)MWU_DEV_BOUNDS);
        recs[n_rec] = make_uint4((unsigned)au, (unsigned)ad, (unsigned)ap, 0u);
    }
    write_header(p);
}

constexpr unsigned OWN_THREADS = 512;
// CTAs to an SM that the registers are cut to: enough warps to hide the gathers of W and u, few enough that their lines stay in
// L1 until the neighbouring blocks' turn (16384 x 4096, 50 % / 25 %, b = 2: 158 us with 12; 181 with 8 and 317 with 16 where 12 took 175;
// b = 4: 105; b = 8: 84 with 16, 88 with 8).  Without a scan: all 512 CTAs of 2048 x 2048 at once, for 8 bytes of spills (b = 8 11.7 us,
// with three to an SM 13.2; b = 16 9.3 / 11.0).
__host__ __device__ constexpr int fill_ctas(int b, bool own) { return own ? (b == 2 ? 3 : 4) : b <= 4 ? 12 : 16; }
// Most blocks (padding rows included) of the form without a scan: every CTA reads on average half of the bitmaps.  Whole
// mwu_pack calls, 50 % / 25 %, us, with it and without: 1024 x 1024, b = 8: 6.2 / 14.1; 1000 x 1216, b = 2: 11.8 / 14.9; 2048 x 1024, b = 4 and
// 2048 x 2048, b = 8, 524288 blocks: 10.8 / 14.7 and 11.7 / 15.2; 3072 x 2048, b = 8, 786432: 17.7 / 19.6; 1024 x 2048, b = 2, 1048576: 23.5 / 15.9.
constexpr long long OWN_BLOCKS = 655360;

// row and block of a tile offset (the inverse of tile_offset)
__device__ __forceinline__ void row_block_of(unsigned off, int b, unsigned *r, unsigned *i) {
    const unsigned rr = (off >> 10) * 8u + ((off >> 7) & 7u);
    const unsigned c = ((off >> 4) & 7u) ^ (rr & 7u);
    *r = rr;
    *i = (c * 16u + (off & 15u)) / (2u * (unsigned)b);
}

// words of a bit matrix over the lanes of a warp: bit b of lane l becomes bit l of lane b
__device__ __forceinline__ unsigned warp_transpose(unsigned w, int lane) {
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) {
        const unsigned m = k == 16 ? 0x0000ffffu : k == 8 ? 0x00ff00ffu : k == 4 ? 0x0f0f0f0fu : k == 2 ? 0x33333333u : 0x55555555u;
        const unsigned y = __shfl_xor_sync(0xffffffffu, w, k);
        w = (lane & k) ? ((w & ~m) | ((y >> k) & m)) : ((w & m) | ((y & m) << k));
    }
    return w;
}

// Bits of a row's blocks moved to their store slots: slot = (number of the block's first one) ^ (r % 8 chunks of STEP slots).
template <int STEP>
__device__ __forceinline__ unsigned to_slots(unsigned w, unsigned r) {
#pragma unroll
    for (int k = 1; k <= 4; k <<= 1) {
        const int d = k * STEP;
        const unsigned m = d == 16 ? 0x0000ffffu : d == 8 ? 0x00ff00ffu : d == 4 ? 0x0f0f0f0fu : d == 2 ? 0x33333333u : 0x55555555u;
        if (r & (unsigned)k) w = ((w & m) << d) | ((w >> d) & m);
    }
    return w;
}

// Bounded by instruction issue and latency (16384 x 4096, b = 16, 80 % / 60 %: 51 us the whole call with a ballot for each
// (class, slot) and 64-bit addresses, 47.6 so; b = 2, 50 % / 25 %, 175 / 158; 1000 x 1216, b = 8: 7.9 / 6.9).
// Bounded by latency where records are few (a chain of some dozen L2 round trips, out of a cold instruction cache).
// OWN: the base of the record's lists is counted here too, from the bitmaps of everything before it: no record table, no
// kernel before this one; the lists are then written by four times the threads.
template <int B, bool OWN>
__global__ void __launch_bounds__(OWN ? OWN_THREADS : 128, fill_ctas(B, OWN)) fill_kernel(Params p) {
    constexpr unsigned NT = OWN ? OWN_THREADS : 128;
    constexpr int NBK = kStageK / B;
    constexpr unsigned MASK = (NBK >= 32) ? 0xffffffffu : ((1u << NBK) - 1u);
    constexpr int STORE = (B >= 8) ? 16 : 2 * B;            // bytes of one shared-memory store
    constexpr int G = 128 / STORE;                          // store slots of a 128-byte row
    constexpr int LPB = (B >= 4) ? B / 4 : 1;               // lanes that share a dense block's run of W
    if (OWN) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned rec = blockIdx.x;
    const unsigned tile_u = rec / p.n_stages;
    const long long tile = tile_u, stage = rec - tile_u * p.n_stages;
    const int r = threadIdx.x, lane = r & 31, warp = r >> 5;
    const uint4 *recs = reinterpret_cast<const uint4 *>(p.packed + p.L.off_rec);
    uint2 *ulist = reinterpret_cast<uint2 *>(p.packed + p.L.off_ulist);
    unsigned short *dpos = reinterpret_cast<unsigned short *>(p.packed + p.L.off_dpos);
    unsigned char *dpay = p.packed + p.L.off_dpay;
    unsigned short *ppos = reinterpret_cast<unsigned short *>(p.packed + p.L.off_ppos);

    // Rows that can have a block in a given slot: every second one where a block takes two.
    constexpr int QMAX = B == 16 ? kTileRows / 2 : kTileRows;
    __shared__ unsigned s_bal[4][3 * G];                    // per warp and (class, slot): the rows that have such a block
    __shared__ unsigned char s_before[4][3 * G];            // ... how many in the warps before
    // ... and in all; slots w and w + G/2 in word w
    __shared__ __align__(4) unsigned short s_len[3][G];
    // per class and q: list entries of rounds 0 .. q-1, and the slots that have a round q (above bit 16 where they fit there)
    constexpr bool ONE_WORD = G <= 16;
    __shared__ unsigned s_round[3][QMAX + 1];
    __shared__ unsigned short s_full[ONE_WORD ? 1 : 3][ONE_WORD ? 1 : QMAX + 1];
    auto full_before = [&](int c, unsigned q) -> unsigned { return ONE_WORD ? s_round[c][q] & 0xffffu : s_full[ONE_WORD ? 0 : c][ONE_WORD ? 0 : q]; };
    // Tile offsets of the pruned, the dense and the unified list.  Without a gap between them where CTAs crowd on an SM (the
    // shared memory of three full lists took b = 4 from 109 to 231 us); with their beginnings fixed in the form of few CTAs.
    __shared__ unsigned short s_off[(OWN ? 3 : 1) * kTileRows * NBK];
    const bool has_row = !OWN || r < kTileRows;             // a thread to a row; the others join at the lists
    unsigned P = 0, U = 0, D = 0;
    if (has_row) {
        unsigned long long sgn;
        row_masks(p, NBK, tile, stage, r, &P, &U, &sgn);
        D = ~P & ~U & MASK;
    }
    __shared__ unsigned s_own[3];                           // unified and pruned blocks before the record; its live slices
    if (OWN) {
        if (r < 3) s_own[r] = 0u;
        // whole tiles before this one, then this tile's columns before this record
        unsigned cu = 0, cp = 0;
        const long long words = tile * kTileRows * p.bpr / 32;
        for (long long w = r; w < words; w += NT) {
            const unsigned x = __ldg(p.pruned_bitmap + w), y = __ldg(p.unified_bitmap + w);
            cp += __popc(x);
            cu += __popc(y & ~x);
        }
        const long long n = tile * kTileRows + (r & (kTileRows - 1)), j0 = n * p.bpr, j1 = j0 + stage * NBK;
        if (n < p.rows) {
            for (long long w = (j0 >> 5) + r / kTileRows; w * 32 < j1; w += NT / kTileRows) {
                unsigned m = 0xffffffffu;
                if (w * 32 < j0) m <<= j0 & 31;
                if (w * 32 + 32 > j1) m &= 0xffffffffu >> (32 - (j1 & 31));
                const unsigned x = __ldg(p.pruned_bitmap + w) & m, y = __ldg(p.unified_bitmap + w) & m;
                cp += __popc(x);
                cu += __popc(y & ~x);
            }
        } else if (r < kTileRows) cp += (unsigned)(stage * NBK);             // padding rows are all-pruned
        const unsigned live = __reduce_or_sync(0xffffffffu, has_row ? live_of(P, B) : 0u);
        cu = __reduce_add_sync(0xffffffffu, cu);
        cp = __reduce_add_sync(0xffffffffu, cp);
        __syncthreads();
        if (lane == 0) {
            if (cu) atomicAdd(&s_own[0], cu);
            if (cp) atomicAdd(&s_own[1], cp);
            if (live) atomicOr(&s_own[2], live);
        }
    }
    // Class 0 pruned, 1 dense, 2 unified.  The row's dense and unified blocks as bits of their store slots (a row never has two
    // blocks in one), and the bits of 32 rows turned into a word per (class, slot) with five shuffles (a ballot for each takes
    // three to four times the instructions).
    if (has_row) {
        constexpr int STEP = 16 / STORE;                        // slots of a 16-byte chunk
        if constexpr (G <= 16) {
            unsigned w = D | (U << 16);
            if (B == 16) {                                      // block i: the slots from 2 i on
                w = (w | (w << 2)) & 0x00330033u;
                w = (w | (w << 1)) & 0x00550055u;
            }
            w = warp_transpose(to_slots<STEP>(w, (unsigned)r), lane);      // lane f: dense slot f; lane 16 + f: unified slot f
            const unsigned other = __shfl_xor_sync(0xffffffffu, w, 16);
            const unsigned there = B == 16 ? 0x55555555u << (lane & 1) : 0xffffffffu;
            const int f = lane & 15;
            if (f < G) {
                s_bal[warp][(lane < 16 ? G : 2 * G) + f] = w;
                if (lane < 16) s_bal[warp][f] = there & ~(w | other);
            }
        } else {
            const unsigned d = warp_transpose(to_slots<STEP>(D, (unsigned)r), lane), u = warp_transpose(to_slots<STEP>(U, (unsigned)r), lane);
            s_bal[warp][lane] = ~(d | u);
            s_bal[warp][G + lane] = d;
            s_bal[warp][2 * G + lane] = u;
        }
    }
    __syncthreads();
    // blocks per (class, slot) in the record, and in the warps before each warp (population counts
    // are few to a clock, so each is taken once per CTA, not once per thread)
    for (int t = r; t < 4 * 3 * G; t += (int)NT) {
        const int ww = t / (3 * G), f = t % (3 * G);
        unsigned before = 0;
        for (int w2 = 0; w2 < ww; ++w2) before += __popc(s_bal[w2][f]);
        s_before[ww][f] = (unsigned char)before;
        if (ww == 3) {
            const int c = f / G, sl = f % G;
            s_len[c][(sl % (G / 2)) * 2 + sl / (G / 2)] = (unsigned short)(before + __popc(s_bal[3][f]));
        }
    }
    __syncthreads();
    // round-robin order of a class list: round q takes the q-th block of every slot that has one.
    for (int t = r; t < 3 * (QMAX + 1); t += (int)NT) {
        const int c = t / (QMAX + 1), q = t - c * (QMAX + 1);
        // two slots at a time, in halves of a word
        unsigned full = 0, more = 0;
        const unsigned q2 = (unsigned)q * 0x00010001u;
        const unsigned *len2 = reinterpret_cast<const unsigned *>(s_len[c]);
#pragma unroll
        for (int w = 0; w < G / 2; ++w) {
            const unsigned l2 = len2[w];
            full += __vminu2(l2, q2);
            more |= (~((q2 | 0x80008000u) - l2) & 0x80008000u) >> (15 - w);      // the top bit of a half stays where q >= length
        }
        full = (full & 0xffffu) + (full >> 16);
        more = (more & 0xffffu) | ((more >> 16) << (G / 2));
        if (ONE_WORD) s_round[c][q] = full | (more << 16);
        else {
            s_round[c][q] = more;
            s_full[ONE_WORD ? 0 : c][ONE_WORD ? 0 : q] = (unsigned short)full;
        }
    }
    __syncthreads();

    // every block's place in its class list
    const unsigned first_d = OWN ? kTileRows * NBK : full_before(0, QMAX);
    const unsigned first_u = OWN ? 2 * kTileRows * NBK : first_d + full_before(1, QMAX);
    const unsigned below = (1u << lane) - 1u;
    if (has_row)
#pragma unroll 4
    for (int i = 0; i < NBK; ++i) {
        const unsigned off = tile_offset((unsigned)r, (unsigned)i, B);
        const unsigned slot = (off & 127u) / STORE;
        const unsigned cls = ((U >> i) & 1u) ? 2u : (((D >> i) & 1u) ? 1u : 0u);
        const unsigned f = cls * G + slot;
        // earlier rows with the same class and slot
        const unsigned q = s_before[warp][f] + __popc(s_bal[warp][f] & below);
        // q full rounds before it, then the lower slots of its own round
        const unsigned round = s_round[cls][q];
        const unsigned idx = ONE_WORD ? (round & 0xffffu) + __popc((round >> 16) & ((1u << slot) - 1u))
                                      : full_before((int)cls, q) + __popc(round & ((1u << slot) - 1u));
        s_off[(cls == 0u ? 0u : cls == 1u ? first_d : first_u) + idx] = (unsigned short)off;
    }
    uint4 me, nx;                                           // (ubase, dbase, pbase, live); the table ends with the totals
    if (OWN) {
        __syncthreads();
        me = make_uint4(s_own[0], rec * (unsigned)(kTileRows * NBK) - s_own[0] - s_own[1], s_own[1], s_own[2]);
        nx = make_uint4(me.x + full_before(2, QMAX), me.y + full_before(1, QMAX), me.z + full_before(0, QMAX), 0u);
        uint4 *table = reinterpret_cast<uint4 *>(p.packed + p.L.off_rec);
        if (r == 0) table[rec] = me;
        if (rec == gridDim.x - 1u && r == 0) {
            table[rec + 1] = nx;
            if (nx.x != (unsigned long long)p.L.n_unified || nx.y != (unsigned long long)p.L.n_dense ||
                nx.z != (unsigned long long)p.L.n_plist)
                atomicOr(p.dev_status, (unsigned)MWU_DEV_BOUNDS);
        }
        if (rec == 0u) write_header(p);
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the record table holds the bases
        me = recs[rec];
        nx = recs[rec + 1];
        __syncthreads();
    }

    bool bad = false;
    constexpr unsigned BMASK = (1u << B) - 1u;
    const unsigned len_u = nx.x - me.x, len_d = nx.y - me.y, len_p = nx.z - me.z;
    // the record's three list ranges must lie inside the sections (checked once, not per entry)
    if (len_u + len_d + len_p != (unsigned)(kTileRows * NBK) ||
        (unsigned long long)me.x + len_u > (unsigned long long)p.L.n_unified ||
        (unsigned long long)me.y + len_d > (unsigned long long)p.L.n_dense ||
        (unsigned long long)me.z + len_p > (unsigned long long)p.L.n_plist)
        bad = true;                                          // the table does not describe this record
    else {
        const long long row_base = tile * kTileRows;
        // the record's first block; block i of its row rr is number rr * bpr + i from there on (blocks are fewer than 2^31)
        const long long j_base = row_base * p.bpr + stage * NBK;
        const unsigned bpr = (unsigned)p.bpr;
        const float *Wb = p.W + j_base * B, *Ub = p.U ? p.U + j_base * B : nullptr;
        // pruned blocks: positions only
        unsigned short *pp = ppos + me.z;
        for (unsigned t = (unsigned)r; t < len_p; t += NT) pp[t] = s_off[t];
        // unified blocks: sign bits, position, magnitude
        uint2 *ul = ulist + me.x;
        const float *ub = p.u + j_base;
        const unsigned *sgn = p.sign_bits + j_base * B / 32;    // (a record begins at a multiple of 64 weights)
        // (with four rounds' loads ahead instead of two: 2048 x 2048, b = 4, 50 % / 25 % 16.7 us instead of 16.2, all unified 15.3 / 14.2; 16384 x 4096,
        // all unified, b = 4 93.6 / 83.3, b = 2 145 / 135; with one 102 and 169; b = 8, 4096 x 2048, 50 % / 25 % four 20.9, two 21.3)
#pragma unroll (B <= 4 ? 2 : 4)
        for (unsigned t = (unsigned)r; t < len_u; t += NT) {
            const unsigned off = s_off[first_u + t];
            unsigned rr, i;
            row_block_of(off, B, &rr, &i);
            const unsigned j = rr * bpr + i;
            unsigned sb;
            if (B == 16) sb = __ldg(reinterpret_cast<const unsigned short *>(sgn) + j);
            else if (B == 8) sb = __ldg(reinterpret_cast<const unsigned char *>(sgn) + j);
            else sb = (__ldg(sgn + j / (32 / B)) >> (j % (32 / B) * B)) & BMASK;
            const unsigned mag = (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(__ldg(ub + j)));
            ul[t] = make_uint2(spread_signs(sb), off | (mag << 16));
        }
        // dense blocks: position, then the values, LPB lanes to a block
        unsigned short *dp = dpos + me.y;
        for (unsigned t = (unsigned)r; t < len_d; t += NT) dp[t] = s_off[first_d + t];
        unsigned char *pay = dpay + (unsigned long long)me.y * (2 * B);
        for (unsigned q = (unsigned)r; q < len_d * (unsigned)LPB; q += NT) {
            const unsigned t = q / (unsigned)LPB, part = q % (unsigned)LPB;
            unsigned rr, i;
            row_block_of(s_off[first_d + t], B, &rr, &i);
            const size_t f = (size_t)(rr * bpr + i) * B + part * 4;
            unsigned char *dst = pay + q * 8u;               // = t * 2B + part * 8 when a block takes LPB lanes
            if (B >= 4) {
                float4 a = __ldg(reinterpret_cast<const float4 *>(Wb + f));
                if (Ub) {
                    const float4 d = __ldg(reinterpret_cast<const float4 *>(Ub + f));
                    a.x = __fadd_rn(a.x, d.x); a.y = __fadd_rn(a.y, d.y); a.z = __fadd_rn(a.z, d.z); a.w = __fadd_rn(a.w, d.w);
                }
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w);
                *reinterpret_cast<uint2 *>(dst) = make_uint2(*reinterpret_cast<const unsigned *>(&h0),
                                                             *reinterpret_cast<const unsigned *>(&h1));
            } else {
                float2 a = __ldg(reinterpret_cast<const float2 *>(Wb + f));
                if (Ub) {
                    const float2 d = __ldg(reinterpret_cast<const float2 *>(Ub + f));
                    a.x = __fadd_rn(a.x, d.x); a.y = __fadd_rn(a.y, d.y);
                }
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y);
                *reinterpret_cast<unsigned *>(pay + q * 4u) = *reinterpret_cast<const unsigned *>(&h0);
            }
        }
    }
    if (bad) atomicOr(p.dev_status, (unsigned)MWU_DEV_BOUNDS);
}

}  // namespace pack
}  // namespace mwu

extern "C" size_t mwu_packed_bytes(const mwu_proj_desc *desc) {
    if (mwu::validate_desc(desc, true) != MWU_OK) return 0;
    // a 2-dim block shape is packed through per-row arrays, which mwu_pack builds behind the packed bytes
    const size_t extra = mwu::shape_of(desc).shaped ? mwu::shapes::lowering_bytes(desc) : 0;
    return mwu::packed_layout(desc).total + extra;
}

extern "C" int mwu_pack(const mwu_proj_desc *desc, const float *W, const float *U_dual, const float *u,
                        const uint32_t *pruned_bitmap, const uint32_t *unified_bitmap,
                        const uint32_t *sign_bits, void *packed, size_t packed_bytes,
                        uint32_t *dev_status, void *cuda_stream) {
    using namespace mwu;
    int rc = validate_desc(desc, true);
    if (rc != MWU_OK) return rc;
    if (!W || !u || !pruned_bitmap || !unified_bitmap || !sign_bits || !packed || !dev_status)
        return MWU_ERR_INVALID_ARG;
    if (!aligned_to(W, 16) || !aligned_to(U_dual, 16) || !aligned_to(u, 16) ||
        !aligned_to(pruned_bitmap, 16) || !aligned_to(unified_bitmap, 16) ||
        !aligned_to(sign_bits, 16) || !aligned_to(packed, 256) || !aligned_to(dev_status, 4))
        return MWU_ERR_ALIGNMENT;
    pack::Params p;
    p.L = packed_layout(desc);
    if (packed_bytes < mwu_packed_bytes(desc)) return MWU_ERR_WORKSPACE;
    if (p.L.n_tiles * p.L.n_stages >= (int64_t(1) << 31)) return MWU_ERR_SHAPE;
    int sm_count = 0;
    rc = check_device(&sm_count);
    if (rc != MWU_OK) return rc;
    if (shape_of(desc).shaped) {
        // every run of `block` entries of a row becomes a 1-dim block with its block's class and magnitude
        rc = shapes::lower(desc, u, pruned_bitmap, unified_bitmap, (char *)packed + p.L.total, &u, &pruned_bitmap,
                           &unified_bitmap, sm_count, (cudaStream_t)cuda_stream);
        if (rc != MWU_OK) return rc;
    }
    p.W = W; p.U = U_dual; p.u = u;
    p.pruned_bitmap = pruned_bitmap; p.unified_bitmap = unified_bitmap; p.sign_bits = sign_bits;
    p.packed = (unsigned char *)packed;
    p.dev_status = dev_status;
    p.rows = desc->rows; p.cols = desc->cols; p.b = desc->block;
    p.bpr = desc->cols / desc->block;
    p.n_stages = (unsigned)p.L.n_stages;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // header and the gaps between sections must read as zero: scan_kernel, or fill_kernel where it runs
    // alone, writes all 32 header words and clears the gaps
    const size_t n_rec = (size_t)p.L.n_tiles * p.L.n_stages;
    const size_t gaps[5][2] = {
        {p.L.off_rec + 16 * (n_rec + 1), p.L.off_ulist},
        {p.L.off_ulist + 8 * (size_t)p.L.n_unified, p.L.off_dpos},
        {p.L.off_dpos + 2 * (size_t)p.L.n_dense, p.L.off_dpay},
        {p.L.off_dpay + 2 * (size_t)desc->block * p.L.n_dense, p.L.off_ppos},
        {p.L.off_ppos + 2 * (size_t)p.L.n_plist, p.L.total}};
    for (int g = 0; g < 5; ++g) { p.gap[g][0] = gaps[g][0]; p.gap[g][1] = gaps[g][1] > gaps[g][0] ? gaps[g][1] : gaps[g][0]; }
    // All three start while their predecessor drains (programmatic stream serialization) and wait for its
    // memory themselves.  Up to two units for every team of the scan cluster it counts them itself, in two
    // rounds of loads at most; beyond that a grid of CTAs is faster.
    const long long units = p.L.n_tiles * ((p.L.n_stages + 31) / 32);
    const bool own = (long long)n_rec * (kTileRows * kStageK / desc->block) <= pack::OWN_BLOCKS;
    const int counted = units > 2 * pack::SCAN_CTAS * (pack::SCAN_THREADS / (32 * pack::COUNT_WARPS)) ? 1 : 0;
    cudaError_t e = cudaSuccess;
    const dim3 grid((unsigned)n_rec), block(own ? pack::OWN_THREADS : 128u);
    if (own) {
        switch (desc->block) {
            case 2: e = launch_chained(pack::fill_kernel<2, true>, grid, block, 0, st, 1, p); break;
            case 4: e = launch_chained(pack::fill_kernel<4, true>, grid, block, 0, st, 1, p); break;
            case 8: e = launch_chained(pack::fill_kernel<8, true>, grid, block, 0, st, 1, p); break;
            default: e = launch_chained(pack::fill_kernel<16, true>, grid, block, 0, st, 1, p); break;
        }
        if (e != cudaSuccess) return MWU_ERR_CUDA;
        count_launch(1);
        return cudaGetLastError() == cudaSuccess ? MWU_OK : MWU_ERR_CUDA;
    }
    if (counted) e = launch_chained(pack::count_kernel, dim3((unsigned)units), dim3(32 * pack::COUNT_WARPS), 0, st, 1, p);
    if (e == cudaSuccess)
        e = launch_chained(pack::scan_kernel, dim3(pack::SCAN_CTAS), dim3(pack::SCAN_THREADS), 0, st, pack::SCAN_CTAS, p, counted);
    if (e == cudaSuccess) {
        switch (desc->block) {
            case 2: e = launch_chained(pack::fill_kernel<2, false>, grid, block, 0, st, 1, p); break;
            case 4: e = launch_chained(pack::fill_kernel<4, false>, grid, block, 0, st, 1, p); break;
            case 8: e = launch_chained(pack::fill_kernel<8, false>, grid, block, 0, st, 1, p); break;
            default: e = launch_chained(pack::fill_kernel<16, false>, grid, block, 0, st, 1, p); break;
        }
    }
    if (e != cudaSuccess) return MWU_ERR_CUDA;
    count_launch(2 + counted);
    return cudaGetLastError() == cudaSuccess ? MWU_OK : MWU_ERR_CUDA;
}
