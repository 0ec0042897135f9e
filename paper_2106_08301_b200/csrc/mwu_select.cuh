// Exact selection of the k smallest (key, block index) pairs, twice in a row (prune keys of all
// blocks, then L_u of the survivors), by a team of CTAs that hold the keys themselves.
//
// The selection needs no key in memory: every CTA knows its own blocks' keys (in shared memory, or
// evaluated again each time) and the team only shares counts and a short candidate list:
//   window   every CTA ranks the same few sample blocks and takes the same window around the sample
//            quantile (any window gives the same result: it only steers the first round);
//   round    keys inside the window are counted in equal bins, keys below it in one counter;
//            after a team barrier every CTA finds the bin of the k-th element and that bin becomes
//            the next window.  One round is the rule; a window that missed, or a bin that holds
//            more than XLIST keys, takes another one.  A bin of one single key value that many
//            blocks share is divided further by block index, so ties of any number are exact;
//   gather   the blocks of the final bin are listed; after a team barrier every CTA ranks them
//            (a few dozen, by counting) and knows the threshold element.
// The survivors' first L_u round runs in the prune selection's gather phase; the listed blocks
// that turn out to survive are added by every CTA to its own copy of the counts.  So the usual
// projection has three team barriers.
//
// What bounds it: latency.  A phase is one or two memory round trips, a barrier, and a few hundred
// instructions that every warp of the CTA executes alike, so the team comes in two forms:
//   ClusterTeam  one cluster of sixteen CTAs.  Counts and candidates live in the CTAs' shared memory (a
//                CTA keeps a sixteenth of the bins, candidates are written to all), so a barrier
//                has no L2 update to wait for.
//   GridTeam     a cooperative grid; counts and candidates in global memory, a counter as barrier.
#pragma once

#include "mwu_common.cuh"

namespace mwu {
namespace sel {

typedef unsigned long long u64;

// Candidates that a gather phase may list, and how many it does: every CTA ranks them all, so more of them take longer than another
// round (64 x 64 zeros in 2x2 blocks, 1024 equal keys: 166 us when they were all listed, so 39).
constexpr int XCAP = 896, XLIST = 256;
constexpr int XSAMP_MAX = 128;      // most sample blocks
constexpr int ABOVE = 0x7fffffff;
constexpr int XROUNDS_MAX = 64;     // 63 key bits and 31 index bits at 10 or 11 a round, plus windows that missed
constexpr u64 KEY_END = 1ull << 63; // keys are non-negative doubles
constexpr long long TEAM_WAIT_CYCLES = 4000000000ll;          // about two seconds

// samples of a team whose CTAs have nt threads: two threads or more rank one
__host__ __device__ constexpr int samples_of(int nt) { return nt / 2 < XSAMP_MAX ? nt / 2 : XSAMP_MAX; }

template <typename T>
__device__ __forceinline__ T ld_volatile(const T *p) { return *reinterpret_cast<const volatile T *>(p); }

struct Problem {
    unsigned n_blocks, k_prune, k_unify;
    unsigned by_group;              // the prune class is the bit of the block's group
    int il, ih, ipos;               // prune selection: sample ranks of the window's edges and of the quantile
    float frac_u;                   // share of the survivors that is unified
};

// Ranks of the window's edges and of the quantile among n sample keys: +-3.5 sigma (binomial; root =
// sigma).  A window that misses costs one more round, so the margin need not be generous.
__host__ __device__ inline void window_ranks(int n, float frac, float root, int *il, int *ih, int *ipos) {
    const float pos = frac * (float)n;
    const float margin = 3.5f * root + 2.f;
    const int a = (int)(pos - margin), b = (int)(pos + margin) + 1, c = (int)pos;
    *il = a < 0 ? 0 : (a > n - 1 ? n - 1 : a);
    *ih = b > n - 1 ? n - 1 : b;
    *ipos = c > n - 1 ? n - 1 : c;
}
inline Problem problem_of(int64_t n_blocks, int64_t k_prune, int64_t k_unify, bool by_group, int nt) {
    Problem pb;
    pb.n_blocks = (unsigned)n_blocks;
    pb.k_prune = (unsigned)k_prune;
    pb.k_unify = (unsigned)k_unify;
    pb.by_group = by_group ? 1u : 0u;
    const int ns = (int)(n_blocks < samples_of(nt) ? n_blocks : samples_of(nt));
    const double f = (double)k_prune / (double)n_blocks;
    window_ranks(ns, (float)f, (float)__builtin_sqrt(ns * f * (1.0 - f)), &pb.il, &pb.ih, &pb.ipos);
    pb.frac_u = k_prune < n_blocks ? (float)((double)(k_unify - k_prune) / (double)(n_blocks - k_prune)) : 0.f;
    return pb;
}

// classes: pruned <=> (kp, j) <= (Tp_key, Tp_idx) (mode 0), never (1), always (2), by the group's bit (3);
// unified <=> not pruned and (ku, j) <= (Tu_key, Tu_idx) (mode 0), never (1), always (2)
struct Thresholds {
    unsigned mode_p, mode_u;
    u64 Tp_key, Tu_key;
    unsigned Tp_idx, Tu_idx;

    __device__ __forceinline__ bool pruned(u64 kp, unsigned j, bool group_bit) const {
        if (mode_p == 0u) return kp < Tp_key || (kp == Tp_key && j <= Tp_idx);
        return mode_p == 2u || (mode_p == 3u && group_bit);
    }
    __device__ __forceinline__ bool unified(u64 ku, unsigned j) const {
        if (mode_u == 0u) return ku < Tu_key || (ku == Tu_key && j <= Tu_idx);
        return mode_u == 2u;
    }
};

// A round's window: keys in [lo, hi), or (by_index) the blocks with exactly this key and an index
// in [lo, hi); bin = offset >> shift.
struct Window {
    u64 lo, hi, key;
    unsigned shift;
    bool by_index;

    __device__ __forceinline__ void set_shift(int bin_bits) {
        const u64 span = hi - lo - 1;
        const int width = 64 - __clzll((long long)span);
        shift = width > bin_bits ? (unsigned)(width - bin_bits) : 0u;
    }
    // bin of (k, j), -1 below the window, ABOVE above it
    __device__ __forceinline__ int place(u64 k, unsigned j) const {
        if (by_index) {
            if (k != key) return k < key ? -1 : ABOVE;
            k = j;
        }
        if (k < lo) return -1;
        if (k >= hi) return ABOVE;
        return (int)((k - lo) >> shift);
    }
};

// what a scan of a round's counts found about the k-th element
struct Found {
    int where;                      // -1 below the window, 0 inside, 1 above
    unsigned bin, r, cnt;           // inside: its bin, its rank (1-based) there, the bin's count
};

struct __align__(16) Cand {
    u64 key;
    unsigned idx, pad;
};

// a CTA's shared memory while it selects
struct SelSmem {
    Cand cand[2][XCAP];             // candidates of the two selections
    u64 aux[XCAP];                  // L_u of a prune candidate
    unsigned extra[XCAP];           // bins of the prune candidates that survive
    __align__(16) unsigned samp[XSAMP_MAX];
    unsigned n_extra, n_extra_below;
    unsigned warp_sum[32];
    Found found;
    u64 T_key;
    unsigned T_idx;
    unsigned edge[3];               // sample keys at the window's ranks and at the quantile
};

// ---------------------------------------------------------------------------------------------
// the two teams.  Rounds take three buffers of counts in turn: a buffer is cleared in the round
// before its next use, two barriers after it was last read.
// ---------------------------------------------------------------------------------------------
// Twice the portable limit (a 128 x 1024 projection, b = 4, takes 18.3 us so and 23.2 with eight; where a device cannot place
// sixteen, the grid form serves).
constexpr int CLUSTER_CTAS = 16;

struct ClusterCounts {              // one CTA's share of the counts
    static constexpr int BIN_BITS = 10, BINS = (1 << BIN_BITS) / CLUSTER_CTAS;
    __align__(16) unsigned bins[3][BINS];
    unsigned below[3];              // used in CTA 0
    unsigned cand_count[2];         // used in CTA 0
};

struct ClusterTeam {
    static constexpr int BIN_BITS = ClusterCounts::BIN_BITS, CL_BINS = ClusterCounts::BINS;
    unsigned cta;
    ClusterCounts *mine;
    SelSmem *s;

    __device__ __forceinline__ static unsigned addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
    __device__ __forceinline__ static unsigned in_cta(unsigned local, unsigned c) {
        unsigned r;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(c));
        return r;
    }
    __device__ __forceinline__ static void arrive() {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    __device__ __forceinline__ static void wait() {
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    // before any other call, by the whole CTA; wait() before the first count
    __device__ __forceinline__ void begin() {
        unsigned *w = reinterpret_cast<unsigned *>(mine);
        for (unsigned i = threadIdx.x; i < sizeof(ClusterCounts) / 4; i += blockDim.x) w[i] = 0u;
        arrive();
    }
    __device__ __forceinline__ bool sync() { arrive(); wait(); return true; }
    __device__ __forceinline__ void add(unsigned at, unsigned n) const {
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(at), "r"(n) : "memory");
    }
    __device__ __forceinline__ void count(unsigned buf, int bin) const {
        add(in_cta(addr(&mine->bins[buf][bin & (CL_BINS - 1)]), (unsigned)bin / CL_BINS), 1u);
    }
    __device__ __forceinline__ void count_below(unsigned buf, unsigned n) const { add(in_cta(addr(&mine->below[buf]), 0u), n); }
    __device__ __forceinline__ void flush(unsigned) const {}
    __device__ __forceinline__ void clear(unsigned buf) const {
        for (unsigned i = threadIdx.x; i < CL_BINS; i += blockDim.x) mine->bins[buf][i] = 0u;
        if (threadIdx.x == 0) mine->below[buf] = 0u;
    }
    // this thread's PER bins of a finished round, and the keys below its window
    template <int PER>
    __device__ __forceinline__ unsigned read(unsigned buf, unsigned (&c)[PER]) const {
        static_assert(PER % 2 == 0 && CL_BINS % PER == 0, "whole vector loads from one CTA");
        const unsigned bin = threadIdx.x * PER;
        const unsigned at = in_cta(addr(&mine->bins[buf][bin % CL_BINS]), bin / CL_BINS);
#pragma unroll
        for (int i = 0; i < PER; i += 2)
            asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(c[i]), "=r"(c[i + 1]) : "r"(at + i * 4) : "memory");
        unsigned below;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(below) : "r"(in_cta(addr(&mine->below[buf]), 0u)) : "memory");
        return below;
    }
    // a candidate goes to the lists of all CTAs
    __device__ __forceinline__ void list(int which, u64 key, unsigned idx, u64 aux) const {
        unsigned slot;
        asm volatile("atom.relaxed.cluster.shared::cluster.add.u32 %0, [%1], 1;"
                     : "=r"(slot) : "r"(in_cta(addr(&mine->cand_count[which]), 0u)) : "memory");
        if (slot >= (unsigned)XCAP) return;
        const unsigned ac = addr(&s->cand[which][slot]), aa = addr(&s->aux[slot]);
#pragma unroll 1
        for (unsigned c = 0; c < CLUSTER_CTAS; ++c) {
            asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(in_cta(ac, c)), "l"(key), "l"((u64)idx) : "memory");
            if (which == 0) asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(in_cta(aa, c)), "l"(aux) : "memory");
        }
    }
    __device__ __forceinline__ void fetch_list(int, unsigned) const {}       // it is here already
};

// Copies of a round's counts, interleaved bin by bin; a CTA counts in one of them.  L2 takes atomics on
// one 128-byte line one after the other, and a grid's counts crowd on a few lines: 1 M blocks on 148
// CTAs took 10 us to count with one copy.
constexpr int XCOPIES = 4;
constexpr int GRID_BIN_BITS = 11, GRID_BINS = 1 << GRID_BIN_BITS;

// GridTeam's state in global memory; the part up to cand_key starts at zero.
struct XWork {
    unsigned bar;                   // arrivals at the barriers (only ever grows)
    unsigned cand_count[2];
    unsigned pad;
    unsigned hist[3][(GRID_BINS + 1) * XCOPIES];    // bin GRID_BINS: keys below the window
    Cand cand[2][XCAP];
    u64 aux[XCAP];
};
constexpr size_t XWORK_ZERO_BYTES = offsetof(XWork, cand);
static_assert(XWORK_ZERO_BYTES % 16 == 0 && offsetof(XWork, hist) % 16 == 0 && XCOPIES == 4, "16-byte accesses");

// LOCAL: a CTA counts in shared memory first (`local`: GRID_BINS words, cleared).  (Projections given up by
// the one pass, 4096 x 4096, b = 4: zeros 7650 us counted in L2, 620 so; 16384 x 4096, b = 4, projected once more 35900, 3660.)
template <bool LOCAL>
struct GridTeam {
    static constexpr int BIN_BITS = GRID_BIN_BITS;
    unsigned cta, n_cta;
    XWork *x;
    SelSmem *s;
    unsigned k;                     // barriers passed
    unsigned *local;

    // All threads of all CTAs call it; what was written before is visible after.  False when the
    // bounded wait ran out (the caller raises MWU_DEV_TIMEOUT and leaves).
    __device__ __forceinline__ bool sync() {
        __shared__ int s_ok;
        ++k;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&x->bar, 1u);
            const unsigned target = k * n_cta;
            int ok = 1;
            const long long t0 = clock64();
            unsigned spins = 0;
            while (ld_volatile(&x->bar) < target) {
                if ((++spins & 63u) == 0u && clock64() - t0 > TEAM_WAIT_CYCLES) { ok = 0; break; }
            }
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    }
    __device__ __forceinline__ void count(unsigned buf, int bin) const {
        if (LOCAL) atomicAdd(&local[bin], 1u);
        else atomicAdd(&x->hist[buf][bin * XCOPIES + (cta & 3u)], 1u);
    }
    // the counts of this CTA, before the barrier that ends their round
    __device__ __forceinline__ void flush(unsigned buf) const {
        if (!LOCAL) return;
        __syncthreads();
        for (unsigned i = threadIdx.x; i < (unsigned)GRID_BINS; i += blockDim.x) {
            const unsigned n = local[i];
            if (n) { atomicAdd(&x->hist[buf][i * XCOPIES + (cta & 3u)], n); local[i] = 0u; }
        }
    }
    __device__ __forceinline__ void count_below(unsigned buf, unsigned n) const {
        atomicAdd(&x->hist[buf][GRID_BINS * XCOPIES + (cta & 3u)], n);
    }
    __device__ __forceinline__ void clear(unsigned buf) const {
        uint4 *z = reinterpret_cast<uint4 *>(x->hist[buf]);
        for (unsigned i = cta * blockDim.x + threadIdx.x; i < (unsigned)GRID_BINS + 1u; i += n_cta * blockDim.x) z[i] = make_uint4(0, 0, 0, 0);
    }
    template <int PER>
    __device__ __forceinline__ unsigned read(unsigned buf, unsigned (&c)[PER]) const {
        const uint4 *h = reinterpret_cast<const uint4 *>(x->hist[buf]);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const uint4 v = __ldcg(h + threadIdx.x * PER + i);
            c[i] = v.x + v.y + v.z + v.w;
        }
        const uint4 v = __ldcg(h + GRID_BINS);
        return v.x + v.y + v.z + v.w;
    }
    __device__ __forceinline__ void list(int which, u64 key, unsigned idx, u64 aux) const {
        const unsigned slot = atomicAdd(&x->cand_count[which], 1u);
        if (slot >= (unsigned)XCAP) return;
        const Cand c = {key, idx, 0u};
        x->cand[which][slot] = c;
        if (which == 0) x->aux[slot] = aux;
    }
    __device__ __forceinline__ void fetch_list(int which, unsigned m) const {
        for (unsigned i = threadIdx.x; i < m; i += blockDim.x) {
            *reinterpret_cast<uint4 *>(&s->cand[which][i]) = __ldcg(reinterpret_cast<const uint4 *>(&x->cand[which][i]));
            if (which == 0) s->aux[i] = __ldcg(&x->aux[i]);
        }
    }
};

// ---------------------------------------------------------------------------------------------
// steps every CTA takes alike (functions of their own: each is needed twice, and a launch runs
// them once out of a cold instruction cache)
// ---------------------------------------------------------------------------------------------
// The k-th smallest of a finished round (counts in buffer buf; s.n_extra more in the bins s.extra[] and
// s.n_extra_below below the window) -> s.found.
template <int NT, class TeamT>
__device__ __noinline__ void scan_round(const TeamT &team, unsigned buf, unsigned k, SelSmem &s) {
    constexpr int PER = (1 << TeamT::BIN_BITS) / NT;
    unsigned c[PER];
    const unsigned below = team.read(buf, c) + s.n_extra_below;
    const unsigned n_extra = s.n_extra;
#pragma unroll 1
    for (unsigned x = 0; x < n_extra; ++x) {
        const unsigned b = s.extra[x] - threadIdx.x * PER;
        if (b < (unsigned)PER) {
#pragma unroll
            for (int i = 0; i < PER; ++i) c[i] += (b == (unsigned)i) ? 1u : 0u;
        }
    }
    unsigned sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) sum += c[i];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned incl = sum;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, m);
        if (lane >= m) incl += y;
    }
    if (lane == 31) s.warp_sum[wid] = incl;
    if (threadIdx.x == 0) s.found.where = k <= below ? -1 : 1;
    __syncthreads();
    // counts of the warps before this one
    const unsigned t = lane < wid ? s.warp_sum[lane] : 0u;
    unsigned run = below + __reduce_add_sync(0xffffffffu, t) + incl - sum;
    if (run < k && k <= run + sum) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (run < k && k <= run + c[i]) {
                s.found.where = 0;
                s.found.bin = threadIdx.x * PER + i;
                s.found.r = k - run;
                s.found.cnt = c[i];
            }
            run += c[i];
        }
    }
    __syncthreads();
}

// the next window after a round; false when nothing can lie in it (an inconsistent count)
__device__ __forceinline__ bool narrow(Window &w, const Found &f, unsigned n_blocks, int bin_bits) {
    if (f.where < 0) { w.hi = w.lo; w.lo = 0; }
    else if (f.where > 0) { w.lo = w.hi; w.hi = w.by_index ? (u64)n_blocks : KEY_END; }
    else {
        const u64 base = w.lo + ((u64)f.bin << w.shift);
        const u64 end = base + (1ull << w.shift);
        w.lo = base;
        if (end < w.hi) w.hi = end;
        if (!w.by_index && f.cnt > (unsigned)XLIST && w.hi - w.lo == 1) {
            w.by_index = true;              // one key value shared by many blocks: go on by index
            w.key = w.lo;
            w.lo = 0;
            w.hi = n_blocks;
        }
    }
    if (w.lo >= w.hi) return false;
    w.set_shift(bin_bits);
    return true;
}

// Sample keys are held as sortable words: the top 24 bits of the float below its (clear) sign bit
// with the sample's number in the low byte, so all are distinct; 0xffffffff: not valid.
__device__ __forceinline__ unsigned samp_word(float key, unsigned i) { return ((__float_as_uint(key) >> 7) << 8) | i; }

// The window between the sample keys of ranks il and ih; s.edge[2] becomes the key of rank ipos.
template <int NT>
__device__ __noinline__ Window sample_window(int il, int ih, int ipos, int n_valid, int bin_bits, SelSmem &s) {
    constexpr int NS = samples_of(NT), PARTS = NT / NS;
    const int a = threadIdx.x / PARTS, part = threadIdx.x % PARTS;
    const unsigned k = s.samp[a];
    int r = 0;
    const uint4 *q = reinterpret_cast<const uint4 *>(s.samp) + part;
#pragma unroll 4
    for (int t = 0; t < NS / 4 / PARTS; ++t) {
        const uint4 x = q[PARTS * t];
        r += (x.x < k ? 1 : 0) + (x.y < k ? 1 : 0) + (x.z < k ? 1 : 0) + (x.w < k ? 1 : 0);
    }
#pragma unroll
    for (int m = 1; m < PARTS; m <<= 1) r += __shfl_xor_sync(0xffffffffu, r, m);
    if (part == 0) {
        if (r == il) s.edge[0] = k;
        if (r == ih) s.edge[1] = k;
        if (r == ipos) s.edge[2] = k;
    }
    __syncthreads();
    Window w;
    w.by_index = false;
    w.key = 0;
    // at the ends of the sample the window reaches a factor of four beyond the sample's own range
    const unsigned e0 = s.edge[0], e1 = s.edge[1];
    const u64 quarter = 2ull << 52;
    w.lo = (u64)__double_as_longlong((double)__uint_as_float((e0 >> 8) << 7));
    w.hi = (u64)__double_as_longlong((double)__uint_as_float(((e1 >> 8) + 1u) << 7));
    if (il == 0) w.lo = w.lo > quarter ? w.lo - quarter : 0;
    if (ih == n_valid - 1) w.hi += quarter;
    if (e0 == 0xffffffffu || w.lo >= KEY_END - 1) w.lo = 0;
    if (w.hi <= w.lo || w.hi > KEY_END || e1 == 0xffffffffu) w.hi = KEY_END;
    w.set_shift(bin_bits);
    return w;
}

// Of the m candidates in list `which` the one of rank r (1-based) by (key, index) becomes s.T_key / s.T_idx.
// As many threads as there are for each candidate (a power of two up to a warp) share its comparisons.
template <int NT, class TeamT>
__device__ __noinline__ void rank_candidates(const TeamT &team, int which, unsigned m, unsigned r, SelSmem &s) {
    team.fetch_list(which, m);
    if (threadIdx.x == 0) { s.T_key = ~0ull >> 1; s.T_idx = 0xffffffffu; }
    __syncthreads();
    const uint4 *cand = reinterpret_cast<const uint4 *>(s.cand[which]);
    const unsigned lg = m * 32u <= (unsigned)NT ? 5u : (m * 8u <= (unsigned)NT ? 3u : (m * 2u <= (unsigned)NT ? 1u : 0u));
    const unsigned parts = 1u << lg, part = threadIdx.x & (parts - 1u), per_warp = 32u >> lg;
#pragma unroll 1
    for (unsigned i = threadIdx.x >> lg; i < ((m + per_warp - 1u) & ~(per_warp - 1u)); i += NT >> lg) {      // whole warps stay together
        const uint4 c = cand[i < m ? i : 0u];
        unsigned rank = 0;
        // (key, index) < (key, index) as the borrow of a 96-bit subtraction
#pragma unroll 4
        for (unsigned t = part; t < m; t += parts) {
            const uint4 y = cand[t];
            unsigned borrow;
            asm("{\n\t.reg .u32 d;\n\tsub.cc.u32 d, %1, %4;\n\tsubc.cc.u32 d, %2, %5;\n\tsubc.cc.u32 d, %3, %6;\n\tsubc.u32 %0, 0, 0;\n\t}"
                : "=r"(borrow) : "r"(y.z), "r"(y.x), "r"(y.y), "r"(c.z), "r"(c.x), "r"(c.y));
            rank -= borrow;
        }
        for (unsigned w = 1; w < parts; w <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, w);
        if (i < m && part == 0u && rank + 1u == r) { s.T_key = (u64)c.y << 32 | c.x; s.T_idx = c.z; }
    }
    __syncthreads();
}

// The selection.  Src:
//   src.for_blocks(f)          f(j, kp, ku) for every block of this thread; a slot without a block
//                              has both keys ~0 (never inside or below a window)
//   src.in_group(j)            grouped pruning: the bit of the block's group
// samp_p, samp_u: approximate keys of this thread's sample block (sample_block_of), samp_ok: it has one
// and that block is in no pruned group.
// Returns false when a barrier's wait ran out.  *dev_status gets MWU_DEV_SELECT when the counts are
// inconsistent (non-finite input); the thresholds are then arbitrary.
template <int NT, class Src, class TeamT>
__device__ bool select_exact(const Src &src, TeamT &team, SelSmem &s, const Problem &pb, float samp_p, float samp_u,
                             bool samp_ok, unsigned *dev_status, Thresholds &T) {
    const unsigned ksel = pb.k_unify - pb.k_prune, elig = pb.n_blocks - pb.k_prune;
    const unsigned mode_p = pb.by_group ? 3u : (pb.k_prune == 0u ? 1u : (pb.k_prune == pb.n_blocks ? 2u : 0u));
    const unsigned mode_u = ksel == 0u ? 1u : (ksel == elig ? 2u : 0u);
    T.mode_p = mode_p;
    T.mode_u = mode_u;
    T.Tp_key = T.Tu_key = ~0ull >> 1;
    T.Tp_idx = T.Tu_idx = 0xffffffffu;
    if (mode_p != 0u && mode_u != 0u) return true;        // the same in every CTA
    const int lane = threadIdx.x & 31;

    // windows
    Window wp, wu;
    {
        constexpr unsigned NS = (unsigned)samples_of(NT);
        constexpr int BITS = TeamT::BIN_BITS;
        if (threadIdx.x < NS) s.samp[threadIdx.x] = samp_ok ? samp_word(samp_p, threadIdx.x) : 0xffffffffu;
        if (threadIdx.x == 0) { s.n_extra = s.n_extra_below = 0; s.edge[0] = s.edge[1] = s.edge[2] = 0xffffffffu; }
        if (mode_p == 0u) {
            __syncthreads();
            wp = sample_window<NT>(pb.il, pb.ih, pb.ipos, pb.n_blocks < NS ? (int)pb.n_blocks : (int)NS, BITS, s);
            // the samples that survive the estimated prune threshold
            samp_ok = samp_ok && samp_word(samp_p, threadIdx.x) > s.edge[2];
            __syncthreads();
        }
        if (mode_u == 0u) {
            if (threadIdx.x < NS) s.samp[threadIdx.x] = samp_ok ? samp_word(samp_u, threadIdx.x) : 0xffffffffu;
            if (threadIdx.x == 0) s.edge[0] = s.edge[1] = s.edge[2] = 0xffffffffu;
            const int n_valid = max(__syncthreads_count(samp_ok), 1);
            float root = (float)n_valid * pb.frac_u * (1.f - pb.frac_u);
            asm("sqrt.approx.f32 %0, %0;" : "+f"(root));
            int il, ih, ipos;
            window_ranks(n_valid, pb.frac_u, root, &il, &ih, &ipos);
            wu = sample_window<NT>(il, ih, ipos, n_valid, BITS, s);
        }
    }

    unsigned rnd = 0, buf = 0;                            // buf = rnd % 3
    auto next_of = [](unsigned b) { return b == 2u ? 0u : b + 1u; };
    // ends a round's counting
    auto end_round = [&](unsigned below) -> bool {
        below = __reduce_add_sync(0xffffffffu, below);
        if (lane == 0 && below) team.count_below(buf, below);
        team.flush(buf);
        team.clear(next_of(buf));
        return team.sync();
    };
    bool fine = true;

    if (mode_p == 0u) {
        unsigned r = 0, cnt = 0;
#pragma unroll 1
        for (;;) {
            unsigned below = 0;
            src.for_blocks([&](unsigned j, u64 kp, u64) {
                const int b = wp.place(kp, j);
                if (b < 0) ++below;
                else if (b != ABOVE) team.count(buf, b);
            });
            if (!end_round(below)) return false;
            scan_round<NT>(team, buf, pb.k_prune, s);
            const Found f = s.found;
            ++rnd;
            buf = next_of(buf);
            r = f.r;
            cnt = f.cnt;
            if (!narrow(wp, f, pb.n_blocks, TeamT::BIN_BITS) || rnd > (unsigned)XROUNDS_MAX) { fine = false; break; }
            if (f.where == 0 && f.cnt <= (unsigned)XLIST) break;
        }
        if (fine) {
            // candidates of the threshold bin; the survivors' first L_u round
            unsigned below = 0;
            src.for_blocks([&](unsigned j, u64 kp, u64 ku) {
                const int b = wp.place(kp, j);
                if (b < 0) return;
                if (b != ABOVE) { team.list(0, kp, j, ku); return; }
                if (mode_u != 0u) return;
                const int bu = wu.place(ku, j);
                if (bu < 0) ++below;
                else if (bu != ABOVE) team.count(buf, bu);
            });
            if (!end_round(below)) return false;
            rank_candidates<NT>(team, 0, cnt, r, s);
            T.Tp_key = s.T_key;
            T.Tp_idx = s.T_idx;
            if (mode_u == 0u) {
                // the candidates that survive count for L_u: kept here as corrections to the counts
                for (unsigned i = threadIdx.x; i < cnt; i += NT) {
                    if (!T.pruned(s.cand[0][i].key, s.cand[0][i].idx, false)) {
                        const int bu = wu.place(s.aux[i], s.cand[0][i].idx);
                        if (bu < 0) atomicAdd(&s.n_extra_below, 1u);
                        else if (bu != ABOVE) s.extra[atomicAdd(&s.n_extra, 1u)] = (unsigned)bu;
                    }
                }
                __syncthreads();
            }
        }
    }
    if (fine && mode_u == 0u) {
        auto survives = [&](unsigned j, u64 kp) { return !T.pruned(kp, j, mode_p == 3u && src.in_group(j)); };
        unsigned r = 0, cnt = 0;
        bool counted = mode_p == 0u;                      // the first round has run (above)
#pragma unroll 1
        for (;;) {
            if (!counted) {
                unsigned below = 0;
                src.for_blocks([&](unsigned j, u64 kp, u64 ku) {
                    const int b = wu.place(ku, j);
                    if (b == ABOVE || !survives(j, kp)) return;
                    if (b < 0) ++below;
                    else team.count(buf, b);
                });
                if (threadIdx.x == 0) s.n_extra = s.n_extra_below = 0;        // this round knows the prune threshold
                if (!end_round(below)) return false;
            }
            counted = false;
            scan_round<NT>(team, buf, ksel, s);
            const Found f = s.found;
            ++rnd;
            buf = next_of(buf);
            r = f.r;
            cnt = f.cnt;
            if (!narrow(wu, f, pb.n_blocks, TeamT::BIN_BITS) || rnd > 2u * (unsigned)XROUNDS_MAX) { fine = false; break; }
            if (f.where == 0 && f.cnt <= (unsigned)XLIST) break;
        }
        if (fine) {
            src.for_blocks([&](unsigned j, u64 kp, u64 ku) {
                const int b = wu.place(ku, j);
                if (b < 0 || b == ABOVE || !survives(j, kp)) return;
                team.list(1, ku, j, 0ull);
            });
            if (!team.sync()) return false;
            rank_candidates<NT>(team, 1, cnt, r, s);
            T.Tu_key = s.T_key;
            T.Tu_idx = s.T_idx;
        }
    }
    if (!fine) {
        // all CTAs come here alike; nobody goes on while another still reads this CTA's counts
        if (team.cta == 0 && threadIdx.x == 0) atomicOr(dev_status, (unsigned)MWU_DEV_SELECT);
        return team.sync();
    }
    return true;
}

// block of a thread's sample: evenly spaced blocks (all of them when there are fewer)
template <int NT>
__device__ __forceinline__ bool sample_block_of(const Problem &pb, unsigned tid, unsigned *j) {
    constexpr unsigned NS = (unsigned)samples_of(NT);
    *j = 0u;
    if (tid >= NS || tid >= pb.n_blocks) return false;
    *j = pb.n_blocks >= NS ? (unsigned)(((u64)tid * pb.n_blocks) / NS) : tid;
    return true;
}

}  // namespace sel
}  // namespace mwu
