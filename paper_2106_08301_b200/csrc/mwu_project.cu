// mwu_project: Q = Unify(W + U), the Q-step of ADMM (Algorithm 1, Eq. 7) for 1-D micro-blocks.
//
// Two pipelines give the same bits (all on the caller's stream, no host synchronisation).
//
// Exact pipeline (exact_kernel; small tensors, and every tensor with MWU_ALGO_MULTI_PASS): one launch.
// A team of CTAs reads W (+U) once, keeps the fp64 keys of its blocks (Section 3.1: q = mean|v|,
// L_u = sum(|v|-q)^2, L_p = sum v^2, fixed pairwise trees) in shared memory, finds both exact
// thresholds (mwu_select.cuh) and writes every output.  Tensors whose keys do not fit evaluate them
// again in every phase (exact_walk_kernel).
//
// One-pass pipeline (MWU_ALGO_ONE_PASS; the default for larger tensors):
//   sample_keys_kernel, sample_kernel
//                   rank the keys of <= 262144 evenly spaced blocks; for each selection (prune key, L_u
//                   of the survivors) the sample quantile is a provisional threshold and the sample
//                   keys 4 sigma of rank to either side a window.
//   pass_kernel     streams W (+U) once, evaluates fp32 keys of bounded error for every block (fp64 keys for
//                   those near a window's edge or inside it) and writes every
//                   output -- Q, u, sign plane, bitmaps -- with the class the provisional
//                   thresholds give.  A block whose key lies outside the window has its final class
//                   (as long as the exact threshold lies inside, which the counts prove afterwards);
//                   the few per cent inside go to a candidate list with their bin codes and into
//                   the window histograms.
//   resolve_kernel  exact thresholds from the window histograms and the list; rewrites the outputs of
//                   the listed blocks whose class changed.
//   If a count shows that a threshold lies outside its window (or a tie group overflows the
//   sort buffer, or the list overflows) a flag is set and the same launch redoes the projection with
//   the exact pipeline's phases.
#include <type_traits>

#include "mwu_blocks.cuh"
#include "mwu_select.cuh"

namespace mwu {
namespace proj {

constexpr int NB_MAX = 65536;   // level-0 bins (codes fit 16 bits): bin 0 = below the window, nb-1 = above it
constexpr int NB_SMALL = 8192;  // used up to NB_SMALL_BLOCKS blocks: fewer bins to clear and scan
constexpr long long NB_SMALL_BLOCKS = 1ll << 27;    // about 1.4 % of them in a window: at most 450 to a bin
constexpr int CAP = 2048;       // candidates sorted by the last step
// sample blocks ranked by sample_kernel: SAMP_PER to a thread at a time
constexpr int SAMP_CTAS = 8, SAMP_THREADS = 1024, SAMP_PER = 8;
constexpr int SAMP_ROUND = SAMP_CTAS * SAMP_THREADS * SAMP_PER;
constexpr int SAMP_A = 128;       // of the samples, ranked first
constexpr int NSAMP_SMALL_LG = 14, NSAMP_LG = 16, NSAMP_LARGE_LG = 18;
static_assert(SAMP_ROUND == 1 << NSAMP_LG, "the middle sample fills the cluster");
constexpr int STAGE_ENTRIES = 64;  // per-warp staging of candidate-list entries in pass_kernel
constexpr int FIN_THREADS = 1024;   // block size of the kernels that scan the histograms
constexpr int PASS_GROUPS = 8;      // groups of CTAs of pass_kernel that share out its last steps

typedef unsigned long long u64;
typedef unsigned __int128 u128;

struct Sel {
    u64 lo0, hi0;               // level-0 window on the key's bit pattern
    unsigned shift0;
    unsigned mode;              // 0: threshold, 1: nothing selected, 2: everything eligible selected
    u64 k;                      // how many to select
    unsigned B;                 // level-0 bin that holds the threshold element
    unsigned pad0;
    u64 r;                      // rank (1-based) of the threshold element inside [lo, hi)
    u64 cnt;                    // eligible elements inside [lo, hi)
    u64 lo_hi, lo_lo, hi_hi, hi_lo;   // composite (key << 32 | index) range, as two 64-bit halves
    u64 T_key, T_idx;           // selected  <=>  (key, index) <= (T_key, T_idx)
};

// Windows and provisional thresholds for pass_kernel's fp32 keys: a block whose keys lie outside [lo, hi) has its
// final class.  The edges are moved outwards by what an fp32 key may differ from the exact one (make_filter).
struct Filter {
    float plo, phi, pt;         // prune key: window, threshold
    float ulo, uhi, ut;         // L_u
};

struct Work {
    Sel sel[2];                 // 0: prune, 1: unify
    Filter filter;
    // one-pass pipeline
    unsigned fcand_count[2];    // threshold-bin candidates of the two halves of resolve_kernel
    unsigned list_count;        // entries appended to the candidate list
    unsigned failed;            // != 0: the one-pass result is void, the exact phases run
    u64 That[2];                // provisional thresholds (key bit patterns)
    unsigned bar;               // resolve_kernel: arrivals at its grid barriers (only ever grows)
    unsigned pad1[2];
    struct __align__(128) { unsigned ticket; } group[PASS_GROUPS];      // pass_kernel: steps of its last part given out to a group of CTAs
};

struct Params {
    const float *W;
    const float *U;
    long long n_floats;         // rows * cols
    long long n_blocks;
    int b;
    int use_l1;
    Work *work;
    int nb;                     // level-0 bins in use (NB_SMALL or NB_MAX)
    sel::XWork *xwork;          // team state of the exact phases
    unsigned *fhist;            // [2][nb]: prune, unify (one-pass kernels)
    uint2 *list;                // [list_cap] candidate list: (block index, bin codes)
    unsigned list_cap;
    // grouped pruning: the prune class of a block is the bit of its group (nullptr: pruning by key)
    const unsigned *gprune;     // [ceil(n_groups / 32)]
    unsigned group_rows, group_cols;     // extent of a prune group in rows and columns of W
    unsigned blocks_per_row;    // cols / b
    unsigned groups_per_row;    // cols / group_cols
    long long k_unify, k_prune;
    float *U_next;              // dual update V - Q (mwu_admm_step), else null
    double *resid;              // ||V - Q||_F^2 accumulator (mwu_admm_step), else null
    u64 *cand_key;              // [CAP]
    unsigned *cand_idx;         // [2 * CAP]
    unsigned *cand_aux;         // [2 * CAP] what resolve_kernel wants to know about a candidate besides its key
    float2 *samp;               // [n_samp] prune key and L_u of the sample blocks (one-pass pipeline; in the list's memory)
    int n_samp, samp_lg;        // their number; its logarithm, or -1: every block is a sample
    unsigned *dev_status;
};

__device__ __forceinline__ u128 make_c(u64 key, u64 idx) { return ((u128)key << 32) | (u128)idx; }
__device__ __forceinline__ u128 from_halves(u64 hi, u64 lo) { return ((u128)hi << 64) | (u128)lo; }

__device__ __forceinline__ unsigned bin_of(u64 key, u64 lo0, u64 hi0, unsigned shift0, unsigned nb) {
    if (key < lo0) return 0u;
    if (key >= hi0) return nb - 1u;
    return 1u + (unsigned)((key - lo0) >> shift0);
}

template <typename T>
__device__ __forceinline__ T ld_vol(const T *p) { return *reinterpret_cast<const volatile T *>(p); }

// Fresh copy of the selection state in shared memory, made by the whole CTA.  Inside a kernel that
// spans several phases (grid barriers between them) plain loads of words another CTA has written
// may be served from a stale L1 line, so every phase reads its own copy, taken with volatile loads.
__device__ __forceinline__ void load_work(const Work *g, Work *s) {
    __syncthreads();
    const volatile unsigned *src = reinterpret_cast<const volatile unsigned *>(g);
    unsigned *dst = reinterpret_cast<unsigned *>(s);
    for (unsigned i = threadIdx.x; i < sizeof(Work) / 4; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
}

// grouped pruning: is block j inside a pruned group?
__device__ __forceinline__ bool group_pruned(const Params &p, unsigned j) {
    const unsigned row = j / p.blocks_per_row, kb = j - row * p.blocks_per_row;
    const unsigned g = (row / p.group_rows) * p.groups_per_row + (kb * (unsigned)p.b) / p.group_cols;
    return (__ldg(p.gprune + (g >> 5)) >> (g & 31u)) & 1u;
}

// Barrier over all CTAs of a cooperative launch (all resident at once).  `counter` only grows:
// the k-th barrier of a kernel is passed when it reaches k * gridDim.x.  The wait is bounded: when
// it runs out the caller raises MWU_DEV_TIMEOUT and leaves.
constexpr long long GRID_WAIT_CYCLES = 4000000000ll;          // about two seconds
__device__ __forceinline__ bool grid_sync(unsigned *counter, unsigned k) {
    __shared__ int s_grid_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(counter, 1u);
        const unsigned target = k * gridDim.x;
        int ok = 1;
        const long long t0 = clock64();
        unsigned spins = 0;
        while (ld_vol(counter) < target) {
            if ((++spins & 63u) == 0u && clock64() - t0 > GRID_WAIT_CYCLES) { ok = 0; break; }
        }
        __threadfence();
        s_grid_ok = ok;
    }
    __syncthreads();
    return s_grid_ok != 0;
}

__device__ __forceinline__ float load_v(const float *W, const float *U, long long f) {
    float w = __ldg(W + f);
    if (U) w = __fadd_rn(w, __ldg(U + f));
    return w;
}

// the B values of block j with the widest loads its alignment allows (a block starts at a
// multiple of 4*B bytes): scalar loads of scattered blocks cost one cache-line lookup per value
template <int B>
__device__ __forceinline__ void load_block(const float *W, const float *U, long long j, float (&v)[B]) {
    if (B == 2) {
        float2 a = __ldg(reinterpret_cast<const float2 *>(W) + j);
        if (U) {
            const float2 d = __ldg(reinterpret_cast<const float2 *>(U) + j);
            a.x = __fadd_rn(a.x, d.x); a.y = __fadd_rn(a.y, d.y);
        }
        v[0] = a.x; v[1 % B] = a.y;
    } else {
#pragma unroll
        for (int c = 0; c < B / 4; ++c) {
            float4 a = __ldg(reinterpret_cast<const float4 *>(W) + j * (B / 4) + c);
            if (U) {
                const float4 d = __ldg(reinterpret_cast<const float4 *>(U) + j * (B / 4) + c);
                a.x = __fadd_rn(a.x, d.x); a.y = __fadd_rn(a.y, d.y); a.z = __fadd_rn(a.z, d.z); a.w = __fadd_rn(a.w, d.w);
            }
            v[(4 * c) % B] = a.x; v[(4 * c + 1) % B] = a.y; v[(4 * c + 2) % B] = a.z; v[(4 * c + 3) % B] = a.w;
        }
    }
}

// Approximate keys of block j in fp32, for the sample only: the sample steers the windows (any
// window gives the same result), so its keys need no more than a few good digits.
template <int B>
__device__ __forceinline__ void block_keys_sample(const float *W, const float *U, long long j, int use_l1, float *kp,
                                                  float *ku) {
    float v[B];
    load_block<B>(W, U, j, v);
    float S = 0.f, sq = 0.f;
#pragma unroll
    for (int l = 0; l < B; ++l) { S += fabsf(v[l]); sq = fmaf(v[l], v[l], sq); }
    const float q = S * (1.f / (float)B);
    float lu = 0.f;
#pragma unroll
    for (int l = 0; l < B; ++l) { const float d = fabsf(v[l]) - q; lu = fmaf(d, d, lu); }
    *kp = use_l1 ? S : sq;
    *ku = lu;
}

// exact keys of block j, read from global memory (threshold-bin blocks)
template <int B>
__device__ __forceinline__ void block_keys_at(const float *W, const float *U, long long j, int use_l1,
                                              double *S, double *Lu, double *Kp) {
    float v[B];
    load_block<B>(W, U, j, v);
    block_keys<B>(v, use_l1, S, Lu, Kp);
}

// which: 0 -> prune key, 1 -> L_u
template <int B>
__device__ __forceinline__ u64 exact_key(const Params &p, long long j, int which) {
    double S, Lu, Kp;
    block_keys_at<B>(p.W, p.U, j, p.use_l1, &S, &Lu, &Kp);
    return key_bits(which ? Lu : Kp);
}

// 16 consecutive floats starting at f (f % 16 == 0); zero beyond n
__device__ __forceinline__ void load16(const float *W, const float *U, long long f, long long n, float (&v)[16]) {
    if (f + 16 <= n) {
        const float4 *src = reinterpret_cast<const float4 *>(W + f);
        float4 a0 = __ldg(src), a1 = __ldg(src + 1), a2 = __ldg(src + 2), a3 = __ldg(src + 3);
        if (U) {
            const float4 *du = reinterpret_cast<const float4 *>(U + f);
            const float4 d0 = __ldg(du), d1 = __ldg(du + 1), d2 = __ldg(du + 2), d3 = __ldg(du + 3);
            a0.x = __fadd_rn(a0.x, d0.x); a0.y = __fadd_rn(a0.y, d0.y); a0.z = __fadd_rn(a0.z, d0.z); a0.w = __fadd_rn(a0.w, d0.w);
            a1.x = __fadd_rn(a1.x, d1.x); a1.y = __fadd_rn(a1.y, d1.y); a1.z = __fadd_rn(a1.z, d1.z); a1.w = __fadd_rn(a1.w, d1.w);
            a2.x = __fadd_rn(a2.x, d2.x); a2.y = __fadd_rn(a2.y, d2.y); a2.z = __fadd_rn(a2.z, d2.z); a2.w = __fadd_rn(a2.w, d2.w);
            a3.x = __fadd_rn(a3.x, d3.x); a3.y = __fadd_rn(a3.y, d3.y); a3.z = __fadd_rn(a3.z, d3.z); a3.w = __fadd_rn(a3.w, d3.w);
        }
        v[0] = a0.x; v[1] = a0.y; v[2] = a0.z; v[3] = a0.w; v[4] = a1.x; v[5] = a1.y; v[6] = a1.z; v[7] = a1.w;
        v[8] = a2.x; v[9] = a2.y; v[10] = a2.z; v[11] = a2.w; v[12] = a3.x; v[13] = a3.y; v[14] = a3.z; v[15] = a3.w;
    } else {
#pragma unroll
        for (int l = 0; l < 16; ++l) v[l] = (f + l < n) ? load_v(W, U, f + l) : 0.f;
    }
}

// ---------------------------------------------------------------------------------------------
// sample_kernel: choose the level-0 windows
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void set_window(Sel *s, u64 lo, u64 hi, int nb) {
    if (hi < lo) hi = lo;
    const int width = 64 - __clzll((long long)(hi - lo));
    const int nb_bits = 31 - __clz(nb);
    unsigned shift = width > nb_bits ? (unsigned)(width - nb_bits) : 0u;      // one more when the last bins would be missed
    while (((hi - lo) >> shift) >= (u64)(nb - 2)) ++shift;
    s->lo0 = lo;
    s->hi0 = hi;
    s->shift0 = shift;
}

// L_u = sum (a_i - q)^2 and *S = sum a_i of a block in fp32, a_i = |v_i| and q their mean, from the differences d_i = a_i - a_0 and not
// from q, which fp32 rounds by more than the spread of an almost uniform block: L_u = sum d_i^2 - (sum d_i)^2 / B.  With u = 2^-24 every
// d_i is within u of itself, sum d_i^2 within (B + 1) u, (sum d_i)^2 / B within 2 B u of sum d_i^2, and that is L_u + B (a_0 - q)^2 <= B L_u.
// So L_u is within B (3 B + 1) u of itself, however small it is beside the block's mean; S within B^2 u.  L_u is NaN where sum d_i
// overflows.
template <int B>
__device__ __forceinline__ float loss_u32(const float *x, float *S) {
    const float a0 = fabsf(x[0]);
    float sum = fabsf(x[1]) - a0;
    if constexpr (B == 2) {
        *S = a0 + fabsf(x[1]);
        return 0.5f * sum * sum;
    } else {
        float sq = sum * sum;
#pragma unroll
        for (int l = 2; l < B; ++l) {
            const float d = fabsf(x[l]) - a0;
            sum += d;
            sq = fmaf(d, d, sq);
        }
        *S = fabsf(fmaf((float)B, a0, sum));            // infinite, not -inf, where sum d_i overflows
        return fmaf(sum * (-1.f / (float)B), sum, sq);
    }
}

// Edges of the windows for pass_kernel's fp32 keys.  The edges hold for any tensor: with a limit on how small L_u may be beside the
// mean (which keys from an fp32 mean need) almost uniform blocks, or a threshold that few blocks reach, overflowed the candidate list
// (16384 x 4096, b = 4, blocks uniform to 1e-4: 1380 us a call, so 165).  A sum of squares, all positive, is within (B + 1) u of the exact one, the others
// within the bounds of loss_u32.  Results that underflow are off by less than TINY more.  Sums that overflow are infinite, and
// the exact key may be a B-th of the largest fp32 number then: an edge not far below that has nothing certainly above it.
__device__ __forceinline__ void make_filter(Filter *f, const Sel &sp, const Sel &su, u64 tp, u64 tu, int B) {
    constexpr double U = 0x1p-24, TINY = 0x1p-138;
    const float inf = __int_as_float(0x7f800000), nan = __int_as_float(0x7fffffff);
    const double rel_p = (double)(B * B + 32) * U, rel_u = (double)(B * (3 * B + 4)) * U;
    auto lower = [](u64 k, double rel) { return __double2float_rd(fma(__longlong_as_double((long long)k), 1.0 - rel, -TINY)); };
    auto upper = [&](u64 k, double rel) {
        const float x = __double2float_ru(fma(__longlong_as_double((long long)k), 1.0 + rel, TINY));
        return x < 0x1p122f ? x : nan;
    };
    auto point = [](u64 k) { return __double2float_rn(__longlong_as_double((long long)k)); };
    // nothing open: no key is >= inf and below -1.  (mode 3, grouped pruning: pass_kernel sets pt by the group's bit.)
    f->plo = sp.mode == 0u ? lower(sp.lo0, rel_p) : inf;
    f->phi = sp.mode == 0u ? upper(sp.hi0, rel_p) : -1.f;
    f->pt = sp.mode == 0u ? point(tp) : (sp.mode == 2u ? inf : -1.f);
    f->ulo = su.mode == 0u ? lower(su.lo0, rel_u) : inf;
    f->uhi = su.mode == 0u ? upper(su.hi0, rel_u) : -1.f;
    f->ut = su.mode == 0u ? point(tu) : (su.mode == 2u ? inf : -1.f);
}

// inclusive prefix sum over the CTA's SAMP_THREADS values (one per thread)
__device__ __forceinline__ unsigned block_scan_incl(unsigned x, unsigned *s_warp) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int m = 1; m < 32; m <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, m);
        if (lane >= m) x += y;
    }
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    const unsigned t = lane < w ? s_warp[lane] : 0u;
    return x + __reduce_add_sync(0xffffffffu, t);
}

// Window around the `frac` quantile of n sample keys: +-4 sigma (binomial) in rank.  Returns the
// two ranks whose keys bound the window and the rank of the quantile itself.
__device__ __forceinline__ void window_ranks_f(int n, float frac, int *il, int *ih, int *ipos) {
    const float pos = frac * (float)n;
    const float margin = 4.f * sqrtf(fmaxf((float)n * frac * (1.f - frac), 0.f)) + 4.f;
    int a = (int)floorf(pos - margin), b = (int)ceilf(pos + margin), c = (int)pos;
    if (a < 0) a = 0;
    if (b > n - 1) b = n - 1;
    if (c > n - 1) c = n - 1;
    if (c < 0) c = 0;
    *il = a; *ih = b; *ipos = c;
}

// A quantile near an end of the sample may lie beyond it: how far (a difference of float bit patterns) a window that begins with
// the smallest sample key, or ends with the largest, should reach beyond, when t sample keys are expected on that side of the
// quantile.  The smallest key's own quantile is rarely above 8 / t times the wanted one, and a key may grow with the square of its
// quantile (L_u of two values).  Without this a unified share of 0.3 % was often missed and one of 0.1 % always, and the
// projection done again by the exact phases (16384 x 4096, b = 4, 0.3 %: 650 us a call, so 134).
__device__ __forceinline__ unsigned beyond(float t) {
    const unsigned e = __float_as_uint(fmaxf(t, 0x1p-20f)) >> 23;         // 127 + log2 t, rounded down
    return t < 8.f ? (2u * (130u - e) + 1u) << 23 : 0u;
}

// Level-B counts of one selection; the cluster adds its eight up
struct __align__(16) SampCounts {
    unsigned bins[SAMP_THREADS];
    unsigned under, n_valid;
};
constexpr unsigned NO_SAMPLE = 0xffffffffu;           // key of a sample that takes no part: above every window

// One selection of sample_kernel, by all CTAs of the cluster alike.  key[t]: this thread's sample keys (bits of non-negative floats, or NO_SAMPLE);
// a_key: the level-A key that this thread and its seven neighbours rank.  `frac` of the keys are to be selected.  Level A
// ranks 128 of the sample keys to get a coarse window; level B counts all in SAMP_THREADS bins across that window and
// reads the final window [lo, hi) and the provisional threshold from the bin edges.  c: cleared before a
// cluster barrier.  all: room for the cluster's counts.  more(f): f(key) for this thread's sample keys beyond those.
template <class More>
__device__ __forceinline__ uint3 sample_select(const unsigned (&key)[SAMP_PER], unsigned a_key, float frac, SampCounts *c, uint4 *all,
                                               More more) {
    constexpr int A_PARTS = SAMP_THREADS / SAMP_A;
    // level-A keys, shortened to the top 25 bits below the (clear) sign bit, with the key's index in
    // the low seven: distinct words, one 32-bit compare per pair; invalid keys rank last
    __shared__ __align__(16) unsigned s_a[SAMP_A];
    __shared__ unsigned s_edge[2];                    // shortened keys at the coarse window's ranks
    __shared__ unsigned s_warp[32];
    __shared__ unsigned s_res[3];
    static_assert(SAMP_A == 128 && A_PARTS == 8, "the index of a level-A key fills the low seven bits of its shortened form");
    const int tid = threadIdx.x, lane = tid & 31, a = tid / A_PARTS, part = tid % A_PARTS;
    const bool a_valid = part == 0 && a_key != NO_SAMPLE;
    __syncthreads();                                  // an earlier call's shared words are no longer read
    if (part == 0) s_a[a] = a_valid ? (((a_key << 1) >> 7) << 7) | (unsigned)a : 0xffffffffu;
    const int na_raw = __syncthreads_count(a_valid);  // also orders the stores above
    const int na = na_raw > 0 ? na_raw : 1;
    int il, ih, ipos;
    window_ranks_f(na, frac, &il, &ih, &ipos);
    {
        // eight threads rank one level-A key, each against an eighth of the keys (neighbours read neighbouring
        // 16 bytes, no bank conflict)
        const unsigned k = s_a[a];
        int r = 0;
        const uint4 *q = reinterpret_cast<const uint4 *>(s_a) + part;
#pragma unroll
        for (int t = 0; t < SAMP_A / 4 / A_PARTS; ++t) {
            const uint4 x = q[A_PARTS * t];
            r += (x.x < k ? 1 : 0) + (x.y < k ? 1 : 0) + (x.z < k ? 1 : 0) + (x.w < k ? 1 : 0);
        }
#pragma unroll
        for (int m = 1; m < A_PARTS; m <<= 1) r += __shfl_xor_sync(0xffffffffu, r, m);
        if (part == 0) {
            if (r == il) s_edge[0] = k;
            if (r == ih) s_edge[1] = k;
        }
    }
    __syncthreads();
    // back to full keys: the low 6 bits of the edges are zero (any window is a valid window)
    unsigned clo = s_edge[0] == 0xffffffffu ? 0x7fffffffu : (s_edge[0] >> 7) << 6;
    unsigned chi = s_edge[1] == 0xffffffffu ? 0x7fffffffu : (s_edge[1] >> 7) << 6;
    const float expected = frac * (float)na;
    if (il == 0) clo -= min(clo, beyond(expected));
    if (ih == na - 1) chi = min(chi + beyond((float)na - expected), 0x7f800000u);
    if (chi < clo) chi = clo;
    // smallest shift with ((chi - clo) >> shift) < SAMP_THREADS (a power of two)
    const int width = 32 - __clz((int)(chi - clo));                    // bits of chi - clo
    const unsigned shift = width > 10 ? (unsigned)(width - 10) : 0u;
    static_assert(SAMP_THREADS == 1024, "ten bits of bin index");
    // level B
    unsigned n_under = 0, n_valid = 0;
    auto count = [&](unsigned k) {
        const unsigned d = k - clo;
        if (d < chi - clo) atomicAdd(&c->bins[d >> shift], 1u);
        n_under += k < clo ? 1u : 0u;
        n_valid += k != NO_SAMPLE ? 1u : 0u;
    };
#pragma unroll
    for (int t = 0; t < SAMP_PER; ++t) count(key[t]);
    more(count);
    n_under = __reduce_add_sync(0xffffffffu, n_under);
    n_valid = __reduce_add_sync(0xffffffffu, n_valid);
    if (lane == 0) {
        if (n_under) atomicAdd(&c->under, n_under);
        if (n_valid) atomicAdd(&c->n_valid, n_valid);
    }
    sel::ClusterTeam::arrive();
    sel::ClusterTeam::wait();
    // The bins of all CTAs come here as 16-byte words, two to a thread, and are added up out of shared memory (eight 4-byte
    // loads by every thread took 1.7 us); the two totals are read by one lane each (32 lanes that read one word of
    // another CTA are served one by one).
    unsigned under = 0, total = 0;
    constexpr int WORDS = SAMP_THREADS / 4;           // of 16 bytes
#pragma unroll
    for (int h = 0; h < SAMP_CTAS * WORDS / SAMP_THREADS; ++h) {
        const int w = h * SAMP_THREADS + tid;
        uint4 x;
        asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                     : "r"(sel::ClusterTeam::in_cta(sel::ClusterTeam::addr(&c->bins[(w % WORDS) * 4]), (unsigned)(w / WORDS))) : "memory");
        all[w] = x;
    }
    if (lane < SAMP_CTAS)
        asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];"
                     : "=r"(under), "=r"(total) : "r"(sel::ClusterTeam::in_cta(sel::ClusterTeam::addr(&c->under), (unsigned)lane)) : "memory");
    under = __reduce_add_sync(0xffffffffu, under);
    total = __reduce_add_sync(0xffffffffu, total);
    __syncthreads();
    unsigned mine = 0;
#pragma unroll
    for (int r = 0; r < SAMP_CTAS; ++r) mine += reinterpret_cast<const unsigned *>(all)[r * SAMP_THREADS + tid];
    const unsigned incl = block_scan_incl(mine, s_warp) + under;
    const unsigned excl = incl - mine;
    window_ranks_f(total > 0u ? (int)total : 1, frac, &il, &ih, &ipos);
    if (tid == 0) {
        // ranks outside the coarse window keep its edge
        s_res[0] = clo;
        s_res[1] = chi;
        s_res[2] = clo;
    }
    __syncthreads();
    const unsigned edge_lo = clo + ((unsigned)tid << shift);
    unsigned edge_hi = clo + ((unsigned)(tid + 1) << shift);
    if (edge_hi > chi) edge_hi = chi;
    if (mine) {
        if (excl <= (unsigned)il && (unsigned)il < incl) s_res[0] = edge_lo < chi ? edge_lo : chi;
        if (excl <= (unsigned)ih && (unsigned)ih < incl) s_res[1] = edge_hi;
        if (excl <= (unsigned)ipos && (unsigned)ipos < incl) s_res[2] = edge_lo < chi ? edge_lo : chi;
    }
    __syncthreads();
    unsigned lo = s_res[0], hi = s_res[1], That = s_res[2];
    if (il == 0) lo -= min(lo, beyond(frac * (float)total));
    if (ih + 1 >= (int)total) hi = min(hi + beyond((1.f - frac) * (float)total), 0x7f800000u);
    if (That < lo) That = lo;
    if (hi > lo && That >= hi) That = hi - 1;         // the provisional threshold lies inside [lo, hi)
    return make_uint3(lo, hi, That);
}

// block of the i-th of the evenly spaced samples, without a division (their number is a power of
// two, or that of all blocks); i < 2^18 and n_blocks < 2^31, so the product fits 64 bits
__device__ __forceinline__ long long sample_block(const Params &p, int i) {
    return p.samp_lg >= 0 ? (long long)(((u64)i * (u64)p.n_blocks) >> p.samp_lg) : (long long)i;
}

// sample_keys_kernel: approximate keys of the evenly spaced sample blocks, one block per thread,
// spread over the SMs: scattered 64-byte reads take one memory round trip (4096 of them issued by a
// single SM take about 9 us).  The same launch clears the histograms.
template <int B>
__global__ void __launch_bounds__(128) sample_keys_kernel(Params p, unsigned *zero_base, unsigned n_zero) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < p.n_samp) {
        const long long j = sample_block(p, i);
        float kp, ku;
        block_keys_sample<B>(p.W, p.U, j, p.use_l1, &kp, &ku);
        // keys are not negative: the sign bit of L_u tells that the block lies in a pruned group
        if (p.gprune && group_pruned(p, (unsigned)j)) ku = __uint_as_float(__float_as_uint(ku) | 0x80000000u);
        p.samp[i] = make_float2(kp, ku);
    }
    uint4 *z = reinterpret_cast<uint4 *>(zero_base);
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < n_zero / 4; q += gridDim.x * blockDim.x)
        z[q] = make_uint4(0, 0, 0, 0);
}

// Second kernel of the one-pass pipeline (one cluster): clears the selection state and chooses windows
// and provisional thresholds of the two selections from the sample keys.  Launched with programmatic stream
// serialization behind sample_keys_kernel, and itself lets pass_kernel's CTAs start early.
//
// Why a cluster: a window is +-4 sigma of rank, so the share of blocks that pass_kernel has to list, and
// resolve_kernel to go through, falls with the root of the sample's size.  With 4096 samples (one CTA) 11 % of the
// blocks of a 50 % / 25 % projection were listed, with 65536 it is 3 %, with 262144 1.4 %.
__global__ void __launch_bounds__(SAMP_THREADS) sample_kernel(Params p) {
    __shared__ SampCounts s_counts[2];
    __shared__ uint4 s_all[SAMP_CTAS * SAMP_THREADS / 4];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0) {
        unsigned *w = reinterpret_cast<unsigned *>(p.work);
        for (unsigned i = threadIdx.x; i < sizeof(Work) / 4; i += blockDim.x) w[i] = 0u;
    }
    unsigned *zc = reinterpret_cast<unsigned *>(s_counts);
    for (unsigned i = threadIdx.x; i < sizeof(s_counts) / 4; i += blockDim.x) zc[i] = 0u;
    asm volatile("griddepcontrol.wait;" ::: "memory");     // the sample keys are complete and visible
    __syncthreads();
    const long long k_unify = p.k_unify, k_prune = p.k_prune;
    const long long mb = p.n_blocks;
    const bool by_group = p.gprune != nullptr;
    const int ns = p.n_samp;
    constexpr unsigned SIGN = 0x80000000u;
    unsigned kp[SAMP_PER], ku[SAMP_PER];
    auto take = [&](int i, unsigned *k0, unsigned *k1) {
        const float2 x = i < ns ? __ldg(&p.samp[i]) : make_float2(0.f, 0.f);
        const bool valid = i < ns && !(by_group && (__float_as_uint(x.y) & SIGN));
        *k0 = valid ? __float_as_uint(x.x) : NO_SAMPLE;
        *k1 = valid ? __float_as_uint(x.y) & ~SIGN : NO_SAMPLE;
    };
    auto index = [](int t) { return (t * SAMP_CTAS + (int)blockIdx.x) * SAMP_THREADS + (int)threadIdx.x; };
#pragma unroll
    for (int t = 0; t < SAMP_PER; ++t) take(index(t), &kp[t], &ku[t]);
    // what a larger sample has beyond that is read again for each selection
    auto later = [&](auto f) {
#pragma unroll 1
        for (int t0 = SAMP_PER; t0 < ns / (SAMP_CTAS * SAMP_THREADS); t0 += SAMP_PER) {
            unsigned k0[SAMP_PER], k1[SAMP_PER];
#pragma unroll
            for (int t = 0; t < SAMP_PER; ++t) take(index(t0 + t), &k0[t], &k1[t]);
#pragma unroll
            for (int t = 0; t < SAMP_PER; ++t) f(k0[t], k1[t]);
        }
    };
    const int a = (int)threadIdx.x / (SAMP_THREADS / SAMP_A);
    unsigned kp_a, ku_a;
    take(p.samp_lg >= 7 ? a << (p.samp_lg - 7) : a, &kp_a, &ku_a);      // SAMP_A of the samples, evenly spaced
    static_assert(SAMP_A == 1 << 7, "");
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    Sel *sp = &p.work->sel[0];
    Sel *su = &p.work->sel[1];
    const long long ksel_u = k_unify - k_prune;
    auto key64 = [](unsigned x) { return key_bits((double)__uint_as_float(x < 0x7f800000u ? x : 0x7f800000u)); };
    unsigned floor_p = 0;                             // estimated prune threshold
    bool any_pruned = false;
    if (lead && p.resid) *p.resid = 0.0;              // the kernels that follow add to it
    sel::ClusterTeam::arrive();                       // every CTA's counts are cleared
    sel::ClusterTeam::wait();
    if (by_group) {
        // the prune classes are known (bit of the block's group): nothing to estimate
        if (lead) {
            set_window(sp, 0, 0, p.nb);
            sp->mode = 3u;
            sp->k = (u64)k_prune;
            p.work->That[0] = 0;
        }
    } else {
        const uint3 wp = sample_select(kp, kp_a, (float)((double)k_prune / (double)mb), &s_counts[0], s_all,
                                       [&](auto count) { later([&](unsigned k0, unsigned) { count(k0); }); });
        if (lead) {
            set_window(sp, key64(wp.x), key64(wp.y), p.nb);
            sp->mode = (k_prune == 0) ? 1u : (k_prune == mb ? 2u : 0u);
            sp->k = (u64)k_prune;
            p.work->That[0] = key64(wp.z);
        }
        // the sample blocks that survive the (estimated) prune threshold
        if (k_prune != 0) {
            floor_p = wp.z;
            any_pruned = true;
#pragma unroll
            for (int t = 0; t < SAMP_PER; ++t) ku[t] = kp[t] > wp.z ? ku[t] : NO_SAMPLE;
            ku_a = kp_a > wp.z ? ku_a : NO_SAMPLE;
        }
    }
    const long long elig = mb - k_prune;
    const uint3 wu = sample_select(ku, ku_a, elig > 0 ? (float)((double)ksel_u / (double)elig) : 0.f, &s_counts[1], s_all, [&](auto count) {
        later([&](unsigned k0, unsigned k1) { count(any_pruned && k0 <= floor_p ? NO_SAMPLE : k1); });
    });
    if (lead) {
        set_window(su, key64(wu.x), key64(wu.y), p.nb);
        su->mode = (ksel_u == 0) ? 1u : (ksel_u == elig ? 2u : 0u);
        su->k = (u64)ksel_u;
        p.work->That[1] = key64(wu.z);
        make_filter(&p.work->filter, *sp, *su, p.work->That[0], p.work->That[1], p.b);
    }
    sel::ClusterTeam::arrive();                       // nobody leaves while its counts are still read
    sel::ClusterTeam::wait();
}

// ---------------------------------------------------------------------------------------------
// finalisation helpers, run by whole CTAs of FIN_THREADS threads
// ---------------------------------------------------------------------------------------------
// A thread's eight bins of a histogram of NB_SMALL, with loads that bypass L1 (other CTAs of the kernel may have updated them)
struct Bins8 {
    unsigned c[8];
};
static_assert(NB_SMALL / FIN_THREADS == 8, "eight bins to a thread");
__device__ __forceinline__ Bins8 load_bins8(const unsigned *hist) {
    const uint4 h0 = __ldcg(reinterpret_cast<const uint4 *>(hist) + threadIdx.x * 2);
    const uint4 h1 = __ldcg(reinterpret_cast<const uint4 *>(hist) + threadIdx.x * 2 + 1);
    return {{h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w}};
}

// What select_bin found, kept in shared memory for the CTA that ran it
struct BinSel {
    unsigned B;
    u64 r, cnt;                 // rank of the k-th element in its bin, and the bin's count
    u64 lo_hi, lo_lo, hi_hi, hi_lo;     // composite range of the bin
};

// Level 0, by the whole CTA: the bin of the k-th element (k >= 1) and its composite range -> *out; bin 0 and MWU_DEV_SELECT when
// the counts are fewer.  Two barriers, the second behind the results; counts add up to less than 2^31.
// first: this thread's bins when there are NB_SMALL.  extra (shared memory, n_extra bin numbers): one more element in each of
// these bins, on top of what the histogram holds (the CTA's own corrections, not in global memory).
// sr: the CTA's copy of the selection (count and window); s: the global one, written when `publish`.
// (With 64-bit sums, five barriers and the bins loaded on entry it took 3 us.)
__device__ void select_bin(const Params &p, const Sel *sr, Sel *s, const unsigned *hist, const Bins8 &first, BinSel *out, bool publish,
                           const unsigned *extra = nullptr, unsigned n_extra = 0) {
    __shared__ unsigned s_part[32];
    const int nb = p.nb, per = nb / FIN_THREADS, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Bins8 mine = first;
    unsigned sum = 0;
    if (per == 8) {
        for (unsigned x = 0; x < n_extra; ++x) {
            const unsigned bx = extra[x];
            if ((bx >> 3) == threadIdx.x) {
#pragma unroll
                for (int i = 0; i < 8; ++i) mine.c[i] += ((bx & 7u) == (unsigned)i) ? 1u : 0u;
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += mine.c[i];
    } else {
        // A thread's 64 bins are 256 bytes: read by the thread itself, every load of a warp would
        // touch 32 cache lines (the L1 tag stage then takes 65 000 cycles per CTA for 65536 bins).
        // The warp sums them together instead: two coalesced loads and a sum per thread.
#pragma unroll 4
        for (int e = 0; e < 32; ++e) {
            const int base = (wid * 32 + e) * 64;
            const unsigned a = __reduce_add_sync(0xffffffffu, ld_vol(&hist[base + lane]) + ld_vol(&hist[base + 32 + lane]));
            if (lane == e) sum = a;
        }
        for (unsigned x = 0; x < n_extra; ++x) sum += ((extra[x] >> 6) == threadIdx.x) ? 1u : 0u;
    }
    static_assert(NB_MAX / FIN_THREADS == 64, "64 bins to a thread, or eight");
    unsigned incl = sum;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, m);
        if (lane >= m) incl += y;
    }
    if (lane == 31) s_part[wid] = incl;
    __syncthreads();
    incl += __reduce_add_sync(0xffffffffu, lane < wid ? s_part[lane] : 0u);
    const unsigned k = (unsigned)sr->k, run = incl - sum;
    auto found = [&](unsigned B, unsigned r, unsigned cnt) {
        u64 klo, khi;
        if (B == 0) { klo = 0; khi = sr->lo0; }
        else if (B == (unsigned)nb - 1u) { klo = sr->hi0; khi = ~0ull >> 1; }     // keys are < 2^63
        else {
            klo = sr->lo0 + ((u64)(B - 1) << sr->shift0);
            khi = sr->lo0 + ((u64)B << sr->shift0);
            if (khi > sr->hi0) khi = sr->hi0;
        }
        const u128 lo = make_c(klo, 0), hi = make_c(khi, 0);
        if (publish) {                                   // for the phases that follow
            s->B = B;
            s->r = r;
            s->cnt = cnt;
            s->lo_hi = (u64)(lo >> 64); s->lo_lo = (u64)lo;
            s->hi_hi = (u64)(hi >> 64); s->hi_lo = (u64)hi;
        }
        out->B = B; out->r = r; out->cnt = cnt;
        out->lo_hi = (u64)(lo >> 64); out->lo_lo = (u64)lo;
        out->hi_hi = (u64)(hi >> 64); out->hi_lo = (u64)hi;
    };
    if (threadIdx.x == FIN_THREADS - 1 && incl < k) {
        atomicOr(p.dev_status, (unsigned)MWU_DEV_SELECT);
        found(0u, 0u, 0u);
    }
    // the k-th element is among this thread's bins
    const bool owner = run < k && k <= incl;
    if (per == 8) {
        if (owner) {
            unsigned before = run, B = 0, cnt = 0, at = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (before < k && k <= before + mine.c[i]) { B = threadIdx.x * 8 + i; at = before; cnt = mine.c[i]; }
                before += mine.c[i];
            }
            found(B, k - at, cnt);
        }
    } else {
        // its warp scans the owner's 64 bins together
        const unsigned who = __ballot_sync(0xffffffffu, owner);
        if (who) {
            const int o = __ffs((int)who) - 1, base = (wid * 32 + o) * 64;
            const unsigned start = __shfl_sync(0xffffffffu, run, o);
            unsigned c0 = ld_vol(&hist[base + 2 * lane]), c1 = ld_vol(&hist[base + 2 * lane + 1]);
            for (unsigned x = 0; x < n_extra; ++x) {
                c0 += (extra[x] == (unsigned)(base + 2 * lane)) ? 1u : 0u;
                c1 += (extra[x] == (unsigned)(base + 2 * lane + 1)) ? 1u : 0u;
            }
            unsigned i1 = c0 + c1;
#pragma unroll
            for (int m = 1; m < 32; m <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, i1, m);
                if (lane >= m) i1 += y;
            }
            const unsigned b1 = start + i1 - c1, b0 = b1 - c0;
            if (b0 < k && k <= b1) found((unsigned)(base + 2 * lane), k - b0, c0);
            else if (b1 < k && k <= b1 + c1) found((unsigned)(base + 2 * lane + 1), k - b1, c1);
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------------------
// classification of a block from its bin code
// ---------------------------------------------------------------------------------------------
struct SelView {
    unsigned mode, B;
    u64 T_key, T_idx;
};

// Selection state written by an EARLIER kernel: plain (L1-cached) loads.  Volatile loads of one
// address by every warp of a large grid all queue at one L2 slice -- tens of microseconds.
__device__ __forceinline__ SelView view_of(const Sel *s) {
    SelView v;
    v.mode = s->mode;
    v.B = s->B;
    v.T_key = s->T_key;
    v.T_idx = s->T_idx;
    return v;
}

template <int B>
__device__ __forceinline__ bool selected(const Params &p, const SelView &s, long long j, unsigned bin,
                                         int which) {
    if (s.mode == 1u) return false;
    if (s.mode == 2u) return true;
    if (s.mode == 3u) return group_pruned(p, (unsigned)j);      // grouped pruning: the group's bit
    if (bin < s.B) return true;
    if (bin > s.B) return false;
    const u64 key = exact_key<B>(p, j, which);
    return key < s.T_key || (key == s.T_key && (u64)j <= s.T_idx);
}

__device__ void sort_candidates(u64 *key, unsigned *idx, int n_pow2) {
    for (int k = 2; k <= n_pow2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n_pow2; i += blockDim.x) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const u64 kx = key[i], ky = key[ixj];
                    const unsigned ix = idx[i], iy = idx[ixj];
                    const bool gt = (kx > ky) || (kx == ky && ix > iy);
                    const bool up = ((i & k) == 0);
                    if (gt == up) { key[i] = ky; key[ixj] = kx; idx[i] = iy; idx[ixj] = ix; }
                }
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------------------------
// exact pipeline
// ---------------------------------------------------------------------------------------------
struct Outs {
    float *Q;
    double *loss_u, *loss_p;
    float *u;
    unsigned *pruned_bitmap, *unified_bitmap, *sign_bits;
};

constexpr u64 NO_KEY = ~0ull;                            // of a slot without a block

// keys of block j with values v; both NO_KEY beyond the tensor.  Sets *bad when a value is not finite.
template <int B>
__device__ __forceinline__ void keys_of(const Params &p, unsigned j, const float *v, u64 *kp, u64 *ku, const Outs &o,
                                        unsigned *bad) {
    double S, Lu, Kp;
    block_keys<B>(v, p.use_l1, &S, &Lu, &Kp);
    const bool there = j < (unsigned)p.n_blocks;
    *bad |= ((unsigned)__double2hiint(S) >= 0x7ff00000u) ? 1u : 0u;
    *kp = there ? key_bits(Kp) : NO_KEY;
    *ku = there ? key_bits(Lu) : NO_KEY;
    if (there && o.loss_u) o.loss_u[j] = Lu;
    if (there && o.loss_p) o.loss_p[j] = Kp;
}

// Every output of one unit from its values and classes (bit e of cls_p / cls_u: block e); all lanes of
// the warp call it, units beyond the tensor included.  ws: 128 float4 of shared memory of the warp.
// Returns the unit's share of ||V - Q||^2.
template <int B>
__device__ __forceinline__ double store_unit(const Params &p, const Outs &o, unsigned unit, const float (&v)[16],
                                             unsigned cls_p, unsigned cls_u, float4 *ws) {
    constexpr int NBT = 16 / B;
    const int lane = threadIdx.x & 31;
    const long long n = p.n_floats, f = (long long)unit * 16;
    const unsigned n_units = (unsigned)((n + 15) / 16), n_blocks = (unsigned)p.n_blocks;
    const bool warp_full = (long long)(unit - lane + 32u) * 16 <= n;      // all 512 floats of this warp step exist
    const unsigned j0 = unit * NBT;
    double resid = 0.0;
    if (unit < n_units) {
        unsigned sb = 0;
#pragma unroll
        for (int l = 0; l < 16; ++l) sb |= (v[l] < 0.f ? 1u : 0u) << l;
        unsigned short *halves = reinterpret_cast<unsigned short *>(o.sign_bits);
        halves[unit] = (unsigned short)sb;
        if (unit == n_units - 1 && (n_units & 1)) halves[unit + 1] = 0;
        float uo[NBT], q[16];
#pragma unroll
        for (int e = 0; e < NBT; ++e) {
            const bool pr = (cls_p >> e) & 1u, un = (cls_u >> e) & 1u;
            double a[B];
#pragma unroll
            for (int l = 0; l < B; ++l) a[l] = (double)fabsf(v[e * B + l]);
            const double qd = __dmul_rn(tree_sum<B>(a), 1.0 / (double)B);
            uo[e] = un ? __double2float_rn(qd) : 0.f;
            if (p.resid && (pr || un)) {
                // the loss of the block's class: distance to zero or to the unified block
                double t[B];
#pragma unroll
                for (int l = 0; l < B; ++l) {
                    const double d = pr ? a[l] : __dsub_rn(a[l], qd);
                    t[l] = __dmul_rn(d, d);
                }
                resid += tree_sum<B>(t);
            }
#pragma unroll
            for (int l = 0; l < B; ++l) {
                const int k = e * B + l;
                q[k] = pr ? 0.f : (un ? (((sb >> k) & 1u) ? -uo[e] : uo[e]) : v[k]);
            }
        }
        if (p.U_next) {
            // dual update: one fp32 subtraction per entry (v for a pruned block, +0 for a kept one)
            if (f + 16 <= n) {
                float4 *dst = reinterpret_cast<float4 *>(p.U_next + f);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    dst[c] = make_float4(__fsub_rn(v[4 * c], q[4 * c]), __fsub_rn(v[4 * c + 1], q[4 * c + 1]),
                                         __fsub_rn(v[4 * c + 2], q[4 * c + 2]), __fsub_rn(v[4 * c + 3], q[4 * c + 3]));
            } else {
#pragma unroll
                for (int l = 0; l < 16; ++l)
                    if (f + l < n) p.U_next[f + l] = __fsub_rn(v[l], q[l]);
            }
        }
        if (o.Q && !warp_full) {
#pragma unroll
            for (int l = 0; l < 16; ++l)
                if (f + l < n) o.Q[f + l] = q[l];
        } else if (o.Q) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                ws[lane * 4 + (c ^ ((lane >> 1) & 3))] = make_float4(q[4 * c], q[4 * c + 1], q[4 * c + 2], q[4 * c + 3]);
        }
#pragma unroll
        for (int e = 0; e < NBT; ++e)
            if (j0 + e < n_blocks) o.u[j0 + e] = uo[e];
    }
    // Q of a whole warp step (2 KB): 16-byte stores at a 64-byte stride reach L2 as four partial writes
    // per 64 bytes, so the step goes through shared memory and leaves as four stores of 512 contiguous
    // bytes.  Thread t keeps piece c at slot c ^ ((t >> 1) & 3): no bank conflicts.
    if (o.Q && warp_full) {
        __syncwarp();
        float4 *dst = reinterpret_cast<float4 *>(o.Q + (long long)(unit - lane) * 16);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int t = 8 * k + (lane >> 2), c = lane & 3;
            dst[k * 32 + lane] = ws[t * 4 + (c ^ ((t >> 1) & 3))];
        }
        __syncwarp();
    }
    // class bitmaps: the warp's 32 * NBT blocks make NBT words
    const unsigned word0 = ((unit - lane) * NBT) >> 5, n_bm_words = (n_blocks + 31u) / 32u;
#pragma unroll
    for (int w = 0; w < NBT; ++w) {
        const int blk = w * 32 + lane;                   // block of this warp step that lane reports
        const unsigned xp = __shfl_sync(0xffffffffu, cls_p, blk / NBT);
        const unsigned xu = __shfl_sync(0xffffffffu, cls_u, blk / NBT);
        const unsigned wp = __ballot_sync(0xffffffffu, (xp >> (blk % NBT)) & 1u);
        const unsigned wu = __ballot_sync(0xffffffffu, (xu >> (blk % NBT)) & 1u);
        if (lane == 0 && word0 + w < n_bm_words) {
            o.pruned_bitmap[word0 + w] = wp;
            o.unified_bitmap[word0 + w] = wu;
        }
    }
    return resid;
}

// class bits of block j from its keys
__device__ __forceinline__ void add_class(const Params &p, const sel::Thresholds &T, unsigned j, unsigned e, u64 kp, u64 ku,
                                          unsigned *cls_p, unsigned *cls_u) {
    if (kp == NO_KEY) return;
    const bool pr = T.pruned(kp, j, T.mode_p == 3u && group_pruned(p, j));
    *cls_p |= (pr ? 1u : 0u) << e;
    *cls_u |= (!pr && T.unified(ku, j) ? 1u : 0u) << e;
}

// What select_exact sees of a tensor: this thread's blocks with their keys in shared memory (slot t * NBT + e
// holds block e of unit first + t * stride) ...
template <int B, int NT>
struct HeldKeys {
    static constexpr int NBT = 16 / B;
    const Params &p;
    unsigned first, stride, units;
    u64 *keys;                                           // this thread's column: prune key, then L_u, of each slot
    template <class F>
    __device__ __forceinline__ void for_blocks(F f) const {
        const u64 *k = keys;
        unsigned j0 = first * NBT;
#pragma unroll 1
        for (unsigned t = 0; t < units; ++t, j0 += stride * NBT) {
#pragma unroll(NBT < 2 ? NBT : 2)
            for (int e = 0; e < NBT; ++e, k += 2 * NT) f(j0 + e, k[0], k[NT]);
        }
    }
    __device__ __forceinline__ bool in_group(unsigned j) const { return group_pruned(p, j); }
};

// ... or evaluated again in every phase
template <int B>
struct WalkedKeys {
    static constexpr int NBT = 16 / B;
    const Params &p;
    unsigned first, stride;
    template <class F>
    __device__ __forceinline__ void for_blocks(F f) const {
        const unsigned n_units = (unsigned)((p.n_floats + 15) / 16);
        const Outs none = {};
        unsigned bad = 0;
        float nxt[16];
        if (first < n_units) load16(p.W, p.U, (long long)first * 16, p.n_floats, nxt);
#pragma unroll 1
        for (unsigned unit = first; unit < n_units; unit += stride) {
            float v[16];
#pragma unroll
            for (int l = 0; l < 16; ++l) v[l] = nxt[l];
            if (unit + stride < n_units) load16(p.W, p.U, (long long)(unit + stride) * 16, p.n_floats, nxt);      // travels meanwhile
#pragma unroll
            for (int e = 0; e < NBT; ++e) {
                u64 kp, ku;
                keys_of<B>(p, unit * NBT + e, v + e * B, &kp, &ku, none, &bad);
                f(unit * NBT + e, kp, ku);
            }
        }
    }
    __device__ __forceinline__ bool in_group(unsigned j) const { return group_pruned(p, j); }
};

// approximate keys of this thread's sample block; false: it has none, or the block lies in a pruned group
template <int B, int NT>
__device__ __forceinline__ bool sample_of(const Params &p, const sel::Problem &pb, float *kp, float *ku) {
    unsigned j;
    *kp = *ku = 0.f;
    if (!sel::sample_block_of<NT>(pb, threadIdx.x, &j)) return false;
    block_keys_sample<B>(p.W, p.U, (long long)j, p.use_l1, kp, ku);
    return !pb.by_group || !group_pruned(p, j);
}

// one CTA's shared memory of the exact phases: candidates while selecting, Q staging afterwards
template <int NT>
union ExactSmem {
    sel::SelSmem sel;
    float4 stage[NT / 32][128];
};

// The projection with keys evaluated in every phase, by all CTAs of a cooperative launch.  `team` has
// its counters cleared.
template <int B, int NT>
__device__ __noinline__ void exact_walk(const Params &p, const Outs &o, const sel::Problem &pb, sel::GridTeam<true> &team, ExactSmem<NT> &sm) {
    constexpr int NBT = 16 / B;
    const WalkedKeys<B> src = {p, team.cta * NT + threadIdx.x, team.n_cta * NT};
    __syncthreads();                                     // a caller's shared memory is no longer read
    for (int i = threadIdx.x; i < sel::GRID_BINS; i += NT) team.local[i] = 0u;
    if (p.resid && team.cta == 0 && threadIdx.x == 0) *p.resid = 0.0;
    sel::Thresholds T;
    float sp, su;
    const bool samp_ok = sample_of<B, NT>(p, pb, &sp, &su);
    // (a barrier before the emit phase orders the cleared residual even when nothing is selected)
    if (!sel::select_exact<NT>(src, team, sm.sel, pb, sp, su, samp_ok, p.dev_status, T) || !team.sync()) {
        if (threadIdx.x == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_TIMEOUT);
        return;
    }
    const unsigned n_units = (unsigned)((p.n_floats + 15) / 16);
    double resid = 0.0;
    unsigned bad = 0;
    float nxt[16];
    load16(p.W, p.U, (long long)src.first * 16, p.n_floats, nxt);
#pragma unroll 1
    for (unsigned unit = src.first; unit < (n_units + 31u) / 32u * 32u; unit += src.stride) {
        float v[16];
        unsigned cp = 0, cu = 0;
#pragma unroll
        for (int l = 0; l < 16; ++l) v[l] = nxt[l];
        if (unit + src.stride < n_units) load16(p.W, p.U, (long long)(unit + src.stride) * 16, p.n_floats, nxt);
#pragma unroll
        for (int e = 0; e < NBT; ++e) {
            u64 kp, ku;
            keys_of<B>(p, unit * NBT + e, v + e * B, &kp, &ku, o, &bad);
            add_class(p, T, unit * NBT + e, e, kp, ku, &cp, &cu);
        }
        resid += store_unit<B>(p, o, unit, v, cp, cu, sm.stage[threadIdx.x >> 5]);
    }
    if (bad) atomicOr(p.dev_status, (unsigned)MWU_DEV_NONFINITE);
    if (p.resid) block_add_double(resid, p.resid);
}

constexpr int CL_THREADS = 512;                          // cluster form
constexpr int GR_THREADS = 512;                          // grid form
constexpr int EX_SLOTS = 8192;                           // most blocks a CTA holds: 16 bytes of keys each

// The whole projection in one launch, keys held in shared memory: `units` units of 64 bytes a thread.
// CLUSTER: one cluster of sixteen CTAs; otherwise a cooperative grid over a counter that the host has
// cleared.
template <int B, bool CLUSTER>
__global__ void __launch_bounds__(CLUSTER ? CL_THREADS : GR_THREADS) exact_kernel(Params p, Outs o, sel::Problem pb, unsigned units) {
    constexpr int NBT = 16 / B, NT = CLUSTER ? CL_THREADS : GR_THREADS;
    extern __shared__ __align__(16) unsigned char mp_smem[];
    __shared__ ExactSmem<NT> sm;
    typename std::conditional<CLUSTER, sel::ClusterTeam, sel::GridTeam<false>>::type team;
    team.cta = blockIdx.x;
    team.s = &sm.sel;
    if constexpr (CLUSTER) {
        __shared__ sel::ClusterCounts counts;
        team.mine = &counts;
        team.begin();
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    } else {
        team.n_cta = gridDim.x;
        team.x = p.xwork;
        team.k = 0;
        team.local = nullptr;
    }
    float v[16];
    // warps are dealt out over the CTAs, so that a tensor with less than a unit a thread keeps all SMs busy
    const unsigned first = (threadIdx.x >> 5) * gridDim.x * 32u + blockIdx.x * 32u + (threadIdx.x & 31u);
    load16(p.W, p.U, (long long)first * 16, p.n_floats, v);              // in flight beside the sample's loads
    float sp, su;
    const bool samp_ok = sample_of<B, NT>(p, pb, &sp, &su);
    if (p.resid && blockIdx.x == 0 && threadIdx.x == 0) *p.resid = 0.0;
    HeldKeys<B, NT> src = {p, first, gridDim.x * NT, units,
                           reinterpret_cast<u64 *>(mp_smem) + threadIdx.x};
    const unsigned n_units = (unsigned)((p.n_floats + 15) / 16);
    unsigned bad = 0;
    {
        u64 *k = src.keys;
#pragma unroll 1
        for (unsigned t = 0; t < units; ++t) {
            const unsigned unit = src.first + t * src.stride;
            if (t) load16(p.W, p.U, (long long)unit * 16, p.n_floats, v);
#pragma unroll
            for (int e = 0; e < NBT; ++e, k += 2 * NT)
                keys_of<B>(p, unit * NBT + e, v + e * B, k, k + NT, o, &bad);
        }
    }
    if (bad) atomicOr(p.dev_status, (unsigned)MWU_DEV_NONFINITE);
    if constexpr (CLUSTER) team.wait();                  // every CTA's counts are cleared
    sel::Thresholds T;
    bool ok = sel::select_exact<NT>(src, team, sm.sel, pb, sp, su, samp_ok, p.dev_status, T);
    // with nothing to select there has been no barrier yet between the cleared residual and its sums
    if (ok && p.resid && T.mode_p != 0u && T.mode_u != 0u) ok = team.sync();
    if (!ok) {
        if (threadIdx.x == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_TIMEOUT);
        return;
    }
    __syncthreads();                                     // the candidates' memory becomes the staging buffer
    double resid = 0.0;
    const u64 *k = src.keys;
#pragma unroll 1
    for (unsigned t = 0; t < units; ++t) {
        const unsigned unit = src.first + t * src.stride;
        if (unit - (threadIdx.x & 31u) >= n_units) break;                // the whole warp is beyond the tensor
        unsigned cp = 0, cu = 0;
        if (units > 1u) load16(p.W, p.U, (long long)unit * 16, p.n_floats, v);
#pragma unroll
        for (int e = 0; e < NBT; ++e, k += 2 * NT) add_class(p, T, unit * NBT + e, e, k[0], k[NT], &cp, &cu);
        resid += store_unit<B>(p, o, unit, v, cp, cu, sm.stage[threadIdx.x >> 5]);
    }
    if (p.resid) block_add_double(resid, p.resid);
}

// MWU_ALGO_MULTI_PASS on tensors whose keys do not fit
constexpr int WALK_THREADS = 512;
constexpr int WALK_SMEM = (int)sizeof(ExactSmem<WALK_THREADS>) + sel::GRID_BINS * 4;
template <int B>
__global__ void __launch_bounds__(WALK_THREADS) exact_walk_kernel(const __grid_constant__ Params p, const __grid_constant__ Outs o,
                                                                  const __grid_constant__ sel::Problem pb) {
    extern __shared__ __align__(16) unsigned char mp_smem[];
    ExactSmem<WALK_THREADS> &sm = *reinterpret_cast<ExactSmem<WALK_THREADS> *>(mp_smem);
    sel::GridTeam<true> team = {blockIdx.x, gridDim.x, p.xwork, &sm.sel, 0u, reinterpret_cast<unsigned *>(mp_smem + sizeof(sm))};
    exact_walk<B, WALK_THREADS>(p, o, pb, team, sm);
}

// ---------------------------------------------------------------------------------------------
// one-pass pipeline
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void one_pass_fail(const Params &p) { atomicExch(&p.work->failed, 1u); }

// Values of warp step `step` (512 floats) that this lane handles; zero beyond the tensor.
// B <= 4: the lane's four pieces of four floats lie a warp apart, so that every access of a warp is 512 contiguous
// bytes and a block lies in one piece.  B >= 8: 64 contiguous bytes, so that a block lies in one lane.
template <int B>
__device__ __forceinline__ void load_step(const float *W, const float *U, unsigned step, int lane, long long n, float (&v)[16]) {
    if constexpr (B <= 4) {
        const long long f0 = (long long)step * 512 + lane * 4;
        if ((long long)step * 512 + 512 <= n) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 a = __ldg(reinterpret_cast<const float4 *>(W + f0) + c * 32);
                v[4 * c] = a.x; v[4 * c + 1] = a.y; v[4 * c + 2] = a.z; v[4 * c + 3] = a.w;
            }
            if (U) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float4 d = __ldg(reinterpret_cast<const float4 *>(U + f0) + c * 32);
                    v[4 * c] = __fadd_rn(v[4 * c], d.x); v[4 * c + 1] = __fadd_rn(v[4 * c + 1], d.y);
                    v[4 * c + 2] = __fadd_rn(v[4 * c + 2], d.z); v[4 * c + 3] = __fadd_rn(v[4 * c + 3], d.w);
                }
            }
        } else {
#pragma unroll
            for (int l = 0; l < 16; ++l) {
                const long long f = f0 + (l >> 2) * 128 + (l & 3);
                v[l] = f < n ? load_v(W, U, f) : 0.f;
            }
        }
    } else {
        load16(W, U, (long long)step * 512 + lane * 16, n, v);
    }
}

// 16 floats of a lane, laid out as by load_step, to step `step` of dst.  ws: 128 float4 of shared memory of the warp.
template <int B>
__device__ __forceinline__ void store_step(float *dst, unsigned step, int lane, long long n, const float (&q)[16], float4 *ws) {
    const long long base = (long long)step * 512;
    if (base + 512 > n) {
#pragma unroll
        for (int l = 0; l < 16; ++l) {
            const long long f = base + (B <= 4 ? (l >> 2) * 128 + lane * 4 + (l & 3) : lane * 16 + l);
            if (f < n) dst[f] = q[l];
        }
        return;
    }
    float4 *d4 = reinterpret_cast<float4 *>(dst + base);
    if constexpr (B <= 4) {
#pragma unroll
        for (int c = 0; c < 4; ++c) d4[c * 32 + lane] = make_float4(q[4 * c], q[4 * c + 1], q[4 * c + 2], q[4 * c + 3]);
    } else {
        // 16-byte stores at a 64-byte stride reach L2 as four partial writes per 64 bytes, so the step goes through
        // shared memory and leaves as four stores of 512 contiguous bytes.  Thread t keeps piece c at slot
        // c ^ ((t >> 1) & 3), so neither side has bank conflicts.
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 4; ++c)
            ws[lane * 4 + (c ^ ((lane >> 1) & 3))] = make_float4(q[4 * c], q[4 * c + 1], q[4 * c + 2], q[4 * c + 3]);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int t = 8 * k + (lane >> 2), c = lane & 3;
            d4[k * 32 + lane] = ws[t * 4 + (c ^ ((t >> 1) & 3))];
        }
    }
}

// Bin codes (prune | L_u << 16) of the exact keys of block j, and the exact losses of step `step`: functions of their own,
// so that the sweep's registers need not hold fp64 keys.
template <int B>
__device__ __noinline__ unsigned exact_codes(const Params &p, unsigned j) {
    const Sel *sp = &p.work->sel[0], *su = &p.work->sel[1];
    double S, Lu, Kp;
    block_keys_at<B>(p.W, p.U, (long long)j, p.use_l1, &S, &Lu, &Kp);
    return bin_of(key_bits(Kp), sp->lo0, sp->hi0, sp->shift0, (unsigned)p.nb) |
           bin_of(key_bits(Lu), su->lo0, su->hi0, su->shift0, (unsigned)p.nb) << 16;
}
template <int B>
__device__ __noinline__ void exact_losses(const Params &p, unsigned step, double *loss_u, double *loss_p) {
#pragma unroll 1
    for (int e = threadIdx.x & 31; e < 512 / B; e += 32) {
        const unsigned j = step * (512 / B) + (unsigned)e;
        if (j >= (unsigned)p.n_blocks) break;
        double S, Lu, Kp;
        block_keys_at<B>(p.W, p.U, (long long)j, p.use_l1, &S, &Lu, &Kp);
        if (loss_u) loss_u[j] = Lu;
        if (loss_p) loss_p[j] = Kp;
    }
}

// pass_kernel: provisional classes and every output in one sweep over W (+U).
// Classes come from fp32 keys: a block whose fp32 keys lie outside the windows by more than their error (Filter) has its
// final class.  The others (a few per cent: those inside the windows, and a few in ten thousand near their edges) are
// staged per warp; when 32 have gathered, the whole warp evaluates their exact fp64 keys and turns them into bin codes,
// window-histogram counts and list entries.  In fp64 every block gets only its sum (u is its rounded mean).
//
// What bounds it: HBM for blocks of 4 and more (16384 x 16384, b = 4: 435 us for 2.45 GB, 5.6 TB/s; 16384 x 4096, b = 16: 95 us,
// 5.9 TB/s), instruction issue for 2.  With fp64 keys of every block and 64-bit comparisons a block of 4 took 240
// instructions, 16384 x 16384 with b = 4 650 us.
// ADMM: also the dual update V - Q and ||V - Q||_F^2 (mwu_admm_step).
constexpr int PASS_THREADS = 256, PASS_WARPS = PASS_THREADS / 32;
// resident CTAs: blocks of 2 need the warps (16384 x 16384: 728 us a call with three, 804 with two), the others the registers
// (b = 4: 537 / 511, b = 16: 477 / 435)
constexpr int pass_ctas_per_sm(int b, bool admm) { return b == 2 && !admm ? 3 : 2; }
template <int B, bool ADMM>
__global__ void __launch_bounds__(PASS_THREADS, pass_ctas_per_sm(B, ADMM))
pass_kernel(const __grid_constant__ Params p, float *Q, double *loss_u, double *loss_p, float *u_out, unsigned *pruned_bitmap,
            unsigned *unified_bitmap, unsigned *sign_bits) {
    constexpr int NBT = 16 / B;                          // blocks of a lane
    constexpr int NBP = B <= 4 ? 4 / B : NBT;            // of them next to one another
    const long long n = p.n_floats;
    const unsigned n_steps = (unsigned)((n + 511) / 512), stride = gridDim.x * PASS_WARPS;
    // The last eighth of the steps goes to whichever warp is free: SMs differ by several per cent in how fast they stream
    // (16384 x 16384, b = 4: with equal shares the last CTA ended 35 us after the first).  Every eighth of those steps belongs
    // to one group of CTAs; one counter for all is asked more often than L2 answers.
    const unsigned n_fixed = max((n_steps - n_steps / 8u) / stride, 1u) * stride;
    unsigned *ticket = &p.work->group[blockIdx.x % PASS_GROUPS].ticket;
    auto last_step = [&]() { return n_fixed + atomicAdd(ticket, 1u) * PASS_GROUPS + blockIdx.x % PASS_GROUPS; };
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned step = blockIdx.x * PASS_WARPS + warp, next = step + stride;
    // Launched with programmatic stream serialization: the CTAs may start while sample_kernel still
    // runs.  The first values do not depend on it and are requested at once; everything
    // sample_kernel writes (windows, cleared histograms) is read only behind the wait.
    float nxt[16];
    if (step < n_steps) load_step<B>(p.W, p.U, step, lane, n, nxt);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const Filter F = p.work->filter;
    const bool some_u = F.ut >= 0.f;
    const bool by_group = p.gprune != nullptr;
    const unsigned nb = (unsigned)p.nb, top = nb - 1u;
    unsigned *hist_p = p.fhist, *hist_u = p.fhist + p.nb;
    __shared__ float4 s_q[B <= 4 ? 1 : PASS_WARPS][B <= 4 ? 1 : 128];       // one warp step of Q per warp
    __shared__ unsigned s_cidx[PASS_WARPS][STAGE_ENTRIES];                   // blocks waiting for a full 32-entry flush
    float4 *wq = s_q[B <= 4 ? 0 : warp];
    unsigned *cidx = s_cidx[warp];
    unsigned fill = 0;                                   // warp-uniform
    unsigned under_p = 0, under_u = 0, nonfinite = 0;
    double resid_acc = 0.0;
    const unsigned n_blocks = (unsigned)p.n_blocks;      // fewer than 2^30

    // staged blocks [from, from + cnt) -> exact keys, bin codes, window histograms, list entries (whole warp)
    auto flush = [&](unsigned from, unsigned cnt) {
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&p.work->list_count, cnt);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base + cnt > p.list_cap) {
            if (lane == 0) one_pass_fail(p);
            return;
        }
        if ((unsigned)lane < cnt) {
            const unsigned ent = cidx[from + lane];
            const unsigned codes = exact_codes<B>(p, ent & 0x3fffffffu), bp = codes & 0xffffu, bu = codes >> 16;
            if (p.work->sel[0].mode == 0u && bp != top) {
                if (bp == 0u) ++under_p;                                     // pruned
                else atomicAdd(&hist_p[bp], 1u);                             // open because of the prune window
            } else if (p.work->sel[1].mode == 0u) {                          // a survivor
                if (bu == 0u) ++under_u;
                else if (bu != top) atomicAdd(&hist_u[bu], 1u);
            }
            p.list[base + lane] = make_uint2(ent, codes);
        }
    };

    if (next >= n_fixed) {
        if (lane == 0) next = last_step();
        next = __shfl_sync(0xffffffffu, next, 0);
    }
#pragma unroll 1
    while (step < n_steps) {
        float v[16];
#pragma unroll
        for (int l = 0; l < 16; ++l) v[l] = nxt[l];
        // the next step's values travel while this one is evaluated
        if (next < n_steps) load_step<B>(p.W, p.U, next, lane, n, nxt);
        unsigned after = next + stride;                      // the step behind the next: asked for a step ahead
        if (after >= n_fixed && lane == 0 && next < n_steps) after = last_step();
        const bool full = (long long)step * 512 + 512 <= n;
        const unsigned j0 = step * (512 / B) + (B <= 4 ? lane * NBP : lane * NBT);   // this lane's first block
        auto block_of = [&](int e) { return j0 + (unsigned)(e / NBP) * (128 / B) + (unsigned)(e % NBP); };
        // Sign plane: bit l = (v[l] < 0).  Without a zero among the warp's values that is the IEEE sign
        // bit, gathered with one funnel shift per value; a zero (it may be -0.0) takes the compare.
        float vmin = fabsf(v[0]);
#pragma unroll
        for (int l = 1; l < 16; ++l) vmin = fminf(vmin, fabsf(v[l]));
        const bool has_zero = __any_sync(0xffffffffu, vmin == 0.f);
        unsigned sb = 0;
        if (!has_zero) {
#pragma unroll
            for (int l = 15; l >= 0; --l) sb = __funnelshift_l(__float_as_uint(v[l]), sb, 1);
        } else {
#pragma unroll
            for (int l = 0; l < 16; ++l) sb |= (v[l] < 0.f ? 1u : 0u) << l;
        }
        {
            const unsigned n_halves = (unsigned)((n + 31) / 32) * 2u;
            if constexpr (B <= 4) {
                // the pieces' four bits each, spread to bytes; a pair of lanes completes the bytes
                unsigned x = (sb | (sb << 8)) & 0x00ff00ffu;
                x = ((x | (x << 4)) & 0x0f0f0f0fu) << (4 * (lane & 1));
                x |= __shfl_xor_sync(0xffffffffu, x, 1);
                if (lane & 1) x >>= 16;
                unsigned char *dst = reinterpret_cast<unsigned char *>(sign_bits);
                const unsigned at = step * 64u + (unsigned)((lane & 1) * 32 + (lane >> 1));
                if (full || at < n_halves * 2u) dst[at] = (unsigned char)x;
                if (full || at + 16u < n_halves * 2u) dst[at + 16u] = (unsigned char)(x >> 8);
            } else {
                const unsigned at = step * 32u + (unsigned)lane;
                if (full || at < n_halves) reinterpret_cast<unsigned short *>(sign_bits)[at] = (unsigned short)sb;
            }
        }
        unsigned cls_p = 0, cls_u = 0, cand = 0;             // bit e: block e of this lane
        float uo[NBT], pt = F.pt;
#pragma unroll
        for (int e = 0; e < NBT; ++e) {
            const float *x = v + e * B;
            if (by_group && (e == 0 || (B <= 4 && e % NBP == 0))) {
                // a lane's 64 bytes, or a piece of 16, lie in one group (groups are at least 16 columns wide)
                pt = block_of(e) < n_blocks && group_pruned(p, block_of(e)) ? __int_as_float(0x7f800000) : -1.f;
            }
            // fp32 keys (see make_filter)
            float S32;
            const float ku = loss_u32<B>(x, &S32);
            float kp = x[0] * x[0];
#pragma unroll
            for (int l = 1; l < B; ++l) kp = fmaf(x[l], x[l], kp);
            if (p.use_l1) kp = S32;
            const bool there = full || block_of(e) < n_blocks;
            // (a NaN is open, and unified where everything is)
            const bool pr = kp <= pt && there, un = !pr && !(ku > F.ut) && some_u && there;
            const bool open = ((kp >= F.plo && !(kp >= F.phi)) || (!pr && !(ku < F.ulo) && !(ku >= F.uhi))) && there;
            cls_p |= pr ? 1u << e : 0u;
            cls_u |= un ? 1u << e : 0u;
            cand |= open ? 1u << e : 0u;
            // the mean as the exact keys have it
            double a[B];
#pragma unroll
            for (int l = 0; l < B; ++l) a[l] = (double)fabsf(x[l]);
            const double S = tree_sum<B>(a), qd = __dmul_rn(S, 1.0 / (double)B);
            // S = sum |v| is Inf or NaN exactly when some value of the block is
            nonfinite |= ((unsigned)__double2hiint(S) >= 0x7ff00000u) ? 1u : 0u;
            uo[e] = un ? __double2float_rn(qd) : 0.f;
            if (ADMM && p.resid && (pr || un)) {
                // squared distance of the block to its image: the loss of its (provisional) class
                double t[B];
#pragma unroll
                for (int l = 0; l < B; ++l) {
                    const double d = pr ? a[l] : __dsub_rn(a[l], qd);
                    t[l] = __dmul_rn(d, d);
                }
                resid_acc += tree_sum<B>(t);
            }
        }
        if (loss_u || loss_p) exact_losses<B>(p, step, loss_u, loss_p);
        under_p += __popc(cls_p & ~cand);
        under_u += __popc(cls_u & ~cand);
        if (full) {
#pragma unroll
            for (int e = 0; e < NBT; e += NBP) {
                if (NBP == 1) u_out[block_of(e)] = uo[e];
                else *reinterpret_cast<float2 *>(u_out + block_of(e)) = make_float2(uo[e], uo[(e + 1) % NBT]);
            }
        } else {
#pragma unroll
            for (int e = 0; e < NBT; ++e)
                if (block_of(e) < n_blocks) u_out[block_of(e)] = uo[e];
        }
        if (Q || (ADMM && p.U_next)) {
            // q = v (kept), +-u (unified: magnitude u, sign of v), or +0
            float q[16];
#pragma unroll
            for (int e = 0; e < NBT; ++e) {
                const bool pr = (cls_p >> e) & 1u, un = (cls_u >> e) & 1u;
                const unsigned mag = __float_as_uint(uo[e]);               // 0 unless unified
                if (!has_zero) {
                    // no zero in the warp: the sign of v is its IEEE sign bit
                    const unsigned m1 = pr ? 0u : (un ? 0x80000000u : 0xffffffffu);
#pragma unroll
                    for (int l = 0; l < B; ++l) q[e * B + l] = __uint_as_float((__float_as_uint(v[e * B + l]) & m1) | mag);
                } else {
                    const unsigned keep = (pr || un) ? 0u : 0xffffffffu;
                    const unsigned sgn = un ? 0x80000000u : 0u;
#pragma unroll
                    for (int l = 0; l < B; ++l) {
                        const int k = e * B + l;
                        q[k] = __uint_as_float((__float_as_uint(v[k]) & keep) | mag | ((sb << (31 - k)) & sgn));
                    }
                }
            }
            if (Q) store_step<B>(Q, step, lane, n, q, wq);
            if (ADMM && p.U_next) {
                // dual update: one fp32 subtraction per entry (v for a pruned block, +0 for a kept one)
#pragma unroll
                for (int l = 0; l < 16; ++l) q[l] = __fsub_rn(v[l], q[l]);
                store_step<B>(p.U_next, step, lane, n, q, wq);
            }
        }
        // class bitmaps: the step's 512 / B blocks make NBT words
        {
            const unsigned n_bm = (n_blocks + 31u) / 32u;
            if constexpr (B == 2) {
                // two bits of every piece, spread to bytes; four lanes complete the bytes, and each stores one piece's
                auto bytes = [&](unsigned x) {
                    x = (x | (x << 12)) & 0x000f000fu;
                    x = ((x | (x << 6)) & 0x03030303u) << (2 * (lane & 3));
                    x |= __shfl_xor_sync(0xffffffffu, x, 1);
                    x |= __shfl_xor_sync(0xffffffffu, x, 2);
                    return (unsigned char)(x >> (8 * (lane & 3)));
                };
                const unsigned char bp = bytes(cls_p), bu = bytes(cls_u);
                const unsigned at = step * 32u + (unsigned)((lane & 3) * 8 + (lane >> 2));
                if (full || at < n_bm * 4u) {
                    reinterpret_cast<unsigned char *>(pruned_bitmap)[at] = bp;
                    reinterpret_cast<unsigned char *>(unified_bitmap)[at] = bu;
                }
            } else if constexpr (B == 8) {
                // two bits of each of 16 lanes make a word: bytes by four lanes, the first stores the pruned, the second the unified
                unsigned x = (cls_p | (cls_u << 16)) << (2 * (lane & 3));
                x |= __shfl_xor_sync(0xffffffffu, x, 1);
                x |= __shfl_xor_sync(0xffffffffu, x, 2);
                const unsigned at = step * 8u + (unsigned)(lane >> 2);
                unsigned char *dst = reinterpret_cast<unsigned char *>((lane & 1) ? unified_bitmap : pruned_bitmap);
                if ((lane & 3) < 2 && (full || at < n_bm * 4u)) dst[at] = (unsigned char)((lane & 1) ? x >> 16 : x);
            } else {
                unsigned wp[NBT], wu[NBT];
#pragma unroll
                for (int e = 0; e < NBT; ++e) {
                    wp[e] = __ballot_sync(0xffffffffu, (cls_p >> e) & 1u);
                    wu[e] = __ballot_sync(0xffffffffu, (cls_u >> e) & 1u);
                }
                // lane e stores a word of the pruned, lane NBT + e of the unified
                unsigned word = wp[0];
#pragma unroll
                for (int e = 0; e < NBT; ++e) {
                    if (lane == e) word = wp[e];
                    if (lane == NBT + e) word = wu[e];
                }
                const unsigned at = step * NBT + (unsigned)(lane % NBT);
                if (lane < 2 * NBT && (full || at < n_bm)) (lane < NBT ? pruned_bitmap : unified_bitmap)[at] = word;
            }
        }
        // open blocks gather in the warp's staging buffer and leave 32 at a time
#pragma unroll 1
        for (;;) {
            const unsigned bal = __ballot_sync(0xffffffffu, cand != 0u);
            if (bal == 0u) break;
            if (cand) {
                const int e = __ffs((int)cand) - 1;
                cand &= cand - 1u;
                // block index with the provisional class in its top bits
                cidx[fill + __popc(bal & ((1u << lane) - 1u))] = block_of(e) | (((cls_p >> e) & 1u) << 31) | (((cls_u >> e) & 1u) << 30);
            }
            fill += __popc(bal);
            __syncwarp();
            if (fill >= 32u) {
                fill -= 32u;
                flush(fill, 32u);
                __syncwarp();
            }
        }
        step = next;
        next = __shfl_sync(0xffffffffu, after, 0);
    }
    if (fill > 0u) flush(0u, fill);
    // block-level totals of the lowest bins
    __shared__ unsigned s_tot[2];
    if (threadIdx.x < 2) s_tot[threadIdx.x] = 0;
    __syncthreads();
    under_p = __reduce_add_sync(0xffffffffu, under_p);
    under_u = __reduce_add_sync(0xffffffffu, under_u);
    if (lane == 0) {
        if (under_p) atomicAdd(&s_tot[0], under_p);
        if (under_u) atomicAdd(&s_tot[1], under_u);
    }
    if (nonfinite) atomicOr(p.dev_status, (unsigned)MWU_DEV_NONFINITE);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_tot[0]) atomicAdd(&hist_p[0], s_tot[0]);
        if (s_tot[1]) atomicAdd(&hist_u[0], s_tot[1]);
        // the highest bins: nobody counts what lies above a window, only that it is enough
        if (blockIdx.x == 0) { hist_p[top] = n_blocks; hist_u[top] = n_blocks; }
    }
    if (ADMM && p.resid) block_add_double(resid_acc, p.resid);
}

constexpr unsigned IDX_MASK = 0x3fffffffu;           // list entry: block index; bit 31 / 30: provisional pruned / unified

// Block idx gets final class (pr, un) where pass_kernel had written (pr0, un0): bitmaps, u, Q (and
// the dual update) are rewritten.  Returns the change of ||V - Q||^2.
// the B values of block j, with stores as wide as load_block's loads; nothing when dst is null
template <int B>
__device__ __forceinline__ void store_block(float *dst, long long j, const float (&q)[B]) {
    if (!dst) return;
    if constexpr (B == 2) {
        *reinterpret_cast<float2 *>(dst + j * 2) = make_float2(q[0], q[1]);
    } else {
#pragma unroll
        for (int c = 0; c < B / 4; ++c)
            *(reinterpret_cast<float4 *>(dst) + j * (B / 4) + c) = make_float4(q[4 * c], q[4 * c + 1], q[4 * c + 2], q[4 * c + 3]);
    }
}

template <int B>
__device__ __forceinline__ double apply_class(const Params &p, float *Q, float *u_out, unsigned *pruned_bitmap,
                                              unsigned *unified_bitmap, unsigned idx, bool pr, bool un, bool pr0,
                                              bool un0) {
    const unsigned bit = 1u << (idx & 31u);
    unsigned *wp = pruned_bitmap + (idx >> 5), *wu = unified_bitmap + (idx >> 5);
    if (pr != pr0) { if (pr) atomicOr(wp, bit); else atomicAnd(wp, ~bit); }
    if (un != un0) { if (un) atomicOr(wu, bit); else atomicAnd(wu, ~bit); }
    // each of these is a trip to DRAM: only what the change needs
    const long long j = (long long)idx;
    float v[B];
    double S = 0.0, Lu = 0.0, Kp = 0.0;
    if (!pr || p.U_next || p.resid) {
        load_block<B>(p.W, p.U, j, v);
        block_keys<B>(v, p.use_l1, &S, &Lu, &Kp);
    } else {
#pragma unroll
        for (int l = 0; l < B; ++l) v[l] = 0.f;
    }
    const float qf = __double2float_rn(__dmul_rn(S, 1.0 / (double)B));
    if (un || un0) u_out[j] = un ? qf : 0.f;
    float q[B];
#pragma unroll
    for (int l = 0; l < B; ++l) q[l] = pr ? 0.f : (un ? (v[l] < 0.f ? -qf : qf) : v[l]);
    store_block<B>(Q, j, q);
    if (p.U_next) {
#pragma unroll
        for (int l = 0; l < B; ++l) q[l] = __fsub_rn(v[l], q[l]);
        store_block<B>(p.U_next, j, q);
    }
    // change of ||V - Q||^2: the loss of the new class minus that of the provisional one
    if (!p.resid) return 0.0;
    const double sq = p.use_l1 ? block_sumsq<B>(v) : Kp;
    return (pr ? sq : (un ? Lu : 0.0)) - (pr0 ? sq : (un0 ? Lu : 0.0));
}

constexpr int CHG_PER_THREAD = 4;                    // list entries a thread classifies before the changed ones are applied
// candidate buffers, corrections and the compaction buffer; the fallback's staging memory
constexpr int RES_SMEM_USED = CAP * 20 + CHG_PER_THREAD * FIN_THREADS * 8;
constexpr int RES_SMEM_EXACT = (int)sizeof(ExactSmem<FIN_THREADS>) + sel::GRID_BINS * 4;
constexpr int RES_SMEM_BYTES = RES_SMEM_USED > RES_SMEM_EXACT ? RES_SMEM_USED : RES_SMEM_EXACT;

// rank the m candidates in shared memory (c_key, c_idx) by (key, index); m <= CAP
// c_aux (when the candidates fit one per thread: the return value) receives g_aux in the same order
__device__ bool rank_candidates(const Params &p, const u64 *g_key, const unsigned *g_idx, const unsigned *g_aux,
                                unsigned m, u64 *c_key, unsigned *c_idx, unsigned *c_aux) {
    if (m <= blockDim.x) {
        // the usual case, a few dozen candidates: every thread ranks its own by counting
        u64 k = ~0ull;
        unsigned ix = ~0u, ax = 0u;
        if (threadIdx.x < m) {
            k = ld_vol(&g_key[threadIdx.x]);
            ix = ld_vol(&g_idx[threadIdx.x]);
            ax = ld_vol(&g_aux[threadIdx.x]);
            c_key[threadIdx.x] = k;
            c_idx[threadIdx.x] = ix;
        }
        __syncthreads();
        unsigned rank = 0;
        if (threadIdx.x < m) {
            for (unsigned t = 0; t < m; ++t) {
                const u64 x = c_key[t];
                const unsigned y = c_idx[t];
                rank += (x < k || (x == k && y < ix)) ? 1u : 0u;
            }
        }
        __syncthreads();
        if (threadIdx.x < m) { c_key[rank] = k; c_idx[rank] = ix; c_aux[rank] = ax; }
        __syncthreads();
        return true;
    }
    for (int i = threadIdx.x; i < CAP; i += blockDim.x) {
        c_key[i] = (i < (int)m) ? ld_vol(&g_key[i]) : ~0ull;
        c_idx[i] = (i < (int)m) ? ld_vol(&g_idx[i]) : ~0u;
    }
    __syncthreads();
    int np2 = 2;
    while (np2 < (int)m) np2 <<= 1;
    sort_candidates(c_key, c_idx, np2);
    return false;
}

// resolve_kernel (cooperative launch: all CTAs resident): the exact thresholds of the one-pass
// pipeline and the final classes of the listed blocks, in one launch.
//   1  every CTA finds the prune threshold bin from the window histogram (the same values in
//      all of them) and scans its slice of the list: blocks of that bin become candidates, listed
//      survivors complete the L_u histogram.
//      -- grid barrier --
//   2  every CTA ranks the few dozen candidates itself (exact threshold element, no hand-over
//      between CTAs), keeps the bins of the surviving candidates as corrections to the L_u
//      histogram, and finds the unify threshold bin.
//   3  every CTA gives the blocks of its list slice their final class: the class pass_kernel wrote
//      travels in the entry, so nothing is read for the nine in ten whose class stands; the others
//      are gathered 32 to a warp and rewritten.  Blocks of the unify threshold bin become candidates.
//   4  the CTA that is through with that last ranks those, which fixes the threshold element and their classes; the
//      others do not wait for it.
//   5  if any step gave the one-pass result up (a threshold outside its window, a threshold bin or
//      tie group too large to rank, a full list), the exact phases redo the projection here.
template <int B>
__global__ void __launch_bounds__(FIN_THREADS) resolve_kernel(const __grid_constant__ Params p,
                                                              const __grid_constant__ sel::Problem pb, float *Q, double *loss_u, double *loss_p,
                                                              float *u_out, unsigned *pruned_bitmap,
                                                              unsigned *unified_bitmap, unsigned *sign_bits) {
    extern __shared__ __align__(16) unsigned char mp_smem[];
    __shared__ Work w;                                 // selection state as the earlier kernels left it
    __shared__ BinSel s_sel;
    __shared__ unsigned s_n_extra, s_n_chg;
    u64 *c_key = reinterpret_cast<u64 *>(mp_smem);
    unsigned *c_idx = reinterpret_cast<unsigned *>(mp_smem + CAP * sizeof(u64));
    unsigned *c_aux = reinterpret_cast<unsigned *>(mp_smem + CAP * 12);
    unsigned *s_extra = reinterpret_cast<unsigned *>(mp_smem + CAP * 16);               // bins of surviving candidates
    unsigned *s_chg = reinterpret_cast<unsigned *>(mp_smem + CAP * 20);                 // entries whose class changes
    unsigned k = 0;                                    // grid barriers passed
    // a thread's first list entries travel while the selection state is read (whatever lies there beyond the list's end: looked
    // at once its length is known), and serve both passes over the list
    const unsigned gstride = gridDim.x * blockDim.x, i_first = blockIdx.x * blockDim.x + threadIdx.x;
    uint2 ent0[CHG_PER_THREAD];
#pragma unroll
    for (int t = 0; t < CHG_PER_THREAD; ++t) {
        const unsigned i = i_first + (unsigned)t * gstride;
        ent0[t] = i < p.list_cap ? __ldg(&p.list[i]) : make_uint2(0u, 0u);
    }
    // (so do its bins of the histogram that is scanned first)
    unsigned *hist_u = p.fhist + p.nb;
    const bool by_key = !p.gprune && p.k_prune != 0 && p.k_prune != p.n_blocks;        // mode_p == 0
    Bins8 bins = {};
    if (p.nb == NB_SMALL) bins = load_bins8(by_key ? p.fhist : hist_u);
    load_work(p.work, &w);
    Sel *sp = &p.work->sel[0];
    Sel *su = &p.work->sel[1];
    const unsigned mode_p = w.sel[0].mode, mode_u = w.sel[1].mode;
    const unsigned nb = (unsigned)p.nb, top = nb - 1u;
    const u64 ulo = w.sel[1].lo0, uhi = w.sel[1].hi0;
    const unsigned ush = w.sel[1].shift0;
    const unsigned n_list = min(w.list_count, p.list_cap);
    // Every condition that gives the one-pass result up comes from the same words in all CTAs, none of which changes while it may
    // still be read: they all take the same path.
    bool alive = w.failed == 0u;
    if (alive && mode_p != 0u && mode_u != 0u) return;         // no threshold: every class is final
    if (threadIdx.x == 0) { s_sel.B = 0; s_sel.r = 0; s_sel.cnt = 0; s_sel.lo_hi = s_sel.lo_lo = s_sel.hi_hi = s_sel.hi_lo = 0; s_n_extra = 0; }
    __syncthreads();

    SelView vp = view_of(&w.sel[0]);
    if (alive && mode_p == 0u) {
        // ---------------- 1: the prune threshold bin, its candidates, the survivors' L_u counts ----------------
        select_bin(p, &w.sel[0], sp, p.fhist, bins, &s_sel, blockIdx.x == 0);
        const unsigned Bp = s_sel.B;
        const u64 r_p = s_sel.r;
        // the threshold bin must be a real bin of the window and small enough to rank
        if (!(Bp >= 1u && Bp <= nb - 2u && s_sel.cnt <= (u64)CAP)) alive = false;
        if (alive) {
            unsigned under = 0;
            const u128 lo0 = from_halves(s_sel.lo_hi, s_sel.lo_lo);
            const u128 hi0 = from_halves(s_sel.hi_hi, s_sel.hi_lo);
            // a thread's entries are requested together (each iteration would otherwise wait for its own load)
#pragma unroll 1
            for (unsigned i0 = i_first; i0 < n_list; i0 += CHG_PER_THREAD * gstride) {
              uint2 ent[CHG_PER_THREAD];
#pragma unroll
              for (int t4 = 0; t4 < CHG_PER_THREAD; ++t4) {
                  const unsigned i = i0 + (unsigned)t4 * gstride;
                  if (i0 == i_first) ent[t4] = i < n_list ? ent0[t4] : make_uint2(0u, 0u);
                  else ent[t4] = i < n_list ? __ldg(&p.list[i]) : make_uint2(0u, 0u);      // code 0: skipped below
              }
#pragma unroll
              for (int t4 = 0; t4 < CHG_PER_THREAD; ++t4) {
                const uint2 e = ent[t4];
                const unsigned idx = e.x & IDX_MASK;
                const unsigned bp = e.y & 0xffffu, bu = e.y >> 16;
                if (bp == 0u || bp == top) continue;          // not in the prune window: counted by pass_kernel
                if (bp < Bp) continue;                        // pruned
                if (bp == Bp) {                               // ranked after the barrier
                    double S, Lu, Kp;
                    block_keys_at<B>(p.W, p.U, (long long)idx, p.use_l1, &S, &Lu, &Kp);
                    const u64 key = key_bits(Kp);
                    const u128 c = make_c(key, (u64)idx);
                    if (c >= lo0 && c < hi0) {
                        const unsigned slot = atomicAdd(&p.work->fcand_count[0], 1u);
                        if (slot < (unsigned)CAP) {
                            p.cand_key[slot] = key;
                            p.cand_idx[slot] = idx;
                            p.cand_aux[slot] = bin_of(key_bits(Lu), ulo, uhi, ush, nb);   // where it counts if it survives
                        }
                    }
                    continue;
                }
                if (mode_u != 0u) continue;
                if (bu == 0u) ++under;
                else if (bu != top) atomicAdd(&hist_u[bu], 1u);
              }
            }
            under = __reduce_add_sync(0xffffffffu, under);
            if ((threadIdx.x & 31) == 0 && under) atomicAdd(&hist_u[0], under);
        }
        if (!grid_sync(&p.work->bar, ++k)) {              // bounded; every CTA runs into the same limit
            if (threadIdx.x == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_TIMEOUT);
            return;
        }
        if (alive) {
            // ---------------- 2: exact prune threshold, corrections, unify threshold bin ----------------
            const unsigned m = ld_vol(&p.work->fcand_count[0]);
            if (m > (unsigned)CAP || r_p < 1 || r_p > (u64)m) alive = false;
            else {
                const bool have_aux = rank_candidates(p, p.cand_key, p.cand_idx, p.cand_aux, m, c_key, c_idx, c_aux);
                vp.B = Bp;
                vp.T_key = c_key[r_p - 1];
                vp.T_idx = (u64)c_idx[r_p - 1];
                if (blockIdx.x == 0 && threadIdx.x == 0) { sp->T_key = vp.T_key; sp->T_idx = vp.T_idx; }
                // the candidates that survive belong in the L_u histogram: kept here as corrections
                if (mode_u == 0u) {
                    for (unsigned i = (unsigned)r_p + threadIdx.x; i < m; i += blockDim.x) {
                        const unsigned bu = have_aux ? c_aux[i] : bin_of(exact_key<B>(p, (long long)c_idx[i], 1), ulo, uhi, ush, nb);
                        s_extra[atomicAdd(&s_n_extra, 1u)] = bu;
                    }
                }
                __syncthreads();
            }
        }
    }
    unsigned Bu = 0;
    u64 r_u = 0;
    u128 lo = 0, hi = 0;
    if (alive && mode_u == 0u) {
        if (mode_p == 0u && p.nb == NB_SMALL) bins = load_bins8(hist_u);                // complete only now
        select_bin(p, &w.sel[1], su, hist_u, bins, &s_sel, blockIdx.x == 0, s_extra, s_n_extra);
        Bu = s_sel.B;
        r_u = s_sel.r;
        lo = from_halves(s_sel.lo_hi, s_sel.lo_lo);
        hi = from_halves(s_sel.hi_hi, s_sel.hi_lo);
        if (!(Bu >= 1u && Bu <= nb - 2u && s_sel.cnt <= (u64)CAP)) alive = false;
    }
    if (alive) {
        // ---------------- 3: final classes of the listed blocks ----------------
        double resid_delta = 0.0;
        const unsigned per_round = CHG_PER_THREAD * gridDim.x * blockDim.x;
        const unsigned rounds = (n_list + per_round - 1u) / per_round;
#pragma unroll 1
        for (unsigned rd = 0; rd < rounds; ++rd) {
            if (threadIdx.x == 0) s_n_chg = 0;
            __syncthreads();
            uint2 ent[CHG_PER_THREAD];
            bool have[CHG_PER_THREAD];
#pragma unroll
            for (int t3 = 0; t3 < CHG_PER_THREAD; ++t3) {
                const unsigned i = ((rd * CHG_PER_THREAD + t3) * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
                have[t3] = i < n_list;
                if (rd == 0u) ent[t3] = ent0[t3];
                else ent[t3] = have[t3] ? __ldg(&p.list[i]) : make_uint2(0u, 0u);
            }
#pragma unroll
            for (int t3 = 0; t3 < CHG_PER_THREAD; ++t3) {
                if (!have[t3]) continue;
                const uint2 e = ent[t3];
                const unsigned idx = e.x & IDX_MASK;
                const bool pr0 = (e.x >> 31) & 1u, un0 = (e.x >> 30) & 1u;
                const unsigned bu = e.y >> 16;
                const bool pr = selected<B>(p, vp, (long long)idx, e.y & 0xffffu, 0);
                bool un = false, held = false;
                if (!pr) {
                    if (mode_u == 2u) un = true;
                    else if (mode_u == 0u) {
                        if (bu == Bu) {                            // ranked after the barrier
                            const u64 key = exact_key<B>(p, (long long)idx, 1);
                            const u128 c = make_c(key, (u64)idx);
                            if (c >= lo && c < hi) {
                                const unsigned slot = atomicAdd(&p.work->fcand_count[1], 1u);
                                if (slot < (unsigned)CAP) {
                                    p.cand_key[CAP + slot] = key;
                                    p.cand_idx[CAP + slot] = idx;
                                    p.cand_aux[CAP + slot] = (pr0 ? 2u : 0u) | (un0 ? 1u : 0u);   // the class pass_kernel wrote
                                }
                                held = true;
                            }
                            un = c < lo;
                        } else un = bu < Bu;
                    }
                }
                if (!held && (pr != pr0 || un != un0)) {
                    // index with the final class in bits 31 / 30, the provisional class in a second word
                    const unsigned slot = atomicAdd(&s_n_chg, 1u);
                    s_chg[2 * slot] = idx | ((pr ? 1u : 0u) << 31) | ((un ? 1u : 0u) << 30);
                    s_chg[2 * slot + 1] = (pr0 ? 2u : 0u) | (un0 ? 1u : 0u);
                }
            }
            __syncthreads();
            // the changed blocks of this round, one per thread (every lane of the leading warps busy)
            const unsigned n_chg = s_n_chg;
            for (unsigned c = threadIdx.x; c < n_chg; c += blockDim.x) {
                const unsigned pe = s_chg[2 * c], old = s_chg[2 * c + 1];
                resid_delta += apply_class<B>(p, Q, u_out, pruned_bitmap, unified_bitmap, pe & IDX_MASK, (pe >> 31) & 1u,
                                              (pe >> 30) & 1u, (old >> 1) & 1u, old & 1u);
            }
            __syncthreads();
        }
        if (p.resid) block_add_double(resid_delta, p.resid);
    }
    if (alive) {
        // ---------------- 4: the blocks of the unify threshold bin, by the CTA that gets here last ----------------
        if (mode_u != 0u) return;
        __shared__ unsigned s_last;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = atomicAdd(&p.work->bar, 1u) == (k + 1u) * gridDim.x - 1u ? 1u : 0u;
            __threadfence();
        }
        __syncthreads();
        if (!s_last) return;
        const unsigned m = ld_vol(&p.work->fcand_count[1]);
        if (m > (unsigned)CAP || r_u < 1 || r_u > (u64)m) {      // (never: they are the blocks that the bin's count had, at most CAP)
            if (threadIdx.x == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_SELECT);
            return;
        }
        const bool have_aux = rank_candidates(p, p.cand_key + CAP, p.cand_idx + CAP, p.cand_aux + CAP, m, c_key, c_idx, c_aux);
        if (threadIdx.x == 0) { su->T_key = c_key[r_u - 1]; su->T_idx = (u64)c_idx[r_u - 1]; }
        const unsigned r = (unsigned)r_u;
        double tail_delta = 0.0;
        for (unsigned i = threadIdx.x; i < m; i += blockDim.x) {
            // the class pass_kernel wrote for this block: carried with the candidate, else read back
            const unsigned idx = c_idx[i], bit = 1u << (idx & 31u);
            const bool pr0 = have_aux ? ((c_aux[i] >> 1) & 1u) != 0u : (ld_vol(pruned_bitmap + (idx >> 5)) & bit) != 0u;
            const bool un0 = have_aux ? (c_aux[i] & 1u) != 0u : (ld_vol(unified_bitmap + (idx >> 5)) & bit) != 0u;
            const bool un = i < r;
            if (pr0 || un != un0)
                tail_delta += apply_class<B>(p, Q, u_out, pruned_bitmap, unified_bitmap, idx, false, un, pr0, un0);
        }
        if (p.resid) block_add_double(tail_delta, p.resid);
        return;
    }
    // ---------------- 5: the fallback, once the one-pass result was given up ----------------
    ExactSmem<FIN_THREADS> &sm = *reinterpret_cast<ExactSmem<FIN_THREADS> *>(mp_smem);
    sel::GridTeam<true> team = {blockIdx.x, gridDim.x, p.xwork, &sm.sel, 0u, reinterpret_cast<unsigned *>(mp_smem + sizeof(sm))};
    const Outs o = {Q, loss_u, loss_p, u_out, pruned_bitmap, unified_bitmap, sign_bits};
    exact_walk<B, FIN_THREADS>(p, o, pb, team, sm);
}

// ---------------------------------------------------------------------------------------------
// grouped pruning: keys of the prune groups, and the groups to zero
// ---------------------------------------------------------------------------------------------
// One CTA takes 256 rows x 64 columns of W (+U).  A half warp reads 64 consecutive values of one row;
// every lane squares (or takes the magnitude of) its four values and the sums climb the pairwise tree
// over the group's columns with shuffles (the pairing of the block keys continued across blocks);
// the rows of a group are then summed as a pairwise tree in shared memory.  Everything is fp64 with
// one rounding per operation, in a fixed order: the keys do not depend on the launch shape.
// Four rows at a time and eight CTAs an SM: the loads in flight are what counts (a grouped projection of 16384 x 4096, b = 16,
// 256 x 64: 213 us; six CTAs 221, eight rows and four CTAs 237, all sixteen rows and three CTAs 270; all lanes at every level of
// the column tree 223).
constexpr int GS_ROWS = 4, GS_CTAS = 8;
template <int GC>                                      // columns of a group: 16, 32 or 64
__global__ void __launch_bounds__(256, GS_CTAS) group_stats_kernel(Params p, double *gkey, long long rows, long long cols) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ double s_row[256][4];
    constexpr unsigned gc = GC;
    const unsigned gr = p.group_rows;
    constexpr unsigned nsl = 64u / gc;                  // group slices per CTA tile: 4, 2 or 1
    constexpr unsigned lanes_per_slice = gc / 4u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long row0 = (long long)blockIdx.y * 256, col0 = (long long)blockIdx.x * 64;
    const long long col = col0 + (lane & 15) * 4;
    const long long first = (row0 + warp * 32 + (lane >> 4)) * cols + col;      // this thread's rows: every second one from here
    const bool l1 = p.use_l1 != 0;
    // ROWS rows at a time.  Up the tree over the columns a lane keeps one of two rows at each level and gives its partner the
    // other, so a level takes half of the shuffles of the one before; after it the row's low bits are lane bits.
    constexpr int ROWS = GS_ROWS, LEVELS = (int)lanes_per_slice < ROWS ? (int)lanes_per_slice : ROWS;      // lanes that share rows out
    constexpr int KEPT = ROWS / LEVELS;                 // rows a lane ends up with
#pragma unroll 1
    for (int it0 = 0; it0 < 16; it0 += ROWS) {
        double t[ROWS];                                 // sums of this thread's four columns, row by row
#pragma unroll
        for (int k = 0; k < ROWS; ++k) {
            const int it = it0 + k, r = warp * 32 + it * 2 + (lane >> 4);
            const long long row = row0 + r;
            const long long at = first + (long long)it * 2 * cols;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < rows && col < cols) {
                v = __ldg(reinterpret_cast<const float4 *>(p.W + at));
                if (p.U) {
                    const float4 d = __ldg(reinterpret_cast<const float4 *>(p.U + at));
                    v.x = __fadd_rn(v.x, d.x); v.y = __fadd_rn(v.y, d.y); v.z = __fadd_rn(v.z, d.z); v.w = __fadd_rn(v.w, d.w);
                }
            }
            const double a0 = (double)fabsf(v.x), a1 = (double)fabsf(v.y), a2 = (double)fabsf(v.z), a3 = (double)fabsf(v.w);
            if (l1) t[k] = __dadd_rn(__dadd_rn(a0, a1), __dadd_rn(a2, a3));
            else t[k] = __dadd_rn(__fma_rn(a0, a0, __dmul_rn(a1, a1)), __fma_rn(a2, a2, __dmul_rn(a3, a3)));   // squares are exact
        }
#pragma unroll
        for (int m = 1, n = ROWS; m < LEVELS; m <<= 1, n >>= 1) {
            const bool odd = (lane & m) != 0;
#pragma unroll
            for (int i = 0; i < n / 2; ++i) {
                const double keep = odd ? t[2 * i + 1] : t[2 * i], give = odd ? t[2 * i] : t[2 * i + 1];
                t[i] = __dadd_rn(keep, __shfl_xor_sync(0xffffffffu, give, m));
            }
        }
#pragma unroll
        for (int m = LEVELS; m < (int)lanes_per_slice; m <<= 1)
#pragma unroll
            for (int k = 0; k < KEPT; ++k) t[k] = __dadd_rn(t[k], __shfl_xor_sync(0xffffffffu, t[k], m));
        if (((lane & 15) % (int)lanes_per_slice) / LEVELS == 0) {
#pragma unroll
            for (int k = 0; k < KEPT; ++k) {
                const int it = it0 + k * LEVELS + (lane & (LEVELS - 1));
                s_row[warp * 32 + it * 2 + (lane >> 4)][((unsigned)lane & 15u) / lanes_per_slice] = t[k];
            }
        }
    }
    __syncthreads();
    // rows of a group: r with r ^ 1, then r ^ 2, ...
    for (unsigned sdist = 1; sdist < gr; sdist <<= 1) {
        for (unsigned i = threadIdx.x; i < 256u * nsl; i += blockDim.x) {
            const unsigned r = i / nsl, sl = i % nsl;
            if ((r & (2u * sdist - 1u)) == 0u) s_row[r][sl] = __dadd_rn(s_row[r][sl], s_row[r + sdist][sl]);
        }
        __syncthreads();
    }
    const long long gpr = cols / gc;                    // groups per row tile
    for (unsigned i = threadIdx.x; i < (256u / gr) * nsl; i += blockDim.x) {
        const unsigned g = i / nsl, sl = i % nsl;
        const long long row = row0 + (long long)g * gr, c = col0 + (long long)sl * gc;
        if (row < rows && c < cols) gkey[(row / gr) * gpr + c / gc] = s_row[g * gr][sl];
    }
}

// One CTA: the kg groups with the smallest (key, index) get their bit in gprune.  Radix selection on
// the keys' bit patterns (eight bits a round, none for those that all keys share) gives the threshold key and how many groups
// holding exactly that key are taken; those are the ones with the lowest indices.
__global__ void __launch_bounds__(FIN_THREADS) group_select_kernel(const double *gkey, unsigned n_groups, unsigned kg,
                                                                   unsigned *gprune) {
    __shared__ unsigned s_hist[256];
    __shared__ u64 s_prefix, s_diff;
    __shared__ unsigned s_r, s_left;             // rank of the wanted key among those with the prefix; their number
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ unsigned s_warp[32];
    const u64 *keys = reinterpret_cast<const u64 *>(gkey);
    const unsigned n_words = (n_groups + 31u) / 32u;
    if (kg == 0u || kg >= n_groups) {
        for (unsigned i = threadIdx.x; i < n_words; i += blockDim.x) {
            unsigned wv = kg == 0u ? 0u : 0xffffffffu;
            if (kg != 0u && i == n_words - 1u && (n_groups & 31u)) wv = (1u << (n_groups & 31u)) - 1u;
            gprune[i] = wv;
        }
        return;
    }
    // the bits that all keys share need no round (keys are sums of like size: their exponents and first digits agree)
    u64 all = ~0ull, any = 0ull;
    for (unsigned i = threadIdx.x; i < n_groups; i += blockDim.x) {
        const u64 k = __ldg(keys + i);
        all &= k;
        any |= k;
    }
    if (threadIdx.x == 0) { s_prefix = 0; s_r = kg; s_diff = 0; s_left = n_groups; }
    __syncthreads();
    {
        // a bit differs when some key has it and some has not
        const u64 first = __ldg(keys);
        const u64 diff = any & ~all;                    // within this thread's keys ...
        const u64 d = n_groups > threadIdx.x ? (diff | (all ^ first)) : 0ull;        // ... or against the first key
        const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)d), hi = __reduce_or_sync(0xffffffffu, (unsigned)(d >> 32));
        if ((threadIdx.x & 31u) == 0u) atomicOr(&s_diff, (u64)hi << 32 | lo);
    }
    __syncthreads();
    const u64 diff = s_diff;
    const int top = diff ? 63 - __clzll((long long)diff) : -1;
    u64 mask = top >= 63 ? 0ull : ~0ull << (top + 1);
    if (threadIdx.x == 0) s_prefix = __ldg(keys) & mask;
    __syncthreads();
    // Rounds of eight bits, until one key is left (its low bits are then read from it) or the bits run out.
    for (int shift = top - 7; top >= 0 && s_left > 1u; shift -= 8) {
        if (shift < 0) shift = 0;
        for (unsigned i = threadIdx.x; i < 256u; i += blockDim.x) s_hist[i] = 0;
        __syncthreads();
        const u64 prefix = s_prefix;
        for (unsigned i = threadIdx.x; i < n_groups; i += blockDim.x) {
            const u64 k = __ldg(keys + i);
            if ((k & mask) == prefix) atomicAdd(&s_hist[(unsigned)(k >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // the digit holding the r-th key: eight bins a lane, a shuffle scan over the lanes
            const unsigned lane = threadIdx.x;
            unsigned mine[8], sum = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { mine[j] = s_hist[lane * 8 + j]; sum += mine[j]; }
            unsigned incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= (unsigned)off) incl += t;
            }
            const unsigned r = s_r;
            const unsigned hit = __ballot_sync(0xffffffffu, incl >= r);      // never empty: the keys left are >= r
            const unsigned owner = hit ? (unsigned)__ffs(hit) - 1u : 31u;
            if (lane == owner) {
                unsigned left = r - (incl - sum), d = 0;
                while (d < 7u && mine[d] < left) { left -= mine[d]; ++d; }
                s_r = left;
                s_left = mine[d];
                s_prefix = (prefix & ~((u64)255 << shift)) | ((u64)(lane * 8u + d) << shift);
            }
        }
        mask |= (u64)255 << shift;
        __syncthreads();
        if (shift == 0) break;
    }
    if (~mask != 0ull && s_left == 1u) {                // the only key with this prefix
        const u64 prefix = s_prefix;
        __syncthreads();
        for (unsigned i = threadIdx.x; i < n_groups; i += blockDim.x) {
            const u64 k = __ldg(keys + i);
            if ((k & mask) == prefix) s_prefix = k;
        }
        __syncthreads();
    }
    const u64 T = s_prefix;
    const unsigned r_ties = s_r;                        // groups with key == T that are taken (>= 1)
    // every thread owns a run of whole bitmap words; ties are numbered in index order
    const unsigned words_per = (n_words + blockDim.x - 1u) / blockDim.x;
    const unsigned w0 = threadIdx.x * words_per, w1 = min(w0 + words_per, n_words);
    unsigned ties = 0;
    for (unsigned wi = w0; wi < w1; ++wi)
        for (unsigned bit = 0; bit < 32u; ++bit) {
            const unsigned i = wi * 32u + bit;
            if (i < n_groups && __ldg(keys + i) == T) ++ties;
        }
    const unsigned incl = block_scan_incl(ties, s_warp);
    unsigned ordinal = incl - ties;                     // ties before this thread's run
    for (unsigned wi = w0; wi < w1; ++wi) {
        unsigned wv = 0;
        for (unsigned bit = 0; bit < 32u; ++bit) {
            const unsigned i = wi * 32u + bit;
            if (i >= n_groups) break;
            const u64 k = __ldg(keys + i);
            bool take = k < T;
            if (k == T) { take = ordinal < r_ties; ++ordinal; }
            wv |= (take ? 1u : 0u) << bit;
        }
        gprune[wi] = wv;
    }
}

}  // namespace proj

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
static size_t ws_off_xwork() { return align_up(sizeof(proj::Work)); }
static size_t ws_off_hist() { return align_up(ws_off_xwork() + sizeof(sel::XWork)); }
static size_t ws_off_cand_key() { return align_up(ws_off_hist() + 2 * proj::NB_MAX * sizeof(unsigned)); }
// two sets of candidates: the two halves of resolve_kernel each keep their own
static size_t ws_off_cand_idx() { return align_up(ws_off_cand_key() + 2 * proj::CAP * sizeof(proj::u64)); }
static size_t ws_off_cand_aux() { return align_up(ws_off_cand_idx() + 2 * proj::CAP * sizeof(unsigned)); }
static size_t ws_off_list() { return align_up(ws_off_cand_aux() + 2 * proj::CAP * sizeof(unsigned)); }
// candidate list of the one-pass pipeline: a quarter of the blocks (the windows hold a few per cent;
// of a small tensor they may hold more)
// (and before pass_kernel the sample's keys are in its place: the list never has fewer entries than those)
static size_t list_capacity(size_t mb) { return mb / 4 + (1 << proj::NSAMP_LG); }
static size_t ws_off_gkey(size_t mb) { return align_up(ws_off_list() + list_capacity(mb) * sizeof(uint2)); }
static size_t n_groups_of(const mwu_proj_desc *d) {
    return grouped(d) ? (size_t)(d->rows / d->prune_group_rows) * (size_t)(d->cols / d->prune_group_cols) : 0;
}
static size_t ws_off_gprune(const mwu_proj_desc *d, size_t mb) { return align_up(ws_off_gkey(mb) + n_groups_of(d) * sizeof(double)); }

// Which pipeline, and how many units of 64 bytes a thread of the exact kernel holds.
//
// All lines were measured on whole mwu_project calls (50 % / 25 %, us).  One cluster of sixteen CTAs against the grid, whose
// launch and barriers cost 10 us more but which has all SMs: 256 x 256, b = 4: 15.5 / 25.7; 256 x 512, b = 2 (a unit a thread):
// 24.8 / 29.9, with 256 x 576 36.2 / 29.9; b = 4, 256 x 768, 49152 blocks: 23.0 / 26.1, 256 x 1024: 26.9 / 25.7; b = 8, 256 x 1152,
// 18432 units: 24.0 / 25.7; b = 16, 256 x 1152: 19.0 / 23.7, 512 x 1024, 32768 units: 24.4 / 23.8.  Up to 4096 blocks a
// CTA on every SM (606208 on 148) the exact kernel beats the one-pass pipeline's four launches (512 x 1152,
// b = 8: 24 against 39; 2048 x 2048, b = 8, 524288 blocks: 45 / 52; 1024 x 2048, b = 4: 42 / 46), beyond it
// does not (1024 x 2048, b = 2, 1048576 blocks: 67 / 54): the phases' L2 counts grow with the blocks.
// Larger samples from here on, 65536 blocks instead of 16384, then 262144 (whole mwu_project calls, 50 % / 25 %, us: 4096 x 4096,
// b = 4, 4 M blocks: 94.7 against 99.3; 16384 x 8192, b = 4, 33 M: 277 / 285; 16384 x 16384, b = 4: 496 / 518 / 610, b = 2: 645 / 695;
// below each line both sizes take the same time).
constexpr long long SAMP_LARGE_BLOCKS = 1ll << 22, SAMP_HUGE_BLOCKS = 1ll << 25;
static_assert((SAMP_HUGE_BLOCKS >> 2) >= 1ll << proj::NSAMP_LARGE_LG, "the largest sample fits the list");
constexpr long long EX_CLUSTER_BLOCKS = 49152, EX_CLUSTER_UNITS = 20480, EX_AUTO_BLOCKS_PER_CTA = 4096;
struct Route {
    bool one_pass, cluster;         // else the exact kernel: as one cluster or as a cooperative grid
    int grid, held;                 // its CTAs and units per thread (0: keys evaluated in every phase)
};
static Route route_of(const mwu_proj_desc *desc, int sm_count) {
    const long long mb = desc->rows * desc->cols / desc->block, units = (desc->rows * desc->cols + 15) / 16;
    Route r = {false, false, 0, 0};
    if (desc->algo == MWU_ALGO_ONE_PASS && mb < (1ll << 30)) {      // list entries keep two class bits above the block index
        r.one_pass = true;
        return r;
    }
    if (desc->algo == MWU_ALGO_AUTO && mb > EX_AUTO_BLOCKS_PER_CTA * sm_count && mb < (1ll << 30)) {
        r.one_pass = true;
        return r;
    }
    r.cluster = ((mb <= EX_CLUSTER_BLOCKS && units <= EX_CLUSTER_UNITS) || units <= sel::CLUSTER_CTAS * proj::CL_THREADS) &&
                cluster_runs<proj::exact_kernel<16, true>, sel::CLUSTER_CTAS, proj::CL_THREADS, proj::EX_SLOTS * 16>();
    const long long threads = r.cluster ? proj::CL_THREADS : proj::GR_THREADS;
    const long long ctas = (units + 127) / 128;                      // four warps with a unit a lane
    r.grid = r.cluster ? sel::CLUSTER_CTAS : (int)(ctas < sm_count ? ctas : sm_count);
    const long long held = (units + r.grid * threads - 1) / (r.grid * threads);
    if (held * threads * (16 / desc->block) <= proj::EX_SLOTS) r.held = (int)held;
    else {
        r.cluster = false;
        r.one_pass = desc->algo == MWU_ALGO_AUTO && mb < (1ll << 30);
    }
    return r;
}

}  // namespace mwu

extern "C" size_t mwu_project_workspace_bytes(const mwu_proj_desc *desc) {
    if (mwu::validate_desc(desc, false) != MWU_OK) return 0;
    if (mwu::shape_of(desc).shaped) return mwu::shapes::workspace_bytes(desc);
    const size_t mb = (size_t)(desc->rows * desc->cols / desc->block);
    return mwu::align_up(mwu::ws_off_gprune(desc, mb) + (mwu::n_groups_of(desc) + 31) / 32 * 4 + 16);
}

// Cooperative launch (every CTA resident at once, which the grid barriers of the kernel rely on):
// the grid is cut to what the device can hold of this kernel.
template <typename... Args>
static cudaError_t launch_cooperative(void (*kern)(Args...), int grid, int threads, size_t smem, int sm_count,
                                      cudaStream_t st, Args... args) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    const long long cap = (long long)per_sm * sm_count;
    if (grid > cap) grid = (int)cap;
    void *argv[] = {(void *)&args...};
    mwu::count_launch();
    return cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3((unsigned)threads), argv, smem, st);
}

template <int B>
static cudaError_t launch_exact_held(const mwu::proj::Params &p, const mwu::proj::Outs &o, const mwu::Route &route, int sm_count,
                                     cudaStream_t st) {
    using namespace mwu::proj;
    const int threads = route.cluster ? CL_THREADS : GR_THREADS;
    const int smem = route.held * (16 / B) * threads * 16;
    const mwu::sel::Problem pb = mwu::sel::problem_of(p.n_blocks, p.k_prune, p.k_unify, p.gprune != nullptr, threads);
    auto kern = route.cluster ? exact_kernel<B, true> : exact_kernel<B, false>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, EX_SLOTS * 16);
    if (e != cudaSuccess) return e;
    if (route.cluster && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return cudaErrorUnknown;
    if (!route.cluster)
        return launch_cooperative(kern, route.grid, threads, (size_t)smem, sm_count, st, p, o, pb, (unsigned)route.held);
    mwu::count_launch();
    return mwu::launch_chained(kern, dim3((unsigned)route.grid), dim3((unsigned)threads), (size_t)smem, st, route.grid, p, o, pb,
                               (unsigned)route.held);
}

template <int B>
static cudaError_t launch_project(const mwu::proj::Params &p, const mwu_proj_desc *desc, const mwu::proj::Outs &o,
                                  int sm_count, const mwu::Route &route, double *gkey, unsigned *gprune, cudaStream_t st) {
    using namespace mwu::proj;
    cudaError_t e;
    if (p.gprune) {
        // grouped pruning: the groups' keys, then the groups to zero (a bit per group)
        const dim3 grid((unsigned)((desc->cols + 63) / 64), (unsigned)((desc->rows + 255) / 256));
        const unsigned n_groups = (unsigned)mwu::n_groups_of(desc);
        const unsigned per_group = (unsigned)(desc->prune_group_rows * desc->prune_group_cols / desc->block);
        auto stats = desc->prune_group_cols == 16 ? group_stats_kernel<16> : desc->prune_group_cols == 32 ? group_stats_kernel<32> : group_stats_kernel<64>;
        e = mwu::launch_chained(stats, grid, dim3(256), 0, st, 1, p, gkey, (long long)desc->rows, (long long)desc->cols);
        if (e == cudaSuccess)
            e = mwu::launch_chained(group_select_kernel, dim3(1), dim3(FIN_THREADS), 0, st, 1, (const double *)gkey, n_groups,
                                    (unsigned)(desc->k_prune / per_group), gprune);
        if (e != cudaSuccess) return e;
        mwu::count_launch(2);
    }
    const long long n_units = (p.n_floats + 15) / 16;
    if (!route.one_pass) {
        // the grid form's barrier counter and counts start at zero; a cluster clears them itself
        if (!route.cluster && mwu::launch_clear(p.xwork, mwu::sel::XWORK_ZERO_BYTES, st) != cudaSuccess) return cudaErrorUnknown;
        if (route.held) return launch_exact_held<B>(p, o, route, sm_count, st);
        const long long want = (n_units + WALK_THREADS - 1) / WALK_THREADS;
        e = cudaFuncSetAttribute(exact_walk_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, WALK_SMEM);
        if (e != cudaSuccess) return e;
        return launch_cooperative(exact_walk_kernel<B>, (int)(want < 2ll * sm_count ? want : 2ll * sm_count), WALK_THREADS, (size_t)WALK_SMEM,
                                  sm_count, st, p, o,
                                  mwu::sel::problem_of(p.n_blocks, p.k_prune, p.k_unify, p.gprune != nullptr, WALK_THREADS));
    }
    const bool admm = p.U_next || p.resid;
    const long long want = (n_units + PASS_THREADS - 1) / PASS_THREADS, resident = (long long)sm_count * pass_ctas_per_sm(B, admm);
    const int grid_stream = (int)(want < resident ? want : resident);
    const long long mb = p.n_blocks;
    const bool need_p = !p.gprune && desc->k_prune > 0 && desc->k_prune < mb;
    const long long ksel_u = desc->k_unify - desc->k_prune;
    const bool need_u = ksel_u > 0 && ksel_u < mb - desc->k_prune;
    e = cudaFuncSetAttribute(resolve_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM_BYTES);
    if (e != cudaSuccess) return e;
    // the sample keys (and the cleared histograms) from all SMs, then one cluster ranks the sample; the two
    // kernels behind are launched with programmatic stream serialization, so their CTAs are in place
    // (and the sweep's first loads in flight) when their predecessor ends
    unsigned *zero = reinterpret_cast<unsigned *>(p.xwork);
    const unsigned n_zero = (unsigned)(p.fhist - zero) + 2u * (unsigned)p.nb;
    e = mwu::launch_chained(sample_keys_kernel<B>, dim3((unsigned)(p.n_samp + 127) / 128), dim3(128), 0, st, 1, p, zero, n_zero);
    if (e == cudaSuccess) e = mwu::launch_chained(sample_kernel, dim3(SAMP_CTAS), dim3(SAMP_THREADS), 0, st, SAMP_CTAS, p);
    if (e != cudaSuccess) return e;
    if (admm)
        e = mwu::launch_chained(pass_kernel<B, true>, dim3((unsigned)grid_stream), dim3(PASS_THREADS), 0, st, 1, p, o.Q, o.loss_u, o.loss_p,
                                o.u, o.pruned_bitmap, o.unified_bitmap, o.sign_bits);
    else
        e = mwu::launch_chained(pass_kernel<B, false>, dim3((unsigned)grid_stream), dim3(PASS_THREADS), 0, st, 1, p, o.Q, o.loss_u, o.loss_p,
                                o.u, o.pruned_bitmap, o.unified_bitmap, o.sign_bits);
    if (e != cudaSuccess) return e;
    mwu::count_launch(3);
    if (!need_p && !need_u) return cudaGetLastError();       // no threshold: every class is final
    // the list holds a few per cent of the blocks: a thread per expected entry, one CTA per SM at most.
    // Should the one-pass result be given up (once in thousands of calls), the same kernel redoes the
    // projection with the exact phases.
    const long long lb = (mb / 8 + FIN_THREADS - 1) / FIN_THREADS;
    const int grid_list = (int)(lb < (long long)sm_count ? (lb > 16 ? lb : 16) : (long long)sm_count);
    return launch_cooperative(resolve_kernel<B>, grid_list, FIN_THREADS, (size_t)RES_SMEM_BYTES, sm_count, st, p,
                              mwu::sel::problem_of(p.n_blocks, p.k_prune, p.k_unify, p.gprune != nullptr, FIN_THREADS), o.Q,
                              o.loss_u, o.loss_p, o.u, o.pruned_bitmap, o.unified_bitmap, o.sign_bits);
}

// mwu_project and mwu_admm_step: the latter also wants U_next and / or residual_sq
static int project_impl(const mwu_proj_desc *desc, const float *W, const float *U_dual, float *Q,
                        float *U_next, double *residual_sq, float *u, uint32_t *pruned_bitmap,
                        uint32_t *unified_bitmap, uint32_t *sign_bits, double *loss_u, double *loss_p,
                        uint32_t *dev_status, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    using namespace mwu;
    int rc = validate_desc(desc, false);
    if (rc != MWU_OK) return rc;
    if (!W || !u || !pruned_bitmap || !unified_bitmap || !sign_bits || !dev_status || !workspace)
        return MWU_ERR_INVALID_ARG;
    if (!aligned_to(U_next, 16) || !aligned_to(residual_sq, 8)) return MWU_ERR_ALIGNMENT;
    if (!aligned_to(W, 16) || !aligned_to(U_dual, 16) || !aligned_to(Q, 16) || !aligned_to(u, 16) ||
        !aligned_to(pruned_bitmap, 16) || !aligned_to(unified_bitmap, 16) ||
        !aligned_to(sign_bits, 16) || !aligned_to(loss_u, 16) || !aligned_to(loss_p, 16) ||
        !aligned_to(dev_status, 4) || !aligned_to(workspace, 256))
        return MWU_ERR_ALIGNMENT;
    if (workspace_bytes < mwu_project_workspace_bytes(desc)) return MWU_ERR_WORKSPACE;
    int sm_count = 0;
    rc = check_device(&sm_count);
    if (rc != MWU_OK) return rc;

    cudaStream_t st = (cudaStream_t)cuda_stream;
    char *ws = (char *)workspace;
    if (shape_of(desc).shaped)                          // 2- and 3-dim blocks: the block-by-block path
        return shapes::project(desc, W, U_dual, Q, U_next, residual_sq, u, pruned_bitmap, unified_bitmap, sign_bits,
                               loss_u, loss_p, dev_status, workspace, sm_count, st);
    const Route route = route_of(desc, sm_count);
    proj::Params p;
    p.W = W;
    p.U = U_dual;
    p.n_floats = desc->rows * desc->cols;
    p.n_blocks = p.n_floats / desc->block;
    p.b = desc->block;
    p.use_l1 = desc->prune_key == MWU_PRUNE_KEY_L1;
    p.work = (proj::Work *)ws;
    p.nb = p.n_blocks <= proj::NB_SMALL_BLOCKS ? proj::NB_SMALL : proj::NB_MAX;
    p.xwork = (sel::XWork *)(ws + ws_off_xwork());
    p.fhist = (unsigned *)(ws + ws_off_hist());
    p.cand_key = (proj::u64 *)(ws + ws_off_cand_key());
    p.cand_idx = (unsigned *)(ws + ws_off_cand_idx());
    p.cand_aux = (unsigned *)(ws + ws_off_cand_aux());
    p.list = (uint2 *)(ws + ws_off_list());
    p.samp = (float2 *)p.list;
    p.samp_lg = p.n_blocks < SAMP_LARGE_BLOCKS ? proj::NSAMP_SMALL_LG : p.n_blocks < SAMP_HUGE_BLOCKS ? proj::NSAMP_LG : proj::NSAMP_LARGE_LG;
    p.n_samp = 1 << p.samp_lg;
    if (p.n_blocks < p.n_samp) {
        p.n_samp = (int)p.n_blocks;
        p.samp_lg = -1;
    }
    p.list_cap = (unsigned)list_capacity((size_t)p.n_blocks);
    p.dev_status = dev_status;
    p.U_next = U_next;
    p.resid = residual_sq;
    p.k_unify = desc->k_unify;
    p.k_prune = desc->k_prune;
    p.blocks_per_row = (unsigned)(desc->cols / desc->block);
    double *gkey = nullptr;
    unsigned *gprune = nullptr;
    p.gprune = nullptr;
    p.group_rows = p.group_cols = p.groups_per_row = 1;
    if (grouped(desc)) {
        gkey = (double *)(ws + ws_off_gkey((size_t)p.n_blocks));
        gprune = (unsigned *)(ws + ws_off_gprune(desc, (size_t)p.n_blocks));
        p.gprune = gprune;
        p.group_rows = (unsigned)desc->prune_group_rows;
        p.group_cols = (unsigned)desc->prune_group_cols;
        p.groups_per_row = (unsigned)(desc->cols / desc->prune_group_cols);
    }

    const proj::Outs o = {Q, loss_u, loss_p, u, pruned_bitmap, unified_bitmap, sign_bits};
    cudaError_t e;
    switch (desc->block) {
        case 2: e = launch_project<2>(p, desc, o, sm_count, route, gkey, gprune, st); break;
        case 4: e = launch_project<4>(p, desc, o, sm_count, route, gkey, gprune, st); break;
        case 8: e = launch_project<8>(p, desc, o, sm_count, route, gkey, gprune, st); break;
        default: e = launch_project<16>(p, desc, o, sm_count, route, gkey, gprune, st); break;
    }
    return e == cudaSuccess ? MWU_OK : MWU_ERR_CUDA;
}

extern "C" int mwu_project(const mwu_proj_desc *desc, const float *W, const float *U_dual, float *Q,
                           float *u, uint32_t *pruned_bitmap, uint32_t *unified_bitmap,
                           uint32_t *sign_bits, double *loss_u, double *loss_p, uint32_t *dev_status,
                           void *workspace, size_t workspace_bytes, void *cuda_stream) {
    return project_impl(desc, W, U_dual, Q, nullptr, nullptr, u, pruned_bitmap, unified_bitmap, sign_bits,
                        loss_u, loss_p, dev_status, workspace, workspace_bytes, cuda_stream);
}

extern "C" int mwu_admm_step(const mwu_proj_desc *desc, const float *W, const float *U_dual, float *Q,
                             float *U_next, double *residual_sq, float *u, uint32_t *pruned_bitmap,
                             uint32_t *unified_bitmap, uint32_t *sign_bits, uint32_t *dev_status,
                             void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (!desc || !W) return MWU_ERR_INVALID_ARG;
    if (!U_next && !residual_sq) return MWU_ERR_INVALID_ARG;       // nothing beyond mwu_project was asked for
    if (U_next) {
        // the kernels read W and U_dual again after U_next has been written: no overlap allowed
        const size_t bytes = (size_t)desc->rows * (size_t)desc->cols * sizeof(float);
        const char *o = (const char *)U_next;
        const char *ins[2] = {(const char *)W, (const char *)U_dual};
        for (int i = 0; i < 2; ++i)
            if (ins[i] && o < ins[i] + bytes && ins[i] < o + bytes) return MWU_ERR_INVALID_ARG;
    }
    return project_impl(desc, W, U_dual, Q, U_next, residual_sq, u, pruned_bitmap, unified_bitmap, sign_bits,
                        nullptr, nullptr, dev_status, workspace, workspace_bytes, cuda_stream);
}
