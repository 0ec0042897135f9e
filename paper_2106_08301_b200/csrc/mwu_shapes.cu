// Projection for 2- and 3-dim block shapes (Section 3.1; Table 1: [2,2], [2,2,2]).
//
// A block spans dk input channels x dr rows x dt kernel taps of W[rows][cin * taps]; its weights are
// not contiguous in memory, so this path works block by block instead of streaming 64-byte units.
// One launch: a team of CTAs gathers every block once, evaluates the fp64 keys (the pairwise trees of
// the 1-dim kernels, members in (row, channel, tap) order), selects exactly (mwu_select.cuh) and writes
// every output.  The keys stay in shared memory while they fit (1.2 million blocks on 148 SMs) and are
// gathered again in every phase beyond that.  A chain of latencies, like the exact kernel of the 1-dim
// blocks; the 3x3 convolution weight 128 x 1152
// with 2x2x2 blocks (20480) takes 25 us, and took 145 with five launches, two of them radix selections by a
// single CTA; 1024 x 1024 with 2x2 blocks 36 us against 1516.
//
// lower_kernel turns the result of a shape whose blocks are runs of dk entries in each of their rows
// (dt = 1, taps = 1) into the per-row 1-dim arrays mwu_pack reads.
#include <type_traits>

#include "mwu_blocks.cuh"
#include "mwu_select.cuh"

namespace mwu {
namespace shapes {

typedef unsigned long long u64;
using proj::key_bits;

struct SParams {
    const float *W;
    const float *U;
    long long rows, cols;
    int ldk, ldr, ldt;          // log2 of the block's extents
    unsigned taps, ntg, cin_groups, mb;
    int use_l1;
    sel::XWork *xwork;
    float *Q, *u, *U_next;
    double *resid, *loss_u, *loss_p;
    unsigned *pruned_bitmap, *unified_bitmap, *sign_bits, *dev_status;
};

// where block j starts, and whether it lies in the short last tap group (half as many weights)
__device__ __forceinline__ long long block_base(const SParams &p, unsigned j, bool *is_short) {
    const unsigned gt = j % p.ntg, g = j / p.ntg, gc = g % p.cin_groups, gi = g / p.cin_groups;
    const unsigned t0 = gt << p.ldt;
    *is_short = p.taps - t0 < (1u << p.ldt);
    return ((long long)gi << p.ldr) * p.cols + ((long long)gc << p.ldk) * p.taps + t0;
}
// distance of weight l from the block's start; ldt: log2 of the taps the block really has
__device__ __forceinline__ long long member(const SParams &p, int l, int ldt) {
    const int r = l >> (p.ldk + ldt), c = (l >> ldt) & ((1 << p.ldk) - 1), t = l & ((1 << ldt) - 1);
    return (long long)r * p.cols + (long long)((unsigned)c * p.taps + (unsigned)t);
}
template <int N>
__device__ __forceinline__ void gather(const SParams &p, long long base, int ldt, float (&v)[N]) {
#pragma unroll
    for (int l = 0; l < N; ++l) {
        const long long f = base + member(p, l, ldt);
        v[l] = __ldg(p.W + f);
        if (p.U) v[l] = __fadd_rn(v[l], __ldg(p.U + f));
    }
}

struct Keys {
    u64 kp, ku;
    bool bad;                   // a weight is not finite
};
template <int N>
__device__ __forceinline__ Keys keys_n(const SParams &p, long long base, int ldt) {
    float v[N];
    gather<N>(p, base, ldt, v);
    double S, Lu, Kp;
    proj::block_keys<N>(v, p.use_l1, &S, &Lu, &Kp);
    Keys k = {key_bits(Kp), key_bits(Lu), (unsigned)__double2hiint(S) >= 0x7ff00000u};
    return k;
}
template <int N>
struct Half { static constexpr int value = N / 2 < 2 ? 2 : N / 2; };      // blocks of two weights have no short form
template <int N>
__device__ __forceinline__ Keys keys_of(const SParams &p, unsigned j) {
    bool is_short;
    const long long base = block_base(p, j, &is_short);
    return is_short ? keys_n<Half<N>::value>(p, base, p.ldt - 1) : keys_n<N>(p, base, p.ldt);
}

// outputs of block j in its class; returns its share of ||V - Q||^2
template <int N>
__device__ __forceinline__ double emit_n(const SParams &p, unsigned j, long long base, int ldt, bool pr, bool un) {
    float v[N];
    gather<N>(p, base, ldt, v);
    double S, Lu, Kp;
    proj::block_keys<N>(v, 1, &S, &Lu, &Kp);
    const float qf = __double2float_rn(__dmul_rn(S, 1.0 / (double)N));
    p.u[j] = un ? qf : 0.f;
#pragma unroll
    for (int l = 0; l < N; ++l) {
        const long long f = base + member(p, l, ldt);
        const float q = pr ? 0.f : (un ? (v[l] < 0.f ? -qf : qf) : v[l]);
        if (p.Q) p.Q[f] = q;
        if (p.U_next) p.U_next[f] = __fsub_rn(v[l], q);
    }
    if (!p.resid || !(pr || un)) return 0.0;
    return pr ? proj::block_sumsq<N>(v) : Lu;
}

constexpr u64 NO_KEY = ~0ull;
constexpr int SH_THREADS = 512;
constexpr int SH_SLOTS = 8192;                           // most blocks a CTA holds: 16 bytes of keys each
// LARGE: a grid whose CTAs count in shared memory first; WALK: one that also gathers the keys again in every phase
enum Form { CLUSTER, GRID, LARGE, WALK };

// what select_exact sees: block first + t * stride in slot t of this thread's column ...
struct Held {
    const SParams &p;
    unsigned first, stride, per;
    const u64 *keys;
    template <class F>
    __device__ __forceinline__ void for_blocks(F f) const {
        const u64 *k = keys;
#pragma unroll 1
        for (unsigned t = 0; t < per; ++t, k += 2 * SH_THREADS) f(first + t * stride, k[0], k[SH_THREADS]);
    }
    __device__ __forceinline__ bool in_group(unsigned) const { return false; }
};
// ... or evaluated each time
template <int N>
struct Walked {
    const SParams &p;
    unsigned first, stride;
    template <class F>
    __device__ __forceinline__ void for_blocks(F f) const {
        for (unsigned j = first; j < p.mb; j += stride) {
            const Keys k = keys_of<N>(p, j);
            f(j, k.kp, k.ku);
        }
    }
    __device__ __forceinline__ bool in_group(unsigned) const { return false; }
};

template <int N, int FORM>
__global__ void __launch_bounds__(SH_THREADS) shape_kernel(const __grid_constant__ SParams p,
                                                           const __grid_constant__ sel::Problem pb, unsigned per) {
    extern __shared__ __align__(16) unsigned char key_smem[];
    __shared__ sel::SelSmem sm;
    typename std::conditional<FORM == CLUSTER, sel::ClusterTeam, sel::GridTeam<FORM != GRID>>::type team;
    team.cta = blockIdx.x;
    team.s = &sm;
    if constexpr (FORM == CLUSTER) {
        __shared__ sel::ClusterCounts counts;
        team.mine = &counts;
        team.begin();
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    } else {
        team.n_cta = gridDim.x;
        team.x = p.xwork;
        team.k = 0;
        if constexpr (FORM == GRID) team.local = nullptr;
        else {
            __shared__ unsigned s_bins[sel::GRID_BINS];
            for (int i = threadIdx.x; i < sel::GRID_BINS; i += SH_THREADS) s_bins[i] = 0u;      // (a barrier comes before any use)
            team.local = s_bins;
        }
    }
    const unsigned first = blockIdx.x * SH_THREADS + threadIdx.x, stride = gridDim.x * SH_THREADS;
    const int lane = threadIdx.x & 31;
    if (p.resid && first == 0u) *p.resid = 0.0;
    float sp = 0.f, su = 0.f;
    unsigned sj;
    const bool samp_ok = sel::sample_block_of<SH_THREADS>(pb, threadIdx.x, &sj);
    if (samp_ok) {
        const Keys k = keys_of<N>(p, sj);
        sp = (float)__longlong_as_double((long long)k.kp);
        su = (float)__longlong_as_double((long long)k.ku);
    }
    u64 *keys = reinterpret_cast<u64 *>(key_smem) + threadIdx.x;
    bool bad = false;
    // keys of this thread's blocks
    for (unsigned t = 0, j = first; FORM == WALK ? j < p.mb : t < per; ++t, j += stride) {
        Keys k = {NO_KEY, NO_KEY, false};
        if (j < p.mb) {
            k = keys_of<N>(p, j);
            bad = bad || k.bad;
            if (p.loss_u) p.loss_u[j] = __longlong_as_double((long long)k.ku);
            if (p.loss_p) p.loss_p[j] = __longlong_as_double((long long)k.kp);
        }
        if (FORM != WALK) { keys[2 * t * SH_THREADS] = k.kp; keys[(2 * t + 1) * SH_THREADS] = k.ku; }
    }
    if (bad) atomicOr(p.dev_status, (unsigned)MWU_DEV_NONFINITE);
    // sign plane: a warp to a word
    {
        const long long n = p.rows * p.cols, n_words = (n + 31) / 32;
#pragma unroll 4
        for (long long wi = first >> 5; wi < n_words; wi += stride >> 5) {
            const long long f = wi * 32 + lane;
            float v = 0.f;
            if (f < n) {
                v = __ldg(p.W + f);
                if (p.U) v = __fadd_rn(v, __ldg(p.U + f));
            }
            const unsigned word = __ballot_sync(0xffffffffu, v < 0.f);
            if (lane == 0) p.sign_bits[wi] = word;
        }
    }
    if constexpr (FORM == CLUSTER) team.wait();          // every CTA's counts are cleared
    typename std::conditional<FORM == WALK, Walked<N>, Held>::type src = [&]() {
        if constexpr (FORM == WALK) return Walked<N>{p, first, stride};
        else return Held{p, first, stride, per, keys};
    }();
    sel::Thresholds T;
    bool ok = sel::select_exact<SH_THREADS>(src, team, sm, pb, sp, su, samp_ok, p.dev_status, T);
    // with nothing to select there has been no barrier yet between the cleared residual and its sums
    if (ok && p.resid && T.mode_p != 0u && T.mode_u != 0u) ok = team.sync();
    if (!ok) {
        if (threadIdx.x == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_TIMEOUT);
        return;
    }
    double resid = 0.0;
    for (unsigned t = 0, j = first; j - (unsigned)lane < p.mb; ++t, j += stride) {      // whole warps stay together
        bool pr = false, un = false;
        if (j < p.mb) {
            u64 kp, ku;
            if (FORM == WALK) { const Keys k = keys_of<N>(p, j); kp = k.kp; ku = k.ku; }
            else { kp = keys[2 * t * SH_THREADS]; ku = keys[(2 * t + 1) * SH_THREADS]; }
            pr = T.pruned(kp, j, false);
            un = !pr && T.unified(ku, j);
            bool is_short;
            const long long base = block_base(p, j, &is_short);
            resid += is_short ? emit_n<Half<N>::value>(p, j, base, p.ldt - 1, pr, un) : emit_n<N>(p, j, base, p.ldt, pr, un);
        }
        const unsigned wp = __ballot_sync(0xffffffffu, pr), wu = __ballot_sync(0xffffffffu, un);
        if (lane == 0) { p.pruned_bitmap[j >> 5] = wp; p.unified_bitmap[j >> 5] = wu; }
    }
    if (p.resid) proj::block_add_double(resid, p.resid);
}

// 1-dim run jb = row * (cols / dk) + kb belongs to block (row / dr, kb): its class and magnitude
__global__ void __launch_bounds__(256) lower_kernel(long long n_runs, long long runs_per_row, int dr,
                                                    const unsigned *pruned_bitmap, const unsigned *unified_bitmap,
                                                    const float *u, unsigned *pruned1, unsigned *unified1, float *u1) {
    const long long n_iter = (n_runs + 31) / 32 * 32;
    for (long long jb = (long long)blockIdx.x * blockDim.x + threadIdx.x; jb < n_iter; jb += (long long)gridDim.x * blockDim.x) {
        bool pr = false, un = false;
        if (jb < n_runs) {
            const long long row = jb / runs_per_row, kb = jb - row * runs_per_row;
            const long long j = (row / dr) * runs_per_row + kb;
            pr = (pruned_bitmap[j >> 5] >> (j & 31)) & 1u;
            un = (unified_bitmap[j >> 5] >> (j & 31)) & 1u;
            u1[jb] = u[j];
        }
        const unsigned wp = __ballot_sync(0xffffffffu, pr), wu = __ballot_sync(0xffffffffu, un);
        if ((threadIdx.x & 31) == 0 && jb < n_runs) { pruned1[jb >> 5] = wp; unified1[jb >> 5] = wu; }
    }
}

constexpr int SH_CLUSTER_PER = 2;                        // most blocks of a thread in the cluster form

// Counting in shared memory costs a microsecond (20480 blocks: 24.8 us without, 26.2 with), and makes up for it above (262144 blocks:
// 35.2 / 35.0; all keys equal: 1930 / 91).
constexpr long long SH_GRID_BLOCKS = 65536;

static int grid_for(long long items, int sm_count) {
    const long long want = (items + 255) / 256, cap = (long long)sm_count * 16;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// scratch of the shape path: the team's state
size_t workspace_bytes(const mwu_proj_desc *) { return align_up(sizeof(sel::XWork)); }

template <int N>
static cudaError_t launch(const SParams &p, const mwu_proj_desc *desc, int sm_count, cudaStream_t st) {
    const long long mb = p.mb, ctas = (mb + SH_THREADS - 1) / SH_THREADS;
    const sel::Problem pb = sel::problem_of(mb, desc->k_prune, desc->k_unify, false, SH_THREADS);
    // One cluster up to 16384 blocks (two a thread): gathering is most of the work, and a grid has more SMs for
    // it than the cluster's barriers save (9216 blocks: 19.4 us as a cluster, 25.8 as a grid; 18432: 25.5 / 25.8; 27648:
    // 30.6 / 26.0).  Keys held while a CTA's fit.
    if (mb <= (long long)SH_CLUSTER_PER * sel::CLUSTER_CTAS * SH_THREADS &&
        cluster_runs<shape_kernel<N, CLUSTER>, sel::CLUSTER_CTAS, SH_THREADS, SH_CLUSTER_PER * SH_THREADS * 16>()) {
        const unsigned per = (unsigned)((ctas + sel::CLUSTER_CTAS - 1) / sel::CLUSTER_CTAS);
        const size_t smem = (size_t)per * SH_THREADS * 16;
        const cudaError_t e = cudaFuncSetAttribute(shape_kernel<N, CLUSTER>, cudaFuncAttributeMaxDynamicSharedMemorySize, SH_CLUSTER_PER * SH_THREADS * 16);
        if (e != cudaSuccess) return e;
        if (cudaFuncSetAttribute(shape_kernel<N, CLUSTER>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return cudaErrorUnknown;
        count_launch();
        return launch_chained(shape_kernel<N, CLUSTER>, dim3(sel::CLUSTER_CTAS), dim3(SH_THREADS), smem, st, sel::CLUSTER_CTAS, p, pb, per);
    }
    if (launch_clear(p.xwork, sel::XWORK_ZERO_BYTES, st) != cudaSuccess) return cudaErrorUnknown;
    const int grid = (int)(ctas < sm_count ? ctas : sm_count);
    unsigned per = (unsigned)((ctas + grid - 1) / grid);
    const bool held = (long long)per * SH_THREADS <= SH_SLOTS;
    auto kern = !held ? shape_kernel<N, WALK> : mb <= SH_GRID_BLOCKS ? shape_kernel<N, GRID> : shape_kernel<N, LARGE>;
    if (held) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SH_SLOTS * 16);
        if (e != cudaSuccess) return e;
    }
    const size_t smem = held ? (size_t)per * SH_THREADS * 16 : 0;
    SParams pc = p;
    sel::Problem pbc = pb;
    void *argv[] = {&pc, &pbc, &per};
    count_launch();
    return cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3(SH_THREADS), argv, smem, st);
}

int project(const mwu_proj_desc *desc, const float *W, const float *U_dual, float *Q, float *U_next,
            double *residual_sq, float *u, uint32_t *pruned_bitmap, uint32_t *unified_bitmap, uint32_t *sign_bits,
            double *loss_u, double *loss_p, uint32_t *dev_status, void *workspace, int sm_count, cudaStream_t st) {
    const ShapeInfo sh = shape_of(desc);
    auto log2_of = [](int x) { int l = 0; while ((1 << l) < x) ++l; return l; };
    SParams p;
    p.W = W; p.U = U_dual;
    p.rows = desc->rows; p.cols = desc->cols;
    p.ldk = log2_of(sh.dk); p.ldr = log2_of(sh.dr); p.ldt = log2_of(sh.dt);
    p.taps = (unsigned)sh.taps; p.ntg = (unsigned)sh.ntg; p.cin_groups = (unsigned)sh.cin_groups; p.mb = (unsigned)sh.mb;
    p.use_l1 = desc->prune_key == MWU_PRUNE_KEY_L1;
    p.xwork = (sel::XWork *)workspace;
    p.Q = Q; p.u = u; p.U_next = U_next; p.resid = residual_sq; p.loss_u = loss_u; p.loss_p = loss_p;
    p.pruned_bitmap = pruned_bitmap; p.unified_bitmap = unified_bitmap; p.sign_bits = sign_bits; p.dev_status = dev_status;
    cudaError_t e;
    switch (sh.dk * sh.dr * sh.dt) {
        case 2: e = launch<2>(p, desc, sm_count, st); break;
        case 4: e = launch<4>(p, desc, sm_count, st); break;
        case 8: e = launch<8>(p, desc, sm_count, st); break;
        default: e = launch<16>(p, desc, sm_count, st); break;
    }
    return e == cudaSuccess ? MWU_OK : MWU_ERR_CUDA;
}

// scratch mwu_pack needs behind the packed bytes for a shaped descriptor: lowered u and bitmaps
size_t lowering_bytes(const mwu_proj_desc *desc) {
    const size_t runs = (size_t)(desc->rows * desc->cols / desc->block);
    return align_up(runs * sizeof(float)) + 2 * align_up((runs + 31) / 32 * 4 + 16);
}

int lower(const mwu_proj_desc *desc, const float *u, const uint32_t *pruned_bitmap, const uint32_t *unified_bitmap,
          void *scratch, const float **u1, const uint32_t **pruned1, const uint32_t **unified1, int sm_count,
          cudaStream_t st) {
    const ShapeInfo sh = shape_of(desc);
    const long long runs = desc->rows * desc->cols / desc->block;
    float *du = (float *)scratch;
    unsigned *dp = (unsigned *)((char *)scratch + align_up((size_t)runs * sizeof(float)));
    unsigned *dun = (unsigned *)((char *)dp + align_up(((size_t)runs + 31) / 32 * 4 + 16));
    lower_kernel<<<grid_for(runs, sm_count), 256, 0, st>>>(runs, desc->cols / desc->block, sh.dr, pruned_bitmap,
                                                          unified_bitmap, u, dp, dun, du);
    count_launch();
    *u1 = du; *pruned1 = dp; *unified1 = dun;
    return cudaGetLastError() == cudaSuccess ? MWU_OK : MWU_ERR_CUDA;
}

}  // namespace shapes
}  // namespace mwu
