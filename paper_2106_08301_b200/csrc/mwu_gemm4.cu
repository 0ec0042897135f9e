// mwu_gemm for few activation rows: the packed weights streamed through the tensor cores once.
//
// With few activation rows the product is bound by the packed bytes (16384 x 4096, b = 16, 80 % / 60 %,
// 16 rows: 41 MB, 6.3 us at the copy bandwidth).  Expanding the weights first writes and reads them again
// as 134 MB of bf16, so here a record is decoded in shared memory and multiplied there, and nothing but
// the output leaves the SM.  The weights are the M operand (128 rows of a record on the 128
// tensor-memory lanes), the activation rows the N operand, so 16 rows cost an MMA of N = 16.
//
// One CTA: one 128-row weight tile, up to 128 activation rows, a range of the 64-wide k stages; the CTAs
// that share a tile's stages form a cluster (`split` of them) and add up their partial sums through
// distributed shared memory, in rank order.  Roles:
//   decode     groups of two warps, each with a weight tile and a box of X of its own, take the records in
//              turn.  A record is a chain of short waits (list entries from L2, the tile's last MMA, clearing,
//              scattering, the proxy fence, the next MMA), about 2000 cycles however many threads share
//              it, so up to ten groups an SM work on as many records at a time.  The lists of a group's next
//              record are brought to L2 one turn ahead.  The tile is cleared first, so pruned blocks need neither
//              their list nor a store.
//   MMA        one warp: tensor memory, the MMAs in record order, a commit per record frees its group.
// Two CTAs to an SM.
//
// What bounds it: 16384 x 4096, b = 16, 16 rows: 19.3 us, about 7 of them before the first record and after the last; the records
// are then at four fifths of what shared memory passes (144 cycles a record for the operands, 104 to clear and write, lists).
// Before, the MMA warp's instructions a record, between those of twelve decode groups' warps, were the limit (26.6 us; with a
// sixth group a CTA 21.8 instead of 19.3, with three groups 20.3).
// Every wait on an mbarrier is bounded; when one runs out the kernel raises MWU_DEV_TIMEOUT, waits for
// its copies in flight, frees tensor memory and returns.  Tensor memory is given back before the cluster
// barrier, so holding it never depends on another CTA.
#include <cstddef>

#include "mwu_gemm_dev.cuh"

namespace mwu {
namespace gemm {

constexpr int ST_GROUP = 64;                        // threads of a decode group
constexpr unsigned ST_BATCH = 4;                    // list entries a thread reads before it stores any
constexpr int ST_MAX_GROUPS = 5;
constexpr int ST_MAX_THREADS = ST_MAX_GROUPS * ST_GROUP + 32;
constexpr int ST_MAX_ROWS = 128;                    // activation rows of a CTA
constexpr int ST_SMEM_CTA = 227 * 512 - 1024;       // two CTAs an SM; each costs 1 KB besides

struct StreamParams {
    int mpad;                   // activation rows of a CTA, a multiple of 16
    int m_tiles;
    int split;                  // CTAs of a cluster
    int stages_per;             // k stages of a CTA (the last one of a cluster may have fewer)
    int groups;
    unsigned tmem_cols;
};

struct StreamSmem {
    unsigned long long tile_full[ST_MAX_GROUPS], tile_empty[ST_MAX_GROUPS], tfull;
    unsigned tmem_base;
    int abort;
    int drain_abort;
    int n_live;
};

__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ float4 ld_cluster_f4(unsigned addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// the lines of `bytes` bytes from p on to L2, spread over a decode group
__device__ __forceinline__ void prefetch_span(const unsigned char *p, unsigned bytes, unsigned t0) {
#pragma unroll 1
    for (unsigned l = t0 * 128u; l < bytes; l += ST_GROUP * 128u) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + l) : "memory");
}

template <int BW>
__global__ void __launch_bounds__(ST_MAX_THREADS, 2)
mwu_gemm_stream_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ Params p,
                       const __grid_constant__ StreamParams q) {
    asm volatile("griddepcontrol.wait;" ::: "memory");      // launched while the kernel before may still run
    MWU_CHECK_HEADER(p);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_raw + smem_pad_1024(smem_raw);
    unsigned char *tiles = base;
    unsigned char *xbuf = tiles + q.groups * REC_BYTES;
    const unsigned x_bytes = (unsigned)q.mpad * (BK * 2);
    StreamSmem *sm = reinterpret_cast<StreamSmem *>(xbuf + q.groups * x_bytes);
    uint4 *srec = reinterpret_cast<uint4 *>(reinterpret_cast<unsigned char *>(sm) + ((sizeof(StreamSmem) + 15) & ~(size_t)15));
    float *part = reinterpret_cast<float *>(base);          // partial sums [mpad][128], once everything is multiplied
    volatile int *abort = &sm->abort;

    const int n_threads = q.groups * ST_GROUP + 32, mma_warp = q.groups * (ST_GROUP / 32);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned rank = blockIdx.x % (unsigned)q.split, unit = blockIdx.x / (unsigned)q.split;
    const unsigned mt = unit % (unsigned)q.m_tiles;
    const long long rt = unit / (unsigned)q.m_tiles;
    const int k0 = (int)rank * q.stages_per;
    int n_st = (int)p.n_stages - k0;
    n_st = n_st < 0 ? 0 : (n_st > q.stages_per ? q.stages_per : n_st);

    if (tid == 0) {
        for (int g = 0; g < ST_MAX_GROUPS; ++g) {
            mbar_init(smem_u32(&sm->tile_full[g]), ST_GROUP / 32 + 1);      // the warps, and the box of X
            mbar_init(smem_u32(&sm->tile_empty[g]), 1);
        }
        mbar_init(smem_u32(&sm->tfull), 1);
        sm->abort = 0;
        sm->drain_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == mma_warp) {
        tmem_alloc(smem_u32(&sm->tmem_base), q.tmem_cols);
        // By this warp, and only now (one thread's trigger is the CTA's): the kernel behind may take all of an SM's tensor
        // memory before it waits for this one, and must not get there first.
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    // the record table of this CTA's stages
    if (n_st > 0) {
        const uint4 *recs = reinterpret_cast<const uint4 *>(p.packed + p.off_rec) + rt * p.n_stages + k0;
        for (int i = tid; i <= n_st; i += n_threads) srec[i] = __ldg(recs + i);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = *reinterpret_cast<volatile unsigned *>(&sm->tmem_base);
    if (warp == 0) {
        // The live stages, in order (z and w of entry j: the j-th one's number and live slices).  A record whose ranges do not lie inside the sections is not touched.
        int n = 0;
        for (int i0 = 0; i0 < n_st; i0 += 32) {
            const int i = i0 + lane;
            bool take = false;
            unsigned live = 0u;
            if (i < n_st) {
                const uint4 a = srec[i], b = srec[i + 1];
                const bool bad = a.x > b.x || b.x > p.n_unified || a.y > b.y || b.y > p.n_dense ||
                                 (b.x - a.x) + (b.y - a.y) > (unsigned)(kTileRows * BK / BW);
                if (bad) atomicOr(p.dev_status, (unsigned)MWU_DEV_BOUNDS);
                live = a.w & 0xFu;
                take = !bad && live != 0u;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, take);       // (and entries i0 to i0 + 31 are read before they are written)
            if (take) *reinterpret_cast<uint2 *>(&srec[n + __popc(bal & ((1u << lane) - 1u))].z) = make_uint2((unsigned)i, live);
            n += __popc(bal);
        }
        if (lane == 0) sm->n_live = n;
    }
    __syncthreads();
    const int n_live = sm->n_live;

    if (warp == mma_warp) {
        // ---------------- MMA issuer ----------------
        // Every record of the CTA passes through this warp in turn, between decode warps that compete for its issue slots, so
        // what counts is its instructions a record.
        const unsigned idesc = make_idesc(q.mpad);
        const unsigned long long adesc0 = make_desc(smem_u32(tiles)), bdesc0 = make_desc(smem_u32(xbuf));
        const unsigned a_step = REC_BYTES / 16, b_step = x_bytes / 16, bar0 = smem_u32(&sm->tile_full[0]);
        constexpr unsigned EMPTY = (unsigned)(offsetof(StreamSmem, tile_empty) - offsetof(StreamSmem, tile_full));
        unsigned g = 0, phase = 0, live = n_live ? srec[0].w : 0u;
#pragma unroll 1
        for (int j = 0; j < n_live; ++j) {
            const unsigned bar = bar0 + g * 8u, next = j + 1 < n_live ? srec[j + 1].w : 0u;
            if (!warp_wait_spin(bar, phase, abort)) break;
            tc_fence_after();
            const unsigned long long adesc = adesc0 + g * a_step, bdesc = bdesc0 + g * b_step;
            if (elect_one()) {
                unsigned acc = j != 0 ? 1u : 0u;
                if (live == 0xFu) {
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)
                        umma_bf16(tmem_base, adesc + (unsigned long long)(k4 * 2), bdesc + (unsigned long long)(k4 * 2), idesc, k4 ? 1u : acc);
                } else {
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4) {
                        if ((live >> k4) & 1u) {
                            umma_bf16(tmem_base, adesc + (unsigned long long)(k4 * 2), bdesc + (unsigned long long)(k4 * 2), idesc, acc);
                            acc = 1u;
                        }
                    }
                }
                umma_commit(bar + EMPTY);
            }
            __syncwarp();
            live = next;
            if (++g == (unsigned)q.groups) { g = 0; phase ^= 1u; }
        }
        if (n_live) {
            if (elect_one()) umma_commit(smem_u32(&sm->tfull));
            __syncwarp();
            // nothing this warp issued may be running when tensor memory is freed
            mbar_wait(smem_u32(&sm->tfull), 0, &sm->drain_abort);
        }
        __syncwarp();
    } else {
        // ---------------- decode: this group takes every q.groups-th live record ----------------
        constexpr unsigned OFF_MASK = DecodeCfg<BW, ST_GROUP>::OFF_MASK;
        constexpr int WORDS = BW / 2;
        constexpr unsigned BATCH = ST_BATCH;
        // Dense blocks: a lane to a block, whose halves then reach different banks in both stores (two lanes to a block of 16 met
        // in one bank every other time).
        constexpr unsigned DBATCH = BW == 16 ? BATCH / 2 : BATCH;
        // Blocks of 16: the tile is cleared where the group's last record wrote, as long as a batch held all of it (clearing
        // the whole tile takes 128 cycles of the SM's shared memory: 16384 x 4096, 16 rows 20.8 us, so 19.3; blocks of 8 gain nothing).
        constexpr bool UNDO = BW == 16;
        const int group = warp / (ST_GROUP / 32);
        const unsigned t0 = (unsigned)tid & (ST_GROUP - 1u);
        unsigned char *tile = tiles + group * REC_BYTES;
        const uint2 *ulist = reinterpret_cast<const uint2 *>(p.packed + p.off_ulist) + t0;
        const unsigned short *dposl = reinterpret_cast<const unsigned short *>(p.packed + p.off_dpos) + t0;
        const unsigned char *dpayl = p.packed + p.off_dpay + t0 * (2u * BW);
        unsigned mine = 0, old_u = 0, old_d = 0;            // entries of the group's last record
        bool ok = true, cleared = false;                    // nothing but those entries is in the tile
        unsigned at_u[BATCH], at_d[DBATCH];                 // where this thread wrote them
#pragma unroll
        for (unsigned k = 0; k < BATCH; ++k) at_u[k] = at_d[k % DBATCH] = 0u;
        // A thread that ran out of time goes through the rest of the loop without touching anything, so that the group's
        // barriers stay matched.
#pragma unroll 1
        for (int j = group; j < n_live; j += q.groups) {
            const unsigned i = srec[j].z;
            const uint2 a = *reinterpret_cast<const uint2 *>(&srec[i]), b = *reinterpret_cast<const uint2 *>(&srec[i + 1]);
            const unsigned n_u = b.x - a.x, n_d = b.y - a.y;
            const uint2 *ul = ulist + a.x;
            const unsigned short *dpos = dposl + a.y;
            const unsigned char *pay = dpayl + (unsigned long long)a.y * (2 * BW);
            // the first entries travel while the tile is waited for and zeroed
            uint2 ent[BATCH];                               // x: spread signs, y: off | bf16(u) << 16
            unsigned off[DBATCH];
            unsigned v[DBATCH][WORDS];
            auto read_u = [&](unsigned e0) {                // entries e0 + t0, and every ST_GROUP-th from there
#pragma unroll
                for (unsigned k = 0; k < BATCH; ++k)
                    if (e0 + t0 + k * ST_GROUP < n_u) ent[k] = __ldg(ul + e0 + k * ST_GROUP);
            };
            auto read_d = [&](unsigned e0) {
#pragma unroll
                for (unsigned k = 0; k < DBATCH; ++k) {
                    if (e0 + t0 + k * ST_GROUP >= n_d) continue;
                    off[k] = __ldg(dpos + e0 + k * ST_GROUP);
                    ld_words<WORDS>(pay + (e0 + k * ST_GROUP) * (2u * BW), v[k]);
                }
            };
            auto write_u = [&](unsigned e0) {
#pragma unroll
                for (unsigned k = 0; k < BATCH; ++k) {
                    if (e0 + t0 + k * ST_GROUP >= n_u) break;
                    const unsigned at = ent[k].y & OFF_MASK;
                    unsigned w[WORDS];
                    unified_words<WORDS>(ent[k], w);
                    st_words<WORDS>(tile, at, w);
                    if (UNDO) at_u[k] = at;
                }
            };
            auto write_d = [&](unsigned e0) {
#pragma unroll
                for (unsigned k = 0; k < DBATCH; ++k) {
                    if (e0 + t0 + k * ST_GROUP >= n_d) break;
                    const unsigned at = off[k] & OFF_MASK;
                    st_words<WORDS>(tile, at, v[k]);
                    if (UNDO) at_d[k] = at;
                }
            };
            read_u(0u);
            read_d(0u);
            // lists of the group's next record
            if (j + q.groups < n_live) {
                const unsigned ni = srec[j + q.groups].z;
                const uint2 na = *reinterpret_cast<const uint2 *>(&srec[ni]), nb = *reinterpret_cast<const uint2 *>(&srec[ni + 1]);
                prefetch_span(p.packed + p.off_ulist + (size_t)na.x * 8u, (nb.x - na.x) * 8u, t0);
                prefetch_span(p.packed + p.off_dpay + (size_t)na.y * (2u * BW), (nb.y - na.y) * (2u * BW), t0);
                prefetch_span(p.packed + p.off_dpos + (size_t)na.y * 2u, (nb.y - na.y) * 2u, t0);
            }
            // tile and box are free once the group's last record is multiplied
            if (ok && mine && !mbar_wait(smem_u32(&sm->tile_empty[group]), (mine - 1u) & 1u, abort)) ok = false;
            __syncwarp();
            if (ok) {
                if (t0 == 0) {
                    mbar_expect_tx(smem_u32(&sm->tile_full[group]), x_bytes);
                    tma_load_2d(smem_u32(xbuf + group * x_bytes), &tmap_x, smem_u32(&sm->tile_full[group]), (k0 + (int)i) * BK, (int)mt * q.mpad);
                }
                if (UNDO && cleared) {
                    const unsigned zero[WORDS] = {};
#pragma unroll
                    for (unsigned k = 0; k < BATCH; ++k) {
                        if (t0 + k * ST_GROUP >= old_u) break;
                        st_words<WORDS>(tile, at_u[k], zero);
                    }
#pragma unroll
                    for (unsigned k = 0; k < DBATCH; ++k) {
                        if (t0 + k * ST_GROUP >= old_d) break;
                        st_words<WORDS>(tile, at_d[k], zero);
                    }
                } else {
                    uint4 *z = reinterpret_cast<uint4 *>(tile) + t0;
#pragma unroll
                    for (int t = 0; t < REC_BYTES / 16 / ST_GROUP; ++t) z[t * ST_GROUP] = make_uint4(0, 0, 0, 0);
                }
            }
            group_barrier<ST_GROUP>(1 + group);
            if (ok) {
                write_u(0u);
                write_d(0u);
                for (unsigned e0 = BATCH * ST_GROUP; e0 < n_u; e0 += BATCH * ST_GROUP) { read_u(e0); write_u(e0); }
                for (unsigned e0 = DBATCH * ST_GROUP; e0 < n_d; e0 += DBATCH * ST_GROUP) { read_d(e0); write_d(e0); }
                if (UNDO) {
                    old_u = n_u;
                    old_d = n_d;
                    cleared = n_u <= BATCH * ST_GROUP && n_d <= DBATCH * ST_GROUP;
                }
                fence_proxy_async();
                ++mine;
            }
            __syncwarp();
            if (ok && lane == 0) mbar_arrive(smem_u32(&sm->tile_full[group]));
        }
        // a box of X that is still on its way must land before this CTA's shared memory goes away
        if (t0 == 0 && mine) mbar_wait(smem_u32(&sm->tile_full[group]), (mine - 1u) & 1u, &sm->drain_abort);
        __syncwarp();
        if (n_live && ok) mbar_wait(smem_u32(&sm->tfull), 0, abort);
        __syncwarp();
    }
    __syncthreads();
    // ---------------- epilogue: partial sums to shared memory, tensor memory given back ----------------
    const bool sums = n_live && *abort == 0;
    const int readers = mma_warp >= 8 ? 2 : 1;              // warps to a quarter of the lanes
    if (warp < 4 * readers) {
        tc_fence_after();
        const int quarter = warp & 3;                       // tensor-memory lanes (weight rows) this warp may read
        for (int c = (warp >> 2) * 16; c < q.mpad; c += 16 * readers) {
            unsigned v[16];
            if (sums) tmem_ld16(tmem_base + ((unsigned)(quarter * 32) << 16) + (unsigned)c, v);
            else {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = 0u;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) part[(c + j) * 128 + quarter * 32 + lane] = __uint_as_float(v[j]);
        }
        tc_fence_before();
    }
    __syncthreads();
    if (warp == mma_warp) {
        tc_fence_after();
        tmem_dealloc(tmem_base, q.tmem_cols);
    }
    if ((*abort || sm->drain_abort) && tid == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_TIMEOUT);
    __syncwarp();
    if (q.split > 1) cluster_sync_all();
    // rows rank, rank + split, ... of the tile: a warp adds up one row of 128 columns
    const long long m0 = (long long)mt * q.mpad;
    const long long n0 = rt * kTileRows + lane * 4;
    for (int m = (int)rank + warp * q.split; m < q.mpad && m0 + m < p.M; m += (n_threads / 32) * q.split) {
        const unsigned at = smem_u32(part + m * 128 + lane * 4);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q.split == 1) acc = *reinterpret_cast<const float4 *>(part + m * 128 + lane * 4);
        else {
#pragma unroll 4
            for (int c = 0; c < q.split; ++c) {
                const float4 v = ld_cluster_f4(mbar_addr_in_cta(at, (unsigned)c));
                acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
            }
        }
        const float r[4] = {acc.x, acc.y, acc.z, acc.w};
        if (p.y_fp32) {
            float *dst = reinterpret_cast<float *>(p.Y) + (m0 + m) * p.ldy + n0;
            if (n0 + 4 <= p.N) *reinterpret_cast<float4 *>(dst) = acc;
            else
                for (int j = 0; j < 4; ++j)
                    if (n0 + j < p.N) dst[j] = r[j];
        } else {
            __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(p.Y) + (m0 + m) * p.ldy + n0;
            if (n0 + 4 <= p.N) {
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(acc.x, acc.y), h1 = __floats2bfloat162_rn(acc.z, acc.w);
                *reinterpret_cast<uint2 *>(dst) = make_uint2(*reinterpret_cast<const unsigned *>(&h0), *reinterpret_cast<const unsigned *>(&h1));
            } else {
                for (int j = 0; j < 4; ++j)
                    if (n0 + j < p.N) dst[j] = __float2bfloat16_rn(r[j]);
            }
        }
    }
    __syncwarp();
    if (q.split > 1) cluster_sync_all();                    // nobody leaves while its sums are still being read
}

// ------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------
// Shape of a launch: rows per CTA, CTAs per cluster, decode groups.  `cost` estimates the call in record times of
// one CTA: waves of resident CTAs, each its stages plus a fixed part; a cluster's barriers and sums count two records and more
// (256 x 256, b = 4, 8192 rows, 128 tiles of four records: 10.2 us unsplit, 13.9 in pieces of two).
struct StreamPlan {
    StreamParams q;
    size_t smem;
    long long grid;
    long long cost;
};

static StreamPlan plan_with(const Params &p, int split, int sm_count) {
    StreamPlan s;
    s.q.m_tiles = (int)((p.M + ST_MAX_ROWS - 1) / ST_MAX_ROWS);
    s.q.mpad = (int)(((p.M + s.q.m_tiles - 1) / s.q.m_tiles + 15) / 16 * 16);
    s.q.split = split;
    s.q.stages_per = (int)((p.n_stages + split - 1) / split);
    s.q.tmem_cols = s.q.mpad <= 32 ? 32u : (s.q.mpad <= 64 ? 64u : 128u);
    // as many groups as tiles and boxes of X fit: five up to 32 rows, three at 128
    const size_t x = (size_t)s.q.mpad * BK * 2;
    const size_t fixed = 1024 + sizeof(StreamSmem) + 16 + (size_t)(s.q.stages_per + 1) * 16;
    size_t groups = ((size_t)ST_SMEM_CTA - fixed) / (REC_BYTES + x);
    if (groups > (size_t)ST_MAX_GROUPS) groups = ST_MAX_GROUPS;
    if (groups > (size_t)s.q.stages_per) groups = s.q.stages_per < 2 ? 2 : s.q.stages_per;
    s.q.groups = (int)groups;
    s.smem = fixed + groups * (REC_BYTES + x);
    const int resident = 2;
    const long long units = p.n_rec_tiles * s.q.m_tiles;
    s.grid = units * split;
    const long long waves = (s.grid + (long long)resident * sm_count - 1) / ((long long)resident * sm_count);
    s.cost = waves * (s.q.stages_per + 4 + (split > 1 ? 1 + split / 2 : 0));
    return s;
}

template <int BW>
static cudaError_t launch_stream_bw(const CUtensorMap &tmap_x, const Params &p, const StreamPlan &s, cudaStream_t st) {
    auto kern = mwu_gemm_stream_kernel<BW>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, ST_SMEM_CTA);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_chained(kern, dim3((unsigned)s.grid), dim3((unsigned)(s.q.groups * ST_GROUP + 32)), s.smem, st, s.q.split, tmap_x,
                          p, s.q);
}

// The tensor core drops what lies below an accumulator's last place, so a sum loses a little of its magnitude at every
// step, and a sum in pieces less.  fp32 results of 128 x K, b = 4, 40 rows, against fp64: K = 6144 5.7e-7 in eight pieces (5.9e-6 in
// one), 6912 1.4e-6 in four (6.7e-6), 16384 8.0e-6 in two (1.7e-5).  bf16 results hide it.  Results of few rows and of many, which the other
// kernels never split, therefore differ by up to 5.6e-6 where this kernel takes over at K <= 6912; the limits keep it from
// growing in proportion to K above (two pieces without a workspace: 5.1e-6 at 8192, 1.05e-5 at 16384).
static int most_pieces(const Params &p) { return !p.y_fp32 || p.K <= 6144 ? 8 : p.K <= 6912 ? 4 : 2; }

static StreamPlan plan_of(const Params &p, int sm_count, int most) {
    StreamPlan best = plan_with(p, 1, sm_count);
    for (int split = 2; split <= most && split <= p.n_stages; split *= 2) {
        const StreamPlan s = plan_with(p, split, sm_count);
        if (s.cost < best.cost) best = s;
    }
    return best;
}

// activation rows of the TMA box of X
int stream_box_rows(const Params &p, int sm_count) { return plan_of(p, sm_count, most_pieces(p)).q.mpad; }

// A record is decoded once per activation tile of 128 rows, so the path that expands the weights once
// overtakes this one as rows are added.  Measured (us, this kernel / expanding): 16384 x 4096, b = 16:
// 19 / 66 at 16 rows, 29 / 68 at 128, 45 / 68 at 256, 85 / 87 at 512; 4096 x 4096, b = 8: 22 / 37 at 256, 35 / 35 at
// 512; b = 2: 35 / 50 at 256, 58 / 56 at 512.  A small weight stays here longer, while the decodes are few to an
// SM: 1000 x 1216, b = 8, 1024 rows (1216 decodes): 15 / 19; 4096 x 1024, b = 4, 512 rows (2048): 22 / 19.
// So do up to 640 rows of a long reduction where the other path's tiles are few, which work through it alone (bf16, 512 rows:
// 2048 x 8192, b = 16, 16 tiles: 28 / 53; b = 8: 37 / 53; 1024 x 4096, b = 16: 17 / 30; 2048 x 2048, b = 2: 22.5 / 24.8, but
// 2048 x 4096, b = 2, 4096 decodes: 41 / 40; 4096 x 2048, b = 4, 32 tiles: 27.4 / 24.7).  Without a workspace the other path decodes
// once per 512 rows (4096 x 4096, b = 4: 43 / 87, b = 2: 58 / 179; 8192 x 8192, b = 4, 32 tiles: 148 / 281; 16384 x 4096, b = 16, 64 tiles: 85 / 74).
// bf16 results of more than 256 rows stay only while the tiles of 128 x 128 outputs are one to an SM, or two where the other path has
// much to expand for its rows, or nothing expanded to work on (us, this kernel / the other: 1024 x 64, b = 4, 8192 rows, 512 tiles: 19.5 / 12.1;
// 256 x 256, 16384 rows, 256 tiles: 14.2 / 11.1; 128 x 192, b = 16, 32768 rows, 256 tiles: 11.5 / 12.7; 4096 x 256, 777 rows, 224 tiles: 11.5 / 12.0;
// without a workspace 512 x 256, 8192 rows, 256 tiles: 14.1 / 18.8, 128 x 192, 256 tiles: 11.0 / 10.6).  Nor where a reduction of less
// than 1024 has to be split to two CTAs an SM (512 x 512, b = 4, 4096 rows: 15.9 / 12.0; 2048 x 512, 300 rows: 12.1 / 13.4).
// fp32 results, which the paths that expand store in pieces of a row, stay (512 x 512, 2048 rows: 13.1 / 15.4), but not where the kernel
// of the short reductions takes over, whose fp32 output leaves through TMA (from two tiles of 128 x 256 outputs an SM, this kernel / that one:
// 256 x 64, b = 4, 37900 rows 20.7 / 14.7, 128 x 64, 38000 rows 11.0 / 10.2, 80000 rows 21.9 / 15.5; 16384 x 64, 1024 rows 33.6 / 18.0; 640 x 128, 12801 rows
// 21.6 / 15.5; 128 x 256, 38000 rows 24.9 / 15.7; b = 16 18.4 / 13.7, 10.4 / 9.9, 19.4 / 15.3, 28.9 / 17.4, 19.4 / 14.5, 20.0 / 14.9).
// Where it may not split as it would (128 x 7168, 55 rows, fp32: 16 us in eight pieces, 43 in two, 41 expanding), the
// other path is taken if the caller's workspace allows it (can_expand).
bool resident_eligible(const Params &p, int sm_count, bool can_expand);      // mwu_gemm5.cu

bool stream_eligible(const Params &p, int sm_count, bool can_expand) {
    const StreamPlan s = plan_of(p, sm_count, most_pieces(p));
    if (can_expand && most_pieces(p) < 8 && 2 * s.cost > 3 * plan_of(p, sm_count, 8).cost) return false;
    if (p.M <= 256) return true;
    const long long tiles = p.n_rec_tiles * s.q.m_tiles;
    if (!p.y_fp32 && p.M <= 640 && p.n_stages >= 32) {
        const long long wide = (p.n_rec_tiles + 1) / 2, pairs = sm_count / 2;          // tiles of a CTA pair along the weight rows
        if (can_expand ? 4 * wide * ((p.M + 255) / 256) <= pairs && (p.bw > 2 || tiles * p.n_stages <= 2048)
                       : 2 * wide * ((p.M + 511) / 512) <= pairs) return true;
    }
    if (tiles * p.n_stages > 9ll * sm_count) return false;
    if (p.y_fp32) return !resident_eligible(p, sm_count, can_expand);
    if (can_expand && p.n_stages < 16 && s.q.split > 1 && s.grid > sm_count && p.M > 512) return false;
    const bool two = can_expand ? p.n_rec_tiles == 1 || s.q.m_tiles <= 8 : p.n_rec_tiles > 1 || p.n_stages > 1;
    return tiles <= (two ? 2ll : 1ll) * sm_count;
}

cudaError_t launch_stream(int bw, const CUtensorMap &tmap_x, const Params &p, int sm_count, cudaStream_t st) {
    const StreamPlan s = plan_of(p, sm_count, most_pieces(p));
    switch (bw) {
        case 2: return launch_stream_bw<2>(tmap_x, p, s, st);
        case 4: return launch_stream_bw<4>(tmap_x, p, s, st);
        case 8: return launch_stream_bw<8>(tmap_x, p, s, st);
        default: return launch_stream_bw<16>(tmap_x, p, s, st);
    }
}

}  // namespace gemm
}  // namespace mwu
