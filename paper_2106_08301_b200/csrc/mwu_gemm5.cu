// mwu_gemm with a short reduction (K <= 256) and many activation rows: a CTA keeps a tile of the weights in shared memory.
//
// A 1x1 convolution as a product (256 weight columns, 1024 rows, 200704 pixels) has four k stages to a tile of outputs, so what
// happens between two tiles counts as much as the multiplication.  The two-operand kernel brought both operands of every tile
// from L2 (822 MB for that product) and passed each accumulator between the two CTAs of a pair, whose messages queue
// behind the outgoing output: 2.2 us a tile of 256 x 256 against 1.1 of tensor time, 132 us with expanding the weights (150 where the
// activations are new in every call).
// Here a CTA works alone on tiles of 128 activation rows x 256 weight rows.  It decodes the weights of its tile column once,
// straight from the packed form (no expansion, no workspace), and then only activations stream in: 411 MB of output, 103 to 118 us
// (the longer the row of calls the slower, as of the other kernel), 125 with new activations.
// What bounds it: activations in (through four slots for K = 256) and output out at the same time; with the stores left out 81
// us, with the loads left out 88, the epilogue and its stores alone 81; the DRAM traffic alone (457 MB) would take 73.
//
// The tiles of a weight tile column follow one another in the list that is dealt out, in equal shares, to the CTAs, so a CTA meets
// one weight tile or two.  In a column neighbouring CTAs take neighbouring activation tiles at the same time, and so do the
// CTAs of the other columns: L2 holds the activations, and whole rows of the output are written at a time (filling 411 MB in this
// order takes 68 us, 78 with a run of consecutive activation tiles to a CTA).
// Roles: warp 0 TMA producer (activation stages), warp 1 tensor memory and MMAs, warps 2 to 9 decode the weights and
// then are the epilogue (two warps to a 32-lane quarter, 128 columns each; accumulators double-buffered in tensor memory; the
// output leaves through TMA stores of 32 rows x 128 bytes).
// Every wait on an mbarrier is bounded; when one runs out the kernel raises MWU_DEV_TIMEOUT, waits for its copies in
// flight, frees tensor memory and returns.
#include "mwu_gemm_dev.cuh"

namespace mwu {
namespace gemm {

constexpr int R_EPI_WARPS = 8;
constexpr int R_THREADS = 32 * (2 + R_EPI_WARPS);
constexpr int R_MAX_STAGES = 4;
constexpr int R_W_STAGE = 2 * REC_BYTES;                // 256 weight rows of a k stage
constexpr int R_EPI_BYTES = 4096;                       // of a warp: 32 rows x 64 bf16 columns
constexpr int R_MAX_SLOTS = 8;                          // activation stages in flight: what fits beside one stage of weights
constexpr int R_DEC = 64;                               // threads that decode a record together

struct ResidentSmem {
    unsigned long long full[R_MAX_SLOTS], empty[R_MAX_SLOTS], tfull[2], tempty[2], wfull, drain;
    unsigned tmem_base;
    int abort;
    int drain_abort;
};

// One record into its tile, by R_DEC threads: zeros, then the unified and the dense blocks (so pruned blocks need no list).
// Bound by trips to L2 and by fetching its own instructions: entries of both lists travel together, the first while the tile is
// zeroed, in one loop whose code is there once.  (One list after the other, from zeroing on: 256 x 256, b = 16, 37900 rows 17.4 us, so
// 16.0; b = 8 17.9 / 16.3, b = 4 18.7 / 17.6, b = 2 23.1 / 20.2; 1024 x 256, b = 8, 200704 rows 104.5 / 103.  Entries at a time: more dense ones take b = 4
// from 19.6 to 20.2 us where all blocks are dense, twice as many unified ones b = 2 from 20.2 to 21.9; b = 8 spills 76 bytes with eight,
// six, which spill none, take 17.7 instead of 16.0 us for 512 x 192 of dense blocks.)
template <int BW>
__device__ __forceinline__ void decode_record(unsigned char *tile, const uint4 a, const uint4 b, const Params &p, unsigned t0, int group) {
    constexpr unsigned OFF_MASK = DecodeCfg<BW, R_DEC>::OFF_MASK;
    constexpr int WORDS = BW / 2;
    constexpr unsigned UB = BW == 16 ? 4 : BW == 2 ? 12 : 8, DB = BW == 16 ? 4 : BW == 2 ? 16 : 8;     // entries of a thread at a time
    // ranges that do not lie inside the sections, or hold more than a record: not touched
    const bool bad = a.x > b.x || b.x > p.n_unified || a.y > b.y || b.y > p.n_dense ||
                     (b.x - a.x) + (b.y - a.y) > (unsigned)(kTileRows * BK / BW);
    const unsigned n_u = bad ? 0u : b.x - a.x, n_d = bad ? 0u : b.y - a.y;
    const uint2 *ul = reinterpret_cast<const uint2 *>(p.packed + p.off_ulist) + (bad ? 0u : a.x);
    const unsigned short *dpos = reinterpret_cast<const unsigned short *>(p.packed + p.off_dpos) + (bad ? 0u : a.y);
    const unsigned char *pay = p.packed + p.off_dpay + (size_t)(bad ? 0u : a.y) * (2 * BW);
    unsigned u0 = 0, d0 = 0;
#pragma unroll 1
    do {
        uint2 ent[UB];
        unsigned off[DB], v[DB][WORDS];
        if (u0 < n_u) {
#pragma unroll
            for (unsigned k = 0; k < UB; ++k) {
                const unsigned e = u0 + k * R_DEC + t0;
                if (e < n_u) ent[k] = __ldg(ul + e);
            }
        }
        if (d0 < n_d) {
#pragma unroll
            for (unsigned k = 0; k < DB; ++k) {
                const unsigned e = d0 + k * R_DEC + t0;
                if (e >= n_d) continue;
                off[k] = __ldg(dpos + e);
                ld_words<WORDS>(pay + (size_t)e * (2 * BW), v[k]);
            }
        }
        if (u0 == 0) {
            uint4 *z = reinterpret_cast<uint4 *>(tile) + t0;
#pragma unroll
            for (int t = 0; t < REC_BYTES / 16 / R_DEC; ++t) z[t * R_DEC] = make_uint4(0, 0, 0, 0);
            group_barrier<R_DEC>(1 + group);
        }
        if (u0 < n_u) {
#pragma unroll
            for (unsigned k = 0; k < UB; ++k) {
                if (u0 + k * R_DEC + t0 >= n_u) break;
                unsigned w[WORDS];
                unified_words<WORDS>(ent[k], w);
                st_words<WORDS>(tile, ent[k].y & OFF_MASK, w);
            }
        }
        if (d0 < n_d) {
#pragma unroll
            for (unsigned k = 0; k < DB; ++k) {
                if (d0 + k * R_DEC + t0 >= n_d) break;
                st_words<WORDS>(tile, off[k] & OFF_MASK, v[k]);
            }
        }
        u0 += UB * R_DEC;
        d0 += DB * R_DEC;
    } while (u0 < n_u || d0 < n_d);
    if (bad) atomicOr(p.dev_status, (unsigned)MWU_DEV_BOUNDS);
}

template <int BW>
__global__ void __launch_bounds__(R_THREADS, 1)
mwu_gemm_resident_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_y,
                         const __grid_constant__ Params p, const int slots, const int boxes) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    MWU_CHECK_HEADER(p);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sW = smem_raw + smem_pad_1024(smem_raw);
    const int n_stages = (int)p.n_stages;
    unsigned char *sX = sW + n_stages * R_W_STAGE;
    unsigned char *stage_buf = sX + slots * AH_BYTES;
    ResidentSmem *sm = reinterpret_cast<ResidentSmem *>(stage_buf + R_EPI_WARPS * boxes * R_EPI_BYTES);
    volatile int *abort = &sm->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < R_MAX_SLOTS; ++s) {
            mbar_init(smem_u32(&sm->full[s]), 1);
            mbar_init(smem_u32(&sm->empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&sm->tfull[b]), 1);
            mbar_init(smem_u32(&sm->tempty[b]), R_EPI_WARPS);
        }
        mbar_init(smem_u32(&sm->wfull), R_EPI_WARPS);
        mbar_init(smem_u32(&sm->drain), 1);
        sm->abort = 0;
        sm->drain_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) {
        tmem_alloc(smem_u32(&sm->tmem_base), 512);
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = *reinterpret_cast<volatile unsigned *>(&sm->tmem_base);

    const uint4 *recs = reinterpret_cast<const uint4 *>(p.packed + p.off_rec);
    const unsigned m_tiles = (unsigned)((p.M + BMH - 1) / BMH), n_tiles = (unsigned)((p.n_rec_tiles + 1) / 2);
    const unsigned long long total = (unsigned long long)m_tiles * n_tiles;
    const unsigned long long t_begin = total * blockIdx.x / gridDim.x, t_end = total * (blockIdx.x + 1) / gridDim.x;
    // A weight tile's activation tiles in the order of its runs: run j takes tiles j, j + runs, j + 2 runs, ...
    const unsigned runs = min((gridDim.x + n_tiles - 1u) / n_tiles, m_tiles), most = (m_tiles + runs - 1u) / runs;
    const unsigned longer = m_tiles - (most - 1u) * runs;       // runs of `most` tiles; the others have one less
    // live slices of weight tile nt: four bits a stage, the OR over its (one or two) records
    auto live_of = [&](unsigned nt) -> unsigned {
        unsigned l = 0;
        if (lane < n_stages) {
            l = __ldg(&recs[(size_t)(nt * 2u) * n_stages + lane].w) & 0xFu;
            if (nt * 2u + 1u < (unsigned long long)p.n_rec_tiles) l |= __ldg(&recs[(size_t)(nt * 2u + 1u) * n_stages + lane].w) & 0xFu;
            l <<= 4 * lane;
        }
        return __reduce_or_sync(0xffffffffu, l);
    };
    // begin(weight tile) and then tile(activation tile) for all of its tiles, weight tile by weight tile of this CTA's share; until
    // one of them returns false
    auto for_tiles = [&](auto begin, auto tile) {
        for (unsigned long long t = t_begin; t < t_end;) {
            const unsigned nt = (unsigned)(t / m_tiles), x = (unsigned)(t - (unsigned long long)nt * m_tiles);
            const unsigned n = (unsigned)min((unsigned long long)(m_tiles - x), t_end - t);
            unsigned j, s;                                      // run, and place in it
            if (x < longer * most) { j = x / most; s = x - j * most; }
            else { const unsigned y = x - longer * most; j = longer + y / (most - 1u); s = y % (most - 1u); }
            if (!begin(nt)) return;
            for (unsigned i = 0; i < n; ++i) {
                if (!tile(s * runs + j)) return;
                if (++s >= (j < longer ? most : most - 1u)) { s = 0; ++j; }
            }
            t += n;
        }
    };

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        unsigned slot = 0, phase = 0, issued = 0, live = 0;
        unsigned column = 0;
        // Stages that the L2 prefetch below brings: those that some weight tile multiplies, the first 1024 records asked (a stage
        // at a time is 103 MB in the product named there: everything pruned 106 us with all of them fetched, 90 by expanding).
        const bool ahead_too = n_tiles >= (unsigned)(p.y_fp32 || n_stages == 1 ? n_stages : 2);
        const unsigned all = (1u << n_stages) - 1u, n_rec = (unsigned)p.n_rec_tiles * (unsigned)n_stages;
        unsigned wanted = ahead_too ? 0u : all;
#pragma unroll 1
        for (unsigned i0 = 0; wanted != all && i0 < n_rec; i0 += 128) {
            if (i0 == 1024) { wanted = all; break; }
            unsigned l = 0;
#pragma unroll
            for (unsigned k = 0; k < 4; ++k) {
                const unsigned i = i0 + 32u * k + (unsigned)lane;
                if (i < n_rec && (__ldg(&recs[i].w) & 0xFu)) l |= 1u << (i % (unsigned)n_stages);
            }
            wanted |= __reduce_or_sync(0xffffffffu, l);
        }
        for_tiles([&](unsigned nt) { live = live_of(nt); column = nt; return true; }, [&](unsigned mt) {
            // The column's next tile to L2, a stage of it by one CTA of the columns that take it at the same time: the slots here do not
            // cover a trip to DRAM behind the output (200704 rows, b = 8, us without and so: 1024 x 256 133 / 107, 768 x 256 92 / 82, 512 x 256 69 / 64,
            // 512 x 192 62 / 59, 2304 x 192 228 / 185; one weight tile: 256 x 192 38.5 / 39.0, 128 x 256 32.9 / 33.2, but 64 x 64 17.7 / 17.0; fp32 with fewer weight
            // tiles than stages: 768 x 256 136 / 139, 512 x 256 110 / 113).  Two tiles ahead 111 where one took 107.
            const unsigned ahead = mt + runs;
            if (ahead_too && ahead < m_tiles) {
                unsigned who = ahead * (unsigned)n_stages % n_tiles;
                for (int ks = 0; ks < n_stages; ++ks) {
                    if (who == column && ((wanted >> ks) & 1u) && elect_one()) tma_prefetch_2d(&tmap_x, ks * BK, (int)(ahead * BMH));
                    __syncwarp();
                    if (++who == n_tiles) who = 0;
                }
            }
            for (int ks = 0; ks < n_stages; ++ks) {
                if (!((live >> (4 * ks)) & 0xFu)) continue;
                const unsigned bar = smem_u32(&sm->full[slot]);
                if (!warp_wait_spin(smem_u32(&sm->empty[slot]), phase ^ 1u, abort)) return false;
                if (elect_one()) {
                    mbar_expect_tx(bar, AH_BYTES);
                    tma_load_2d(smem_u32(sX + slot * AH_BYTES), &tmap_x, bar, ks * BK, (int)(mt * BMH));
                }
                __syncwarp();
                ++issued;
                if (++slot == (unsigned)slots) { slot = 0; phase ^= 1u; }
            }
            return true;
        });
        // copies still on their way land before this CTA's shared memory goes away
        for (unsigned s = 0; s < (unsigned)slots && s < issued; ++s)
            mbar_wait(smem_u32(&sm->full[s]), ((issued - 1u - s) / (unsigned)slots) & 1u, &sm->drain_abort);
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        const unsigned long long xdesc = make_desc(smem_u32(sX)), wdesc = make_desc(smem_u32(sW));
        unsigned slot = 0, phase = 0, k = 0, wphase = 0, live = 0, idesc = 0;
        for_tiles([&](unsigned nt) {
            live = live_of(nt);
            idesc = make_idesc(nt * 2u + 1u < (unsigned long long)p.n_rec_tiles ? 256 : 128);
            if (!warp_wait_spin(smem_u32(&sm->wfull), wphase, abort)) return false;
            wphase ^= 1u;
            return true;
        }, [&](unsigned) {
            const unsigned buf = k & 1u;
            if (!warp_wait_spin(smem_u32(&sm->tempty[buf]), ((k >> 1) & 1u) ^ 1u, abort)) return false;
            tc_fence_after();
            unsigned acc = 0;
            for (int ks = 0; ks < n_stages; ++ks) {
                const unsigned l = (live >> (4 * ks)) & 0xFu;
                if (!l) continue;
                if (!warp_wait_spin(smem_u32(&sm->full[slot]), phase, abort)) return false;
                tc_fence_after();
                const unsigned long long a = xdesc + slot * (AH_BYTES / 16), b = wdesc + (unsigned)ks * (R_W_STAGE / 16);
                if (elect_one()) {
                    unsigned add = acc;
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4) {
                        if ((l >> k4) & 1u) {
                            umma_bf16(tmem_base + buf * 256u, a + (unsigned long long)(k4 * 2), b + (unsigned long long)(k4 * 2), idesc, add);
                            add = 1u;
                        }
                    }
                    umma_commit(smem_u32(&sm->empty[slot]));
                }
                __syncwarp();
                acc = 1u;
                if (++slot == (unsigned)slots) { slot = 0; phase ^= 1u; }
            }
            if (elect_one()) {
                if (acc) umma_commit(smem_u32(&sm->tfull[buf]));
                else mbar_arrive(smem_u32(&sm->tfull[buf]));
            }
            __syncwarp();
            ++k;
            return true;
        });
        // nothing this warp issued may be running when tensor memory is freed
        if (elect_one()) umma_commit(smem_u32(&sm->drain));
        __syncwarp();
        mbar_wait(smem_u32(&sm->drain), 0, &sm->drain_abort);
        __syncwarp();
    } else {
        // ---------------- decode, then epilogue ----------------
        const int e = (int)threadIdx.x - 64, group = e / R_DEC;
        const unsigned t0 = (unsigned)e % R_DEC;
        const int quarter = warp & 3;                       // tensor-memory lanes (activation rows) this warp may read
        const int chalf = (warp - 2) >> 2;                  // which 128 columns
        unsigned char *const stg = stage_buf + (warp - 2) * boxes * R_EPI_BYTES;
        // Place of the next store's box.  Two boxes alternate from store to store, whichever tiles those belong to: a tile may
        // have an odd number of them (weight rows that end inside a box), and bulk_wait_read_1 leaves the latest store unwaited for.
        unsigned box_at = 0;
        const unsigned box_flip = boxes == 2 ? R_EPI_BYTES : 0;
        unsigned k = 0;
        bool any = false, dead = false;
        long long ncol0 = 0;
        // A warp that ran out of time goes on without touching an accumulator, so that the barriers of the decode stay matched.
        for_tiles([&](unsigned nt) {
            const unsigned live = live_of(nt);
            const int nrec = nt * 2u + 1u < (unsigned long long)p.n_rec_tiles ? 2 : 1;
            any = live && chalf < nrec;
            ncol0 = (long long)nt * 256 + chalf * 128;
            // (what was multiplied with the weights before has been waited for: the last tile's accumulator)
            for (int i = group; i < n_stages * nrec; i += R_EPI_WARPS * 32 / R_DEC) {
                const int ks = i / nrec, r = i - ks * nrec;
                if (!((live >> (4 * ks)) & 0xFu)) continue;
                const uint4 *rec = recs + (size_t)(nt * 2u + (unsigned)r) * n_stages + ks;
                decode_record<BW>(sW + ks * R_W_STAGE + r * REC_BYTES, __ldg(rec), __ldg(rec + 1), p, t0, group);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sm->wfull));
            return true;
        }, [&](unsigned mt) {
            if (dead) return true;
            const unsigned buf = k & 1u;
            const bool ok = mbar_wait(smem_u32(&sm->tfull[buf]), (k >> 1) & 1u, abort);
            dead = !__all_sync(0xffffffffu, ok);
            if (dead) return true;
            ++k;
            tc_fence_after();
            const long long mrow0 = (long long)mt * BMH + quarter * 32;
            const unsigned trow = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * 256u + (unsigned)(chalf * 128);
            auto load = [&](int q, unsigned (&v)[32]) {
                if (any) tmem_ld32_issue(trow + (unsigned)(32 * q), v);
                else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0u;
                }
            };
            auto hand_back = [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sm->tempty[buf]));
            };
            // 32 rows of 128 bytes leave through a box of the warp; the tensor map clips them
            auto store_box = [&](const unsigned (&w)[32], int col, int row) {
                unsigned char *box = stg + box_at;
                box_at ^= box_flip;
                if (lane == 0) { if (boxes == 2) bulk_wait_read_1(); else bulk_wait_read(); }      // the last store out of it has read it
                __syncwarp();
                stage_row64(w, box, lane);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&tmap_y, smem_u32(box), col, row);
                    bulk_commit();
                }
            };
            if (!p.y_fp32) {
                unsigned w[2][32];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    unsigned v[32];
                    load(q, v);
                    tmem_ld_wait(v);
                    pack_bf16(v, w[q >> 1] + 16 * (q & 1));
                }
                hand_back();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (ncol0 + 64 * h >= p.N || mrow0 >= p.M) break;
                    store_box(w[h], (int)(ncol0 + 64 * h), (int)mrow0);
                }
            } else {
                // boxes of 32 columns
#pragma unroll 1
                for (int q = 0; q < 4; ++q) {
                    unsigned v[32];
                    load(q, v);
                    tmem_ld_wait(v);
                    if (q == 3) hand_back();
                    if (ncol0 + 32 * q >= p.N || mrow0 >= p.M) continue;
                    store_box(v, (int)(ncol0 + 32 * q), (int)mrow0);
                }
            }
            return true;
        });
        if (lane == 0) bulk_wait_all();                     // this warp's tile stores are done
        __syncwarp();
    }

    // teardown
    tc_fence_before();
    __syncthreads();
    // after the barrier: a role that finished its own work early must still see a flag raised later
    if ((*abort || sm->drain_abort) && threadIdx.x == 0) atomicOr(p.dev_status, (unsigned)MWU_DEV_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------
constexpr size_t R_SMEM_MAX = 227 * 1024;
static_assert((R_SMEM_MAX - 1024 - R_W_STAGE - 2 * R_EPI_WARPS * R_EPI_BYTES - sizeof(ResidentSmem)) / AH_BYTES <= R_MAX_SLOTS,
              "one stage of weights leaves most slots");

// From two tiles an SM on, so that decoding the weights is shared (us, this kernel / expanding the weights: 256 x 256, b = 16, 37888
// rows, 296 tiles: 15.1 / 17.1; 256 x 192, b = 2: 17.4 / 21.9; 65536 x 256, b = 2, 300 rows, three tiles to a weight tile: 46 / 58; 4096 x 128,
// b = 4, 4096 rows, 512 tiles: 13.9 / 17.7; 1024 x 256, b = 8, 20000 rows, 628 tiles: 19.5 / 22.2, 200704 rows 103 / 132 (fused, without a
// workspace: 215); 640 x 192, 200704 rows: 62 / 94, 65536 rows of fp32 output 52 / 83; 96 x 256, 200704 rows: 33 / 40).
// Narrow blocks that are mostly in one list take many trips to L2.  Where the weights could be expanded, few weight tiles (whose
// activations are not brought to L2 ahead) then need more than four tiles an SM, and more weight tiles than SMs more than five tiles each:
// 256 x 256, all dense, b = 4, 297 tiles 19.6 / 17.7, 592 tiles 24.8 / 24.2, 740 tiles 27.9 / 27.5; b = 2 22.9 / 20.3, 27.9 / 26.0, 31.1 / 29.5; 65536 x 256, b = 4,
// all dense, four tiles to a weight tile 47 / 41, seven 59.4 / 59.1.  Not so with 70 % of the blocks dense and b = 2 (256 x 256, 297 tiles 21.7 / 23.5),
// half of them and b = 4 (17.6 / 17.9), four weight tiles (1024 x 256, b = 4, all dense, 372 tiles 18.2 / 18.3) or two stages (40000 x 128, b = 4, all
// dense, three tiles to a weight tile 20.9 / 24.6).
bool resident_eligible(const Params &p, int sm_count, bool can_expand) {
    if (p.n_stages > R_MAX_STAGES) return false;
    const long long n_tiles = (p.n_rec_tiles + 1) / 2, tiles = (p.M + BMH - 1) / BMH * n_tiles;
    if (can_expand && !p.y_fp32 && p.n_stages >= 3) {
        const long long blocks = p.n_rec_tiles * p.n_stages * (kTileRows * BK / p.bw), longest = p.n_unified > p.n_dense ? p.n_unified : p.n_dense;
        const bool one_list = p.bw == 2 ? 4ll * p.n_dense > 3 * blocks : p.bw == 4 && 5 * longest > 3 * blocks;
        if (one_list && (n_tiles < p.n_stages ? tiles <= 4ll * sm_count : n_tiles > sm_count && tiles <= 5 * n_tiles)) return false;
    }
    return tiles >= 2ll * sm_count;
}

template <int BW>
static cudaError_t launch_resident_bw(const CUtensorMap &tmap_x, const CUtensorMap &tmap_y, const Params &p, int sm_count, cudaStream_t st) {
    auto kern = mwu_gemm_resident_kernel<BW>;
    // Two boxes a warp where the weights leave room for them and four activation stages (us with one and two boxes: 200704 x 192 x 1024
    // 116 / 107, 200704 x 192 x 640 78 / 73; with two boxes and two stages for K = 256, 200704 x 256 x 1024: 138).
    const int boxes = p.n_stages <= 3 ? 2 : 1;
    const size_t fixed = 1024 + (size_t)p.n_stages * R_W_STAGE + (size_t)(R_EPI_WARPS * boxes * R_EPI_BYTES) + sizeof(ResidentSmem);
    const int slots = (int)((R_SMEM_MAX - fixed) / AH_BYTES);
    const size_t smem = fixed + (size_t)slots * AH_BYTES;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R_SMEM_MAX);
    if (e != cudaSuccess) return e;
    // Equal shares on all SMs make some CTAs change weights on the way, which costs them about two tiles; with the same number of
    // CTAs to every weight tile none does, but some SMs may stay without a CTA (640 x 192, 200704 rows, 49 CTAs to each of three
    // tiles: 92.7 / 78.2 us; 2304 x 256, 65536 rows, 16 to each of nine: 101 / 92).
    const long long m_tiles = (p.M + BMH - 1) / BMH, n_tiles = (p.n_rec_tiles + 1) / 2, each = sm_count / n_tiles;
    long long grid = sm_count;
    if (each > 0 && (m_tiles + each - 1) / each <= (m_tiles * n_tiles + sm_count - 1) / sm_count + 2) grid = each * n_tiles;
    count_launch();
    return launch_chained(kern, dim3((unsigned)grid), dim3(R_THREADS), smem, st, 1, tmap_x, tmap_y, p, slots, boxes);
}

cudaError_t launch_resident(int bw, const CUtensorMap &tmap_x, const CUtensorMap &tmap_y, const Params &p, int sm_count, cudaStream_t st) {
    switch (bw) {
        case 2: return launch_resident_bw<2>(tmap_x, tmap_y, p, sm_count, st);
        case 4: return launch_resident_bw<4>(tmap_x, tmap_y, p, sm_count, st);
        case 8: return launch_resident_bw<8>(tmap_x, tmap_y, p, sm_count, st);
        default: return launch_resident_bw<16>(tmap_x, tmap_y, p, sm_count, st);
    }
}

}  // namespace gemm
}  // namespace mwu
