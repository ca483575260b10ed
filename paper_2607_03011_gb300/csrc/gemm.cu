// gemm.cu -- batched split-precision GEMM on tcgen05 tensor cores (sm_103a).
//
// Computes, for every matrix b of a group and every BM x BN output tile,
//     D[b](i, j) = sum_k A[b](i, k) B[b](j, k)
// where an fp32 operand is carried as 16-bit planes hi = round(x), lo = round(x - hi)
// (bf16 or fp16, chosen per launch).  The tensor core sums hi*hi, plus hi*lo_B when B
// carries a lo plane and lo_A*hi when A does, into an fp32 accumulator in tensor memory:
// three passes give ~16 (bf16) or ~22 (fp16) significant bits per operand, two passes
// keep one operand at 11 bits (fp16).  The polar iteration uses three bf16 passes on
// the unnormalised pseudo-gradient (iteration 0) and on the final polish step, and two
// fp16 passes elsewhere (the operand that is not split only perturbs the iterate's
// spectrum, which later steps correct).
//
// Roles (352 threads): warp 0 issues TMA loads into a ring of shared
// memory stages; warp 1 owns the tensor-memory accumulator and issues tcgen05.mma
// from one thread; warps 2..9 drain the accumulator (tcgen05.ld) and run the
// epilogue; warp 10 decodes the tiles for all of them, through a queue in shared memory.
// Stage hand-off uses mbarriers: `full` (TMA bytes landed), `empty` (the MMAs reading a stage
// finished, via tcgen05.commit), `tfull` / `tempty` (an accumulator written / read).
//
// Operand layouts: K-major operands (K contiguous in global memory) use swizzled
// tiles BK deep; MN-major operands (M or N contiguous) use 128-byte swizzled tiles of
// 64 MN-elements x BK rows, two (A) or four (B) boxes per stage.  This lets X^T X,
// X P and P X all read the row-major iterate without transposes.  The layout is a
// property of each group, so one launch can mix them (the Grams X^T X of tall and
// X X^T of wide matrices share a launch).
#include <cstdio>

#include "gemm_tile.cuh"
#include "per_device.h"

namespace isoloco {

// Active-tile prefix of the launch: group i owns active tiles [pre[i], pre[i + 1]).
__device__ __forceinline__ void active_prefix(const GemmParams& p, int* pre) {
    pre[0] = 0;
    for (int i = 0; i < p.num_groups; ++i) {
        const GemmGroup& g = p.g[i];
        const int mats = p.list ? p.cnt[g.bucket] : g.batch;
        pre[i + 1] = pre[i] + mats * (g.sym ? g.tiles_sym : g.tiles_m * g.tiles_n) * g.splits;
    }
}

__device__ __forceinline__ TileFlags tile_flags(const GemmParams& p) {
    return {p.gate, p.in_f16, p.out_f16, p.split_on_polish, p.gram_y, p.poly_horner, p.unit_scale};
}

// Decodes active tile t (group gi) for the CTA of rank `crank` in its pair.  Returns false
// when the matrix does no work in this launch.
template <int EPI>
__device__ __forceinline__ bool decode_tile(const GemmParams& p, const int* pre, int t, uint32_t crank, int& gi,
                                            TileInfo& ti) {
    gi = 0;
    while (gi + 1 < p.num_groups && t >= pre[gi + 1]) ++gi;
    const GemmGroup& g = p.g[gi];
    int local = t - pre[gi];
    const int split = local % g.splits;
    local /= g.splits;
    const int ntiles = g.sym ? g.tiles_sym : g.tiles_m * g.tiles_n;
    const int j = local / ntiles;
    const int b = p.list ? p.list[g.mat_base + j] : j;
    if (b >= g.batch) return false;
    const MatState* st = p.state + g.mat_base + b;
    if (g.gate_fb && st->final_buf != g.gate_fb - 1) return false;
    if (p.gate == kGateActive && st->done) return false;
    if (p.gate == kGateStep && st->mode == 0) return false;
    setup_tile<EPI>(tile_flags(p), g, st, b, local % ntiles, split, crank, ti);
    return true;
}

// One tile, decoded by the scheduler for the other roles (gi < 0: no more tiles).
struct GemmTile {
    TileInfo ti;
    int gi;
};

// Persistent kernel, one instantiation per epilogue.  The grid is made of clusters of two CTAs
// (ranks 0 and 1, on neighbouring SMs); cluster c processes tiles c, c + clusters, ...
// and both CTAs walk that sequence together: each loads its rows of A and its half of B,
// the TMA bytes of both complete on rank 0's `full` barrier, rank 0 alone issues the
// cta_group::2 MMAs, whose commits arrive on the `empty` / `tfull` barriers of both CTAs,
// and each CTA's epilogue drains its own half of the accumulator and reports to rank 0's
// `tempty`.  The TMA ring runs continuously across tile boundaries, and the accumulator
// is double buffered in tensor memory (2 x 256 columns): the epilogue of one tile
// overlaps the MMAs of the next.
template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1) k_gemm_split(const __grid_constant__ GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint8_t* staging = smem + kRingBytes;  // kEpiWarps x kStageBlocks blocks
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kRingBytes + kEpiStagingBytes);
    uint64_t* empty = full + kMaxStages;
    uint64_t* tfull = empty + kMaxStages;  // [2] accumulator buffer ready for the epilogue
    uint64_t* tempty = tfull + 2;        // [2] accumulator buffer released by the epilogue
    uint64_t* drain = tempty + 2;        // teardown: every issued MMA has completed
    uint64_t* tq_full = drain + 1;       // [kTileQueue] tile written by the scheduler
    uint64_t* tq_empty = tq_full + kTileQueue;  // [kTileQueue] read by the TMA, MMA and epilogue warps
    GemmTile* tq = reinterpret_cast<GemmTile*>(tq_empty + kTileQueue);
    int* pre = reinterpret_cast<int*>(tq + kTileQueue);  // [kMaxGroups + 1] active-tile prefix
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(pre + kMaxGroups + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    static_assert(8 * (2 * kMaxStages + 5 + 2 * kTileQueue) + kTileQueue * sizeof(GemmTile) + 4 * (kMaxGroups + 3) <=
                      kGemmTailBytes, "shared memory behind the staging blocks");

    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);  // warp-uniform
    const int lane = threadIdx.x & 31;
    const uint32_t crank = cluster_ctarank();  // rank in the CTA pair
    const bool leader = crank == 0;            // issues the MMAs
    // ring geometry of this launch: room for the planes its tiles can load
    const uint32_t stage_stride = kTileABytes * (p.a_split || p.split_on_polish ? 2u : 1u) +
                                  kTileBBytes * (p.b_split || p.split_on_polish ? 2u : 1u);
    const int nstages = min(kMaxStages, static_cast<int>(kRingBytes / stage_stride));

    if (threadIdx.x == 0) {
        for (int s = 0; s < nstages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], kEpiWarps * 2);  // one arrival per epilogue warp of the pair
        }
        mbar_init(drain, 1);
        for (int q = 0; q < kTileQueue; ++q) {
            mbar_init(&tq_full[q], 1);
            mbar_init(&tq_empty[q], kTileReaders);  // the TMA and MMA threads, a lane per epilogue warp
        }
        active_prefix(p, pre);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 2 * kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers exist before either signals the other's
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ================= TMA producer (one thread)
        if (elect_one()) {
            const uint32_t sbase = smem_u32(smem);
            const uint32_t fbar0 = mapa_shared(smem_u32(full), 0);
            RingPos pos = {0, 0u};
            bool wrapped = false;  // the ring has been filled once
            int prefetched = -1;
            int q = 0;
            uint32_t qphase = 0;
            for (;;) {
                if (!mbar_wait(&tq_full[q], qphase)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                const TileInfo& ti = tq[q].ti;
                const int gi = tq[q].gi;
                if (gi < 0) break;
                // (after a timeout the queue only drains)
                if (ti.run_mma && !*abort_flag) {
                    const GemmGroup& g = p.g[gi];
                    if (prefetched != gi) {
                        tma_prefetch_desc(g.a_hi);
                        tma_prefetch_desc(g.b_hi);
                        if (ti.a_split) tma_prefetch_desc(g.a_hi + 1);
                        if (ti.b_split) tma_prefetch_desc(g.b_hi + 1);
                        prefetched = gi;
                    }
                    const bool ok = load_tile(g, ti, sbase, stage_stride, nstages, full, empty, fbar0, crank, pos);
                    wrapped |= pos.phase != 0u || ti.kb_end - ti.kb_begin >= nstages;
                    if (!ok) {
                        *abort_flag = 1;
                        atomicOr(p.err, kErrTimeout);
                    }
                }
                mbar_arrive(&tq_empty[q]);
                if (++q == kTileQueue) {
                    q = 0;
                    qphase ^= 1u;
                }
            }
            if (*abort_flag) {
                // Let the copies already in flight land before the CTA exits (rank 0's
                // barriers also count rank 1's copies; rank 1 cannot observe its own, so it
                // leaves them a generous margin).
                if (leader) {
                    // stages before pos were last filled in this pass of the ring, the others in
                    // the pass before it (if there was one)
                    drain_barriers(nstages, [&](int s, uint64_t*& bar, uint32_t& parity) {
                        bar = &full[s];
                        parity = s < pos.stage ? pos.phase : pos.phase ^ 1u;
                        return s < pos.stage || wrapped;
                    });
                } else {
                    const uint64_t t0 = globaltimer_ns();
                    while (globaltimer_ns() - t0 < 100000ull) {
                    }
                }
            }
        }
    } else if (warp == kSchedWarp) {
        // ================= scheduler (one thread): decodes the cluster's tiles ahead of the other
        // roles.  In the TMA thread the decoding of a tile (~2.5 us: cold code, one thread) came
        // between two tiles' loads and left the MMAs waiting.
        if (elect_one()) {
            const int T = pre[p.num_groups];
            int q = 0;
            uint32_t qphase = 0;
            // cluster c takes tiles c, c + clusters, ... (both CTAs of the pair agree)
            const int tile_stride = static_cast<int>(gridDim.x >> 1);
            for (int t = static_cast<int>(blockIdx.x >> 1);; t += tile_stride) {
                // the next tile with work (gi < 0: no more)
                TileInfo ti = {};
                int gi = -1;
                while (t < T && !decode_tile<EPI>(p, pre, t, crank, gi, ti)) t += tile_stride;
                if (t >= T || *abort_flag) gi = -1;
                if (!mbar_wait(&tq_empty[q], qphase ^ 1u)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                tq[q].ti = ti;
                tq[q].gi = gi;
                mbar_arrive(&tq_full[q]);
                if (++q == kTileQueue) {
                    q = 0;
                    qphase ^= 1u;
                }
                if (gi < 0) break;
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (one thread of rank 0)
        if (elect_one()) {
            const uint32_t sbase = smem_u32(smem);
            RingPos pos = {0, 0u};
            uint32_t n = 0;  // active tiles processed
            int q = 0;
            uint32_t qphase = 0;
            for (;;) {
                if (!mbar_wait(&tq_full[q], qphase)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                const int gi = tq[q].gi;
                const TileInfo ti = tq[q].ti;
                mbar_arrive(&tq_empty[q]);
                if (++q == kTileQueue) {
                    q = 0;
                    qphase ^= 1u;
                }
                if (gi < 0 || *abort_flag) break;
                if (!leader) continue;  // rank 1 issues no MMAs; it only keeps its tile queue moving
                const uint32_t buf = n & 1u, use = n >> 1;
                ++n;
                if (!mbar_wait(&tempty[buf], (use & 1u) ^ 1u)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                tc_fence_after();
                if (ti.run_mma) {
                    const bool as = ti.a_split, bs = ti.b_split;
                    const uint32_t tacc = tmem_base + buf * kTmemCols, st16 = stage_stride >> 4;
                    uint32_t acc = 0u;
                    const bool ok = for_k_runs(ti, [&](int from, int to, bool at, bool bt) {
                        // instruction and operand descriptors for the layouts of this run
                        const bool a_mn = p.g[gi].a_mn || at, b_mn = p.g[gi].b_mn || bt;
                        const uint32_t idesc = make_idesc_16bit(kTileM, ti.n_mma, a_mn, b_mn, p.in_f16 != 0);
                        const uint64_t da = operand_desc(sbase, a_mn);
                        const uint64_t db = operand_desc(sbase + kTileABytes * (as ? 2u : 1u), b_mn);
                        const uint32_t a_lo = static_cast<uint32_t>(da), a_hi = static_cast<uint32_t>(da >> 32);
                        const uint32_t b_lo = static_cast<uint32_t>(db), b_hi = static_cast<uint32_t>(db >> 32);
                        const uint32_t sa = slice_step(a_mn), sb = slice_step(b_mn);
                        const int n = to - from;
                        if (as)
                            return bs ? issue_tile<true, true>(full, empty, nstages, st16, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc)
                                      : issue_tile<true, false>(full, empty, nstages, st16, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc);
                        return bs ? issue_tile<false, true>(full, empty, nstages, st16, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc)
                                  : issue_tile<false, false>(full, empty, nstages, st16, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc);
                    });
                    if (!ok) {
                        *abort_flag = 1;
                        atomicOr(p.err, kErrTimeout);
                    }
                }
                // completes once every MMA of this tile has finished (in both CTAs' barriers)
                umma_commit_pair_mc(&tfull[buf], 0x3);
            }
            if (leader) {
                umma_commit_pair(drain);
                (void)mbar_wait(drain, 0);
            }
        }
    } else {
        // ================= epilogue (warps 2..9): warp w reads TMEM lanes 32 (w % 4) ..,
        // warps 2..5 store the first half of the tile's column blocks, warps 6..9 the others
        const int eg = warp & 3;  // tensor-memory lane quarter this warp may access
        const int half = (warp - 2) >> 2;
        uint32_t n = 0;
        int q = 0;
        uint32_t qphase = 0;
        for (;;) {
            if (!__all_sync(0xffffffffu, mbar_wait(&tq_full[q], qphase))) {
                if (lane == 0) atomicOr(p.err, kErrTimeout);
                break;
            }
            // read from the queue as needed (registers are short here); the slot is given back
            // with the tile
            const TileInfo& ti = tq[q].ti;
            const int gi = tq[q].gi;
            if (gi < 0) break;
            const uint32_t buf = n & 1u, use = n >> 1;
            ++n;
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], use & 1u));
            if (!ok) {
                if (lane == 0) atomicOr(p.err, kErrTimeout);
                break;
            }
            __syncwarp();
            tc_fence_after();
            tile_epilogue<EPI, false>(tile_flags(p), p.g[gi], ti, tmem_base + buf * kTmemCols, ok, eg, half, lane, crank,
                          smem_u32(staging) + (warp - 2) * kStageBlocks * kStageBlockBytes);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (leader)
                    mbar_arrive(&tempty[buf]);
                else
                    mbar_arrive_cluster(mapa_shared(smem_u32(&tempty[buf]), 0));  // rank 0 issues the MMAs
                mbar_arrive(&tq_empty[q]);
            }
            if (++q == kTileQueue) {
                q = 0;
                qphase ^= 1u;
            }
        }
        if (elect_one()) bulk_wait0();  // this warp's TMA stores have completed
        __syncwarp();
    }

    // ---- teardown: the MMA thread has waited for all its MMAs (drain barrier); neither CTA
    // leaves (or frees tensor memory) while rank 0's MMAs could still read rank 1's shared
    // memory or write its tensor memory
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 2 * kTmemCols);
    }
}

// ------------------------------------------------------------------ host launcher
namespace {

cudaLaunchConfig_t pair_config(unsigned grid, cudaStream_t stream, cudaLaunchAttribute* at) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = kGemmSmemBytes;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <int EPI>
cudaError_t launch_epi(const GemmParams& p, int max_ctas, cudaStream_t stream) {
    static PerDevice clusters_that_fit;  // clusters of two that can be resident at once
    cudaLaunchAttribute at[1];
    int device = 0, max_clusters = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    e = clusters_that_fit.get<cudaError_t>(device, &max_clusters, [&](int* n) {
        const cudaError_t r = cudaFuncSetAttribute(k_gemm_split<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kGemmSmemBytes);
        if (r != cudaSuccess) return r;
        const cudaLaunchConfig_t cfg = pair_config(static_cast<unsigned>(max_ctas & ~1), stream, at);
        return cudaOccupancyMaxActiveClusters(n, k_gemm_split<EPI>, &cfg);
    });
    if (e != cudaSuccess) return e;
    if (max_clusters < 1) max_clusters = 1;
    int clusters = p.total_tiles;
    clusters = clusters < max_clusters ? clusters : max_clusters;
    clusters = clusters < max_ctas / 2 ? clusters : (max_ctas / 2 > 0 ? max_ctas / 2 : 1);
    const cudaLaunchConfig_t cfg = pair_config(static_cast<unsigned>(2 * clusters), stream, at);
    return cudaLaunchKernelEx(&cfg, k_gemm_split<EPI>, p);
}

}  // namespace

// Launches one persistent GEMM over the groups of `p` (p.total_tiles output tiles) on at
// most `max_ctas` CTAs (one per SM, in clusters of two).
cudaError_t launch_gemm(const GemmParams& p, int max_ctas, cudaStream_t stream) {
    if (p.total_tiles <= 0) return cudaSuccess;
    switch (p.epi) {
        case kEpiF32: return launch_epi<kEpiF32>(p, max_ctas, stream);
        case kEpiPoly: return launch_epi<kEpiPoly>(p, max_ctas, stream);
        case kEpiXSplit: return launch_epi<kEpiXSplit>(p, max_ctas, stream);
        default: return launch_epi<kEpiGram>(p, max_ctas, stream);
    }
}

}  // namespace isoloco
