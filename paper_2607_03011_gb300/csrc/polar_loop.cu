// polar_loop.cu -- iterations 1, 2, ... of the polar iteration as one persistent kernel.
//
// An iteration is a chain of GEMM phases per matrix (Gram, polynomial, update; on the Gram
// side W = A Z before the Gram) with the control step between the Gram and the polynomial.  As
// separate launches each phase pays its launch, its set-up, the latency of its first loads,
// its last partly filled wave and the drain of its stores: ~11 us for a phase of a few tiles,
// 45 us per iteration, however small the matrices.  Here every cluster (CTA pair) walks the same
// sequence of output tiles
//     for t = 1, 2, ...:  W | Gram | Gram-side Gram | polynomial | update
// taking every C-th one, and a tile only waits for the tiles of its own matrix that it reads:
//   arr[mat][kind] : arrivals of the tiles of one kind (two per tile, one from each CTA)
//   ctl[mat]       : (iterations decided << 4) | done << 3 | mode, written by the control step
// The last arrival in a matrix's Gram runs its control step.  Every wait points
// to tiles earlier in the sequence and all clusters are resident at once (cooperative launch),
// so the walk cannot lock up; every wait is bounded all the same.
//
// Roles per CTA as in gemm.cu: warp 10 walks the sequence (all lanes: the control words
// and states of up to 32 matrices at a time) and queues this cluster's tiles; warp 0 waits for
// a tile's operands and issues its TMA loads; warp 1 issues the MMAs; warps 2..9 run the
// epilogues.  The ring of shared memory is cut into 16 KB slots, one operand plane each, so that
// single-, two- and three-pass tiles can follow one another: a k-block takes two to four
// consecutive slots and one of kKb barrier pairs.
//
// Measured (GB300, whole outer step against the same kernels as a graph of launches): eight
// matrices of 64 to 256 (K = 2) 586 -> 399 us, ragged 515-wide set (K = 3) 2052 -> 1546, the 180M set
// (K = 8) 10.70 -> 10.12 ms; 2048- and 3072-wide sets, whose phases are hundreds of waves long,
// are level.  A scheduler warp of its own (the TMA thread used to walk: 5,800 cycles between two
// tiles' loads, the MMAs idle for most of them): 180M 10.23 -> 9.59 ms, 2048-wide 31.0 -> 28.6,
// 3072-wide 21.0 -> 19.8.  Log of a 180M iteration (two passes): polynomial and update tiles start
// every 17,000 to 18,000 cycles, their MMAs alone take 16,400.  A phase of a few tiles takes 7 to 13 us: operands' arrival seen ~0.4, decode and
// loads ~1, MMAs, epilogue ~3 (its code is cold every time: ~12 cycles per instruction),
// arrival ~1, control ~2.5.
#include "control.cuh"
#include "gemm_tile.cuh"
#include "per_device.h"
#include "polar_loop.h"

namespace isoloco {

namespace {

constexpr int kSlotBytes = kTileABytes;  // one operand plane of a k-block
constexpr int kSlots = kRingBytes / kSlotBytes;
constexpr int kKb = 8;  // k-blocks in flight at most (>= kSlots / 2)
constexpr int kLoopQueue = 6;
static_assert(kTileABytes == kTileBBytes && kSlots / 2 <= kKb, "slot ring");
static_assert(kKb * 4 <= 32, "slot counts of the k-blocks in flight packed in 4 bits each");

// One tile, decoded by the scheduler for the other roles.
struct LoopTile {
    TileInfo ti;
    TileFlags f;
    int group;    // index in LoopParams::groups
    int kind;     // LoopKind, or -1: no more tiles
    int t;        // iteration
    uint32_t want;        // arrivals at *dep that the tile's operands wait for (dep null: none)
    const uint32_t* dep;
    int first;    // the matrix's first tile here in this phase: its operands come from other SMs
};

// What the walk needs of a matrix's state.
struct TileState {
    float a, b, c, xscale, resid, yb, yc;
    int mode, step, x_hi_only;
};

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

// Waits until *p >= want (acquire), at most kWaitTimeoutNs and not once some CTA has timed out.
__device__ __forceinline__ bool wait_count(const uint32_t* p, uint32_t want, const uint32_t* err) {
    if (ld_acquire(p) >= want) return true;
    const uint64_t t0 = globaltimer_ns();
#pragma unroll 1
    for (uint32_t i = 1;; ++i) {
        if (ld_acquire(p) >= want) return true;
        if ((i & 63u) == 0 && (globaltimer_ns() - t0 > kWaitTimeoutNs || (ld_acquire(err) & kErrTimeout))) return false;
    }
}

__device__ __forceinline__ int next_slot(int s) { return s + 1 == kSlots ? 0 : s + 1; }

// Producer's view of the slot ring.
struct SlotRing {
    int slot = 0;          // next free slot
    int free_slots = kSlots;
    int head = 0, tail = 0;          // k-block barriers: next to use, oldest in flight
    uint32_t hphase = 0, tphase = 0; // their phases
    int inflight = 0;
    uint32_t hist = 0;     // slots of each k-block in flight, oldest in the low 4 bits
};

// As load_run (gemm_tile.cuh), each plane in its own slot.
template <bool AMN, bool BMN>
__device__ __forceinline__ bool loop_load(const CUtensorMap* a_hi, const CUtensorMap* b_hi, const TileInfo& ti, int from,
                                          int to, uint32_t sbase, uint64_t* full, uint64_t* empty, uint32_t fbar0,
                                          uint32_t crank, SlotRing& r) {
    const CUtensorMap *a_lo = a_hi + 1, *b_lo = b_hi + 1;
    const bool as = ti.a_split, bs = ti.b_split;
    const int need = 2 + (as ? 1 : 0) + (bs ? 1 : 0);
    const uint32_t pair_bytes = 2u * kSlotBytes * need;
    const int m0 = ti.m0, nb0 = ti.n0 + static_cast<int>(crank) * (ti.n_mma / 2), b = ti.b;
    const int k_end = to * BK;
#pragma unroll 1
    for (int k0 = from * BK; k0 < k_end; k0 += BK) {
        while (r.free_slots < need || r.inflight == kKb) {
            if (!mbar_wait(&empty[r.tail], r.tphase)) return false;
            r.free_slots += r.hist & 15u;
            r.hist >>= 4;
            --r.inflight;
            if (++r.tail == kKb) {
                r.tail = 0;
                r.tphase ^= 1u;
            }
        }
        if (crank == 0) mbar_arrive_expect_tx(&full[r.head], pair_bytes);
        const uint32_t fbar = fbar0 + 8u * r.head;
        auto next = [&]() {
            const uint32_t at = sbase + r.slot * kSlotBytes;
            r.slot = next_slot(r.slot);
            return at;
        };
        auto load_a = [&](const CUtensorMap* map, uint32_t at) {
            if (AMN) {
#pragma unroll
                for (int c = 0; c < BM / 64; ++c) tma_load_3d_pair(at + c * (BK * 128), map, fbar, m0 + 64 * c, k0, b);
            } else {
                tma_load_3d_pair(at, map, fbar, k0, m0, b);
            }
        };
        auto load_b = [&](const CUtensorMap* map, uint32_t at) {
            if (BMN) {
#pragma unroll
                for (int c = 0; c < kBRows / 64; ++c)
                    tma_load_3d_pair(at + c * (BK * 128), map, fbar, nb0 + 64 * c, k0, b);
            } else {
                tma_load_3d_pair(at, map, fbar, k0, nb0, b);
            }
        };
        load_a(a_hi, next());
        if (as) load_a(a_lo, next());
        load_b(b_hi, next());
        if (bs) load_b(b_lo, next());
        r.free_slots -= need;
        r.hist |= static_cast<uint32_t>(need) << (4 * r.inflight);
        ++r.inflight;
        if (++r.head == kKb) {
            r.head = 0;
            r.hphase ^= 1u;
        }
    }
    return true;
}

// MMA issuer's view of the slot ring.
struct SlotPos {
    int slot = 0, kb = 0;
    uint32_t phase = 0;
};

// As issue_tile (gemm_tile.cuh), with each plane in its own slot.
template <bool AS, bool BS>
__device__ __forceinline__ bool loop_issue(uint64_t* full, uint64_t* empty, int nkb, uint32_t tacc, uint32_t idesc,
                                           uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                           uint32_t step_a, uint32_t step_b, SlotPos& pos, uint32_t& acc) {
    constexpr uint32_t kSlot16 = kSlotBytes >> 4;
    bool ready = mbar_test(&full[pos.kb], pos.phase);
#pragma unroll 1
    for (int i = 0; i < nkb; ++i) {
        const int k = pos.kb;
        if (!ready && !mbar_wait(&full[k], pos.phase)) return false;
        tc_fence_after();
        const uint32_t ah = a_lo + pos.slot * kSlot16;
        pos.slot = next_slot(pos.slot);
        const uint32_t al = a_lo + pos.slot * kSlot16;
        if (AS) pos.slot = next_slot(pos.slot);
        const uint32_t bh = b_lo + pos.slot * kSlot16;
        pos.slot = next_slot(pos.slot);
        const uint32_t bl = b_lo + pos.slot * kSlot16;
        if (BS) pos.slot = next_slot(pos.slot);
        if (++pos.kb == kKb) {
            pos.kb = 0;
            pos.phase ^= 1u;
        }
#pragma unroll
        for (int ks = 0; ks < BK / 16; ++ks) {
            const uint32_t da = ks * step_a, db = ks * step_b;
            umma_16bit_pair(tacc, ah + da, a_hi, bh + db, b_hi, idesc, acc);
            if (BS) umma_16bit_pair(tacc, ah + da, a_hi, bl + db, b_hi, idesc, 1u);
            if (AS) umma_16bit_pair(tacc, al + da, a_hi, bh + db, b_hi, idesc, 1u);
            acc = 1u;
            if (ks == BK / 16 - 2) ready = mbar_test(&full[pos.kb], pos.phase);
        }
        umma_commit_pair_mc(&empty[k], 0x3);
    }
    return true;
}

__device__ __forceinline__ void load_state(const MatState* s, TileState& o) {
    o.a = __ldcg(&s->a);
    o.b = __ldcg(&s->b);
    o.c = __ldcg(&s->c);
    o.xscale = __ldcg(&s->xscale);
    o.resid = __ldcg(&s->resid);
    o.yb = __ldcg(&s->yb);
    o.yc = __ldcg(&s->yc);
    o.mode = __ldcg(&s->mode);
    o.step = __ldcg(&s->step);
    o.x_hi_only = __ldcg(&s->x_hi_only);
}

__device__ __forceinline__ float shfl_f(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ int shfl_i(int v, int src) { return __shfl_sync(0xffffffffu, v, src); }

}  // namespace

// The matrix (of the phase's groups, in their order) at position i of a phase's walk.
__device__ __forceinline__ int walk_matrix(const LoopPhase& L, int i) {
    const int side = L.count - L.regular;
    if (i >= L.side_at) {
        if (i < L.side_at + side) return L.regular + i - L.side_at;
        i -= side;
    }
    if (i < 2 * L.skip) i += i < L.skip ? L.skip : -L.skip;
    return L.falling ? L.regular - 1 - i : i;
}

// The cluster size is part of the kernel, not only of its launch: a profiler that launches a
// cooperative kernel in its own way drops the launch's cluster attribute (seen with ncu 2025.3), and
// pair instructions outside a cluster of two fault.
template <int NG>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1) k_polar_loop(const __grid_constant__ LoopParams<NG> p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align1024(smem_raw);
    uint8_t* staging = smem + kRingBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kRingBytes + kEpiStagingBytes);  // [kKb]
    uint64_t* empty = full + kKb;
    uint64_t* tfull = empty + kKb;        // [2]
    uint64_t* tempty = tfull + 2;         // [2]
    uint64_t* drain = tempty + 2;
    uint64_t* tq_full = drain + 1;        // [kLoopQueue]
    uint64_t* tq_empty = tq_full + kLoopQueue;
    LoopTile* tq = reinterpret_cast<LoopTile*>(tq_empty + kLoopQueue);  // [kLoopQueue]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tq + kLoopQueue);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    unsigned* epi_done = reinterpret_cast<unsigned*>(tmem_slot + 2);  // [4] epilogue warps through with tile n (n mod 4)
    static_assert(8 * (2 * kKb + 5 + 2 * kLoopQueue) + kLoopQueue * sizeof(LoopTile) + 24 <= kLoopTailBytes,
                  "shared memory behind the staging blocks");

    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const uint32_t crank = cluster_ctarank();
    const bool leader = crank == 0;
    const int C = static_cast<int>(gridDim.x >> 1), cluster = static_cast<int>(blockIdx.x >> 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kKb; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], kEpiWarps * 2);
        }
        mbar_init(drain, 1);
        for (int q = 0; q < kLoopQueue; ++q) {
            mbar_init(&tq_full[q], 1);
            mbar_init(&tq_empty[q], kTileReaders);
        }
        *abort_flag = 0;
        for (int i = 0; i < 4; ++i) epi_done[i] = 0u;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 2 * kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ================= TMA producer (one thread)
        if (elect_one()) {
            const uint32_t sbase = smem_u32(smem);
            const uint32_t fbar0 = mapa_shared(smem_u32(full), 0);
            SlotRing ring;
            int q = 0;
            uint32_t qphase = 0;
            for (;;) {
                // (a wait for another cluster's decisions ends in the scheduler, which then says so
                // here: longer than its limit)
                if (!mbar_wait(&tq_full[q], qphase, 3 * kWaitTimeoutNs)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                const LoopTile& lt = tq[q];
                if (lt.kind < 0) break;
                const TileInfo& ti = lt.ti;
                if (!*abort_flag) {  // after a timeout the queue only drains
                    bool good = true;
                    if (lt.first) {
                        if (lt.dep) good = wait_count(lt.dep, lt.want, p.err);
                        fence_proxy_async_all();  // operands written by other SMs, read by TMA
                    }
                    if (good && ti.run_mma) {
                        const GemmGroup& g = p.groups[lt.group].g;
                        good = for_k_runs(ti, [&](int from, int to, bool at, bool bt) {
                            const CUtensorMap *a = map_a(g, at), *b = map_b(g, bt);
                            if (g.a_mn || at)
                                return g.b_mn || bt ? loop_load<true, true>(a, b, ti, from, to, sbase, full, empty, fbar0, crank, ring)
                                                    : loop_load<true, false>(a, b, ti, from, to, sbase, full, empty, fbar0, crank, ring);
                            return g.b_mn || bt ? loop_load<false, true>(a, b, ti, from, to, sbase, full, empty, fbar0, crank, ring)
                                                : loop_load<false, false>(a, b, ti, from, to, sbase, full, empty, fbar0, crank, ring);
                        });
                    }
                    if (!good) {
                        *abort_flag = 1;
                        atomicOr(p.err, kErrTimeout);
                    }
                }
                mbar_arrive(&tq_empty[q]);
                if (++q == kLoopQueue) {
                    q = 0;
                    qphase ^= 1u;
                }
            }
            if (*abort_flag) {
                // let the copies in flight land before the CTA exits (rank 0's barriers also
                // count rank 1's copies; rank 1 cannot observe its own, so it leaves a margin)
                if (leader) {
                    drain_barriers(ring.inflight, [&](int i, uint64_t*& bar, uint32_t& parity) {
                        const int k = ring.tail + i;
                        bar = &full[k < kKb ? k : k - kKb];
                        parity = k < kKb ? ring.tphase : ring.tphase ^ 1u;
                        return true;
                    });
                } else {
                    const uint64_t t0 = globaltimer_ns();
                    while (globaltimer_ns() - t0 < 100000ull) {
                    }
                }
            }
        }
    } else if (warp == kSchedWarp) {
        // ================= scheduler: the walk
        int q = 0;
        uint32_t qphase = 0;
        int off = 0;      // tiles handed out so far, modulo C
        bool ok = true;   // no wait has run out (warp-uniform at the checks)
        uint64_t stamp = p.prof ? globaltimer_ns() : 0;
        int stamp_ph = -1;
        for (int t = 1; ok && t <= p.max_t; ++t) {
            unsigned any = 0;
            for (int ph = 0; ok && ph < kLoopPhases; ++ph) {
                const LoopPhase& L = p.phases[((t & 1) ^ 1) * kLoopPhases + ph];
                const int count = L.count, kind = L.kind;
                if (count == 0) continue;
                const bool stepping = kind == kLoopPoly || kind == kLoopUpdate;
                // arrivals the operands of this kind wait for: W and the (row x column) Gram read
                // the last iteration's update, the Gram-side Gram W, the update the polynomial
                const int dep = kind == kLoopUpdate ? kArrPoly : kind == kLoopGramGs ? kArrW : kArrUpdate;
                const uint32_t dep_iters = (kind == kLoopUpdate || kind == kLoopGramGs) ? t : t - 1;
                const int passes = p.prof ? 2 : 1;  // profiling: first wait for the whole last phase
                for (int pass = 0; ok && pass < passes; ++pass) {
                    const bool only_wait = pass + 1 < passes;
                    int n = 0;  // matrices taken at a time: the next ones already decided, up to 32
                    // (waiting for 32 at a time idled every cluster 3-7 % of an iteration)
                    for (int e0 = 0; ok && e0 < count; e0 += n) {
                        bool valid = e0 + lane < count;
                        // this lane's matrix of the phase
                        int grp = L.first, b = valid ? walk_matrix(L, e0 + lane) : 0;
                        if (valid)
                            while (b >= p.groups[grp].g.batch) b -= p.groups[grp++].g.batch;
                        const int mat = valid ? p.groups[grp].g.mat_base + b : 0;
                        // the matrix's decisions up to the one this phase follows
                        const uint32_t need = stepping ? t + 1 : t;
                        uint32_t w = 0;
                        {
                            bool have = !valid;
                            uint64_t t0 = 0;
#pragma unroll 1
                            for (uint32_t i = 0;; ++i) {
                                if (!have) {
                                    w = ld_acquire(&p.ctl[mat]);
                                    have = (w >> 4) >= need || (w & 8u);
                                }
                                const unsigned wait = ~__ballot_sync(0xffffffffu, have);
                                n = wait ? __ffs(wait) - 1 : 32;
                                if (n > 0) break;
                                if ((i & 63u) == 63u) {
                                    if (!t0) t0 = globaltimer_ns();
                                    const bool out = *abort_flag || globaltimer_ns() - t0 > kWaitTimeoutNs ||
                                                     (ld_acquire(p.err) & kErrTimeout);
                                    if (__any_sync(0xffffffffu, out)) {
                                        ok = false;
                                        break;
                                    }
                                }
                            }
                        }
                        if (!ok) break;
                        valid = valid && lane < n;
                        // active: its Gram until it is done; its step in the iterations it decided
                        // one for (an undone matrix always steps; the last step is the one it
                        // finished in, unless it stopped without one)
                        const uint32_t decided = w >> 4;
                        const bool done = (w & 8u) != 0;
                        bool active = valid;
                        if (stepping)
                            active = active && (decided > need || (decided == need && (w & 7u) != 0)) &&
                                     !(done && decided < need);
                        else
                            active = active && (!done || decided > need);
                        if (!stepping) any |= __ballot_sync(0xffffffffu, active);
                        const int tiles = active ? p.groups[grp].tiles : 0;
                        int pre = tiles;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int x = __shfl_up_sync(0xffffffffu, pre, o);
                            if (lane >= o) pre += x;
                        }
                        const int total = __shfl_sync(0xffffffffu, pre, 31);
                        pre -= tiles;  // exclusive
                        const uint32_t want = dep_iters * static_cast<uint32_t>(p.groups[grp].dep_tiles) * 2u;
                        const uint32_t* cnt = p.arr + static_cast<int64_t>(mat) * kArrKinds + dep;
                        if (only_wait) {
                            bool good = true;
                            if (active && kind != kLoopPoly) good = wait_count(cnt, want, p.err);
                            ok = __all_sync(0xffffffffu, good);
                            continue;
                        }
                        int j0 = cluster - (off + pre) % C;
                        if (j0 < 0) j0 += C;
                        const bool has = j0 < tiles;
                        off = (off + total) % C;
                        // this cluster's matrices: their states, and whether their operands are there
                        // (if not, the TMA thread waits for them).  A state is that of the decision this
                        // phase follows: the next one waits for this cluster's tiles
                        TileState st = {};
                        bool there = true;
                        if (has) {
                            load_state(p.state + mat, st);
                            if (kind != kLoopPoly) there = ld_acquire(cnt) >= want;
                        }
                        unsigned m = __ballot_sync(0xffffffffu, has);
                        while (m && ok) {
                            const int src = __ffs(m) - 1;
                            m &= m - 1;
                            MatState ms;
                            ms.a = shfl_f(st.a, src);
                            ms.b = shfl_f(st.b, src);
                            ms.c = shfl_f(st.c, src);
                            ms.xscale = shfl_f(st.xscale, src);
                            ms.resid = shfl_f(st.resid, src);
                            ms.yb = shfl_f(st.yb, src);
                            ms.yc = shfl_f(st.yc, src);
                            ms.mode = shfl_i(st.mode, src);
                            ms.step = shfl_i(st.step, src);
                            ms.x_hi_only = shfl_i(st.x_hi_only, src);
                            const int mmat = shfl_i(mat, src), mgrp = shfl_i(grp, src), mb = shfl_i(b, src);
                            const int mt = shfl_i(tiles, src), js = shfl_i(j0, src);
                            const bool ready = shfl_i(there, src) != 0;
                            const uint32_t mwant = __shfl_sync(0xffffffffu, want, src);
                            bool good = true;
                            if (elect_one()) {
                                const GemmGroup& g = p.groups[mgrp].g;
                                const TileFlags f = L.f;
                                for (int j = js; j < mt; j += C) {
                                    if (!mbar_wait(&tq_empty[q], qphase ^ 1u, 2 * kWaitTimeoutNs) || *abort_flag) {
                                        good = false;
                                        break;
                                    }
                                    LoopTile& lt = tq[q];
                                    TileInfo ti;
                                    if (kind == kLoopPoly)
                                        setup_tile<kEpiPoly>(f, g, &ms, mb, j, 0, crank, ti);
                                    else if (kind == kLoopGram || kind == kLoopGramGs)
                                        setup_tile<kEpiGram>(f, g, &ms, mb, j, 0, crank, ti);
                                    else
                                        setup_tile<kEpiXSplit>(f, g, &ms, mb, j, 0, crank, ti);
                                    lt.ti = ti;
                                    lt.f = f;
                                    lt.group = mgrp;
                                    lt.kind = kind;
                                    lt.t = t;
                                    lt.first = j == js;
                                    lt.want = mwant;
                                    lt.dep = (j == js && !ready) ? p.arr + static_cast<int64_t>(mmat) * kArrKinds + dep : nullptr;
                                    mbar_arrive(&tq_full[q]);
                                    if (++q == kLoopQueue) {
                                        q = 0;
                                        qphase ^= 1u;
                                    }
                                }
                            }
                            ok = __all_sync(0xffffffffu, good);
                        }
                    }
                    if (only_wait && ok && blockIdx.x == 0 && lane == 0) {
                        // profiling: the last phase ends here
                        const uint64_t now = globaltimer_ns();
                        if (stamp_ph >= 0) p.prof[stamp_ph] += now - stamp;
                        stamp = now;
                        stamp_ph = kind;
                    }
                }
            }
            if (!any) break;
        }
        if (p.prof && ok && blockIdx.x == 0 && lane == 0 && stamp_ph >= 0) p.prof[stamp_ph] += globaltimer_ns() - stamp;
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicOr(p.err, kErrTimeout);
        }
        // no more tiles
        __syncwarp();
        if (elect_one()) {
            if (mbar_wait(&tq_empty[q], qphase ^ 1u, 2 * kWaitTimeoutNs)) {
                tq[q].kind = -1;
                mbar_arrive(&tq_full[q]);
            } else {
                *abort_flag = 1;
                atomicOr(p.err, kErrTimeout);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issuer (one thread of rank 0)
        if (elect_one()) {
            const uint32_t sbase = smem_u32(smem);
            SlotPos pos;
            uint32_t n = 0;
            int q = 0;
            uint32_t qphase = 0;
            for (;;) {
                if (!mbar_wait(&tq_full[q], qphase, 3 * kWaitTimeoutNs)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                const LoopTile& lt = tq[q];
                const int kind = lt.kind;
                const TileInfo ti = lt.ti;
                const int f16 = lt.f.in_f16, grp = lt.group;
                mbar_arrive(&tq_empty[q]);
                if (++q == kLoopQueue) {
                    q = 0;
                    qphase ^= 1u;
                }
                if (kind < 0 || *abort_flag) break;
                if (!leader) continue;
                const uint32_t buf = n & 1u, use = n >> 1;
                ++n;
                if (!mbar_wait(&tempty[buf], (use & 1u) ^ 1u, 2 * kWaitTimeoutNs)) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
                tc_fence_after();
                if (ti.run_mma) {
                    const bool as = ti.a_split, bs = ti.b_split;
                    const uint32_t tacc = tmem_base + buf * kTmemCols;
                    uint32_t acc = 0u;
                    const bool ok = for_k_runs(ti, [&](int from, int to, bool at, bool bt) {
                        const bool a_mn = p.groups[grp].g.a_mn || at, b_mn = p.groups[grp].g.b_mn || bt;
                        const uint32_t idesc = make_idesc_16bit(kTileM, ti.n_mma, a_mn, b_mn, f16 != 0);
                        const uint64_t da = operand_desc(sbase, a_mn), db = operand_desc(sbase, b_mn);
                        const uint32_t a_lo = static_cast<uint32_t>(da), a_hi = static_cast<uint32_t>(da >> 32);
                        const uint32_t b_lo = static_cast<uint32_t>(db), b_hi = static_cast<uint32_t>(db >> 32);
                        const uint32_t sa = slice_step(a_mn), sb = slice_step(b_mn);
                        const int n = to - from;
                        if (as)
                            return bs ? loop_issue<true, true>(full, empty, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc)
                                      : loop_issue<true, false>(full, empty, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc);
                        return bs ? loop_issue<false, true>(full, empty, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc)
                                  : loop_issue<false, false>(full, empty, n, tacc, idesc, a_lo, a_hi, b_lo, b_hi, sa, sb, pos, acc);
                    });
                    if (!ok) {
                        *abort_flag = 1;
                        atomicOr(p.err, kErrTimeout);
                    }
                }
                umma_commit_pair_mc(&tfull[buf], 0x3);
            }
            if (leader) {
                umma_commit_pair(drain);
                (void)mbar_wait(drain, 0);
            }
        }
    } else {
        // ================= epilogue (warps 2..9)
        const int eg = warp & 3;
        const int half = (warp - 2) >> 2;
        const uint32_t stg = smem_u32(staging) + (warp - 2) * kStageBlocks * kStageBlockBytes;
        uint32_t n = 0;
        int q = 0;
        uint32_t qphase = 0;
        for (;;) {
            const bool got = __all_sync(0xffffffffu, mbar_wait(&tq_full[q], qphase, 3 * kWaitTimeoutNs));
            if (!got) {
                if (lane == 0) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                }
                break;
            }
            const LoopTile& lt = tq[q];
            const int kind = lt.kind;
            if (kind < 0) break;
            // (read from the queue as needed; the slot is given back with the tile)
            const TileInfo& ti = lt.ti;
            const TileFlags& f = lt.f;
            const LoopGroup& lg = p.groups[lt.group];
            const GemmGroup& g = lg.g;
            const uint32_t buf = n & 1u, use = n >> 1;
            unsigned* through = epi_done + (n & 3u);
            ++n;
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&tfull[buf], use & 1u, 2 * kWaitTimeoutNs));
            if (!ok) {
                if (lane == 0) {
                    *abort_flag = 1;
                    atomicOr(p.err, kErrTimeout);
                }
                break;
            }
            tc_fence_after();
            const uint32_t tacc = tmem_base + buf * kTmemCols;
            if (kind == kLoopPoly)
                tile_epilogue<kEpiPoly, true>(f, g, ti, tacc, ok, eg, half, lane, crank, stg);
            else if (kind == kLoopGram || kind == kLoopGramGs)
                tile_epilogue<kEpiGram, true>(f, g, ti, tacc, ok, eg, half, lane, crank, stg);
            else
                tile_epilogue<kEpiXSplit, true>(f, g, ti, tacc, ok, eg, half, lane, crank, stg);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (leader)
                    mbar_arrive(&tempty[buf]);
                else
                    mbar_arrive_cluster(mapa_shared(smem_u32(&tempty[buf]), 0));
            }
            // arrival: the last of the CTA's epilogue warps through with the tile publishes its
            // stores (one fence and one count per tile and CTA).  A warp
            // can be at most two tiles ahead of another here (the accumulator buffers), so four
            // counters keep the tiles apart.
            if (elect_one()) bulk_wait0();
            const int t = lt.t, mat = ti.mat, b = ti.b;
            __syncwarp();
            if (lane == 0) mbar_arrive(&tq_empty[q]);
            if (++q == kLoopQueue) {
                q = 0;
                qphase ^= 1u;
            }
            uint32_t last = 0, old = 0;
            const int arr = kind == kLoopW ? kArrW : kind == kLoopPoly ? kArrPoly : kind == kLoopUpdate ? kArrUpdate : kArrGram;
            if (lane == 0) {
                __threadfence_block();
                last = (atomicAdd(through, 1u) & (kEpiWarps - 1)) == kEpiWarps - 1;
                if (last) {
                    __threadfence();
                    old = atomicAdd(p.arr + static_cast<int64_t>(mat) * kArrKinds + arr, 1u);
                }
            }
            if (arr != kArrGram) continue;
            last = __shfl_sync(0xffffffffu, last, 0);
            if (!last) continue;
            old = __shfl_sync(0xffffffffu, old, 0);
            if (old + 1u == static_cast<uint32_t>(t) * lg.tiles * 2u) {
                // the matrix's Gram is complete: its control step
                __threadfence();
                ControlMat cm = lg.cm;
                cm.gpart_slot += static_cast<int64_t>(b) * cm.n_gtiles;
                const uint32_t w = control_matrix(cm, p.state + mat, p.fin_part, t, p.max_iter, p.tol, p.err, lane,
                                                  p.fast_steps, p.gram_one, p.upd_one, p.gs_on);
                if (lane == 0) {
                    __threadfence();
                    st_relaxed(&p.ctl[mat], w);
                }
                __syncwarp();
            }
        }
    }

    // ---- teardown, as in k_gemm_split
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
template <int NG>
cudaError_t launch_polar_loop(const LoopParams<NG>& p, int clusters, cudaStream_t stream) {
    static PerDevice clusters_that_fit;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = kLoopSmemBytes;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    int device = 0, max_clusters = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    e = clusters_that_fit.get<cudaError_t>(device, &max_clusters, [&](int* n) {
        const cudaError_t r = cudaFuncSetAttribute(k_polar_loop<NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLoopSmemBytes);
        return r != cudaSuccess ? r : cudaOccupancyMaxActiveClusters(n, k_polar_loop<NG>, &cfg);
    });
    if (e != cudaSuccess) return e;
    if (max_clusters < 1) max_clusters = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(2 * (clusters < max_clusters ? clusters : max_clusters)));
    return cudaLaunchKernelEx(&cfg, k_polar_loop<NG>, p);
}

template cudaError_t launch_polar_loop<kLoopGroupsSmall>(const LoopParams<kLoopGroupsSmall>&, int, cudaStream_t);
template cudaError_t launch_polar_loop<kLoopGroups>(const LoopParams<kLoopGroups>&, int, cudaStream_t);

}  // namespace isoloco
