// gemm_tile.cuh -- one output tile of the split-precision GEMM: its decoding, operand loads,
// MMA issue and epilogue, shared by the batched GEMM (gemm.cu) and the polar loop
// (polar_loop.cu).
#pragma once
#include "common.cuh"
#include "types.h"

namespace isoloco {

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Descriptor of an operand plane at shared address `plane` (first 16-deep K slice) in its
// layout, and the start-address step (16-byte units) to the next slice.
__device__ __forceinline__ uint64_t operand_desc(uint32_t plane, bool mn) {
    // 128B swizzle, MN-major: 64-element MN chunks are BK * 128 bytes apart (LBO), 8-row K
    // groups 1024 bytes (SBO).  K-major: rows of BK 16-bit values (128 bytes), 8-row groups
    // 1024 bytes apart (SBO).
    return mn ? make_sdesc(plane, BK * 128, 1024, 2) : make_sdesc(plane, 16, 8 * BK * 2, 2);
}
__device__ __forceinline__ uint32_t slice_step(bool mn) { return mn ? (2048 >> 4) : (32 >> 4); }
static_assert(BK * 2 == 128, "K-major rows fill one 128-byte swizzle row");

// Symmetric outputs: the t-th of the tiles that touch the upper triangle (col >= row),
// in row-major order of tiles.
__device__ __forceinline__ void sym_tile(int t, int tiles_m, int tiles_n, int& tm, int& tn) {
    for (tm = 0; tm < tiles_m; ++tm) {
        const int lo = sym_first_tile_n(tm);
        const int cnt = tiles_n - lo;
        if (t < cnt) {
            tn = lo + t;
            return;
        }
        t -= cnt;
    }
    tm = tiles_m - 1;
    tn = tiles_n - 1;
}

// Everything a role needs to know about one output tile of a group.
struct TileInfo {
    int b, tile, split, m0, n0, mat, kb_begin, kb_end;
    int n_mma;       // columns the MMAs compute: half a tile for up to 128 (whole 64-wide boxes of B per CTA)
    int a_sw, b_sw;  // k-blocks below these come from the transposed tile (GemmGroup::a_tri, b_tri)
    bool run_mma, a_split, b_split;
    bool horner;     // kEpiPoly: P = acc + a I (the MMA computed G Y); else P = a I + b G + c acc
    bool hi_only;    // write the hi plane only (a single-pass Gram's G; an update's X whose lo
                     // plane no later step reads)
    bool trace;      // the output is a matrix's final Q: also sum Q o Delta (GemmGroup::d_hi)
    float ca, cb, cc, xs;
    float yb, yc;    // kEpiGram with p.gram_y: Y = yb I + yc G for the next quintic step
};

// Fills `ti` for tile `tile` (K split `split`) of matrix b of group g and the CTA of rank
// `crank` in its pair; st: the matrix's state (only read with a gate).
template <int EPI>
__device__ __forceinline__ void setup_tile(const TileFlags& f, const GemmGroup& g, const MatState* st, int b, int tile,
                                           int split, uint32_t crank, TileInfo& ti) {
    ti.tile = tile;
    ti.split = split;
    ti.b = b;
    int tm, tn;
    if (g.sym) {
        sym_tile(tile, g.tiles_m, g.tiles_n, tm, tn);
    } else {
        tm = tile / g.tiles_n;
        tn = tile % g.tiles_n;
    }
    ti.m0 = tm * kTileM + static_cast<int>(crank) * BM;  // this CTA's rows of the tile
    ti.n0 = tn * BN;
    ti.mat = g.mat_base + b;
    ti.run_mma = true;
    ti.a_split = g.a_split != 0;
    ti.b_split = g.b_split != 0;
    ti.ca = 0.f, ti.cb = 0.f, ti.cc = 1.f, ti.xs = 1.f, ti.yb = 0.f, ti.yc = 0.f;
    ti.horner = false;
    ti.hi_only = false;
    // the final Q of a matrix: the polish update, or an ungated launch (the Gram side's
    // Q = Delta Z, which writes only matrices that have a Q)
    ti.trace = EPI == kEpiXSplit && g.d_hi != nullptr && f.gate == kGateNone;
    if (f.gate != kGateNone) {
        if (f.gate == kGateActive) {
            if (f.gram_y) {  // coefficients of the quintic step this Gram may lead to
                ti.yb = st->yb;
                ti.yc = st->yc;
            }
        } else {
            if (EPI == kEpiPoly && st->mode == 2) ti.run_mma = false;  // cubic polish: no G^2
            ti.horner = (EPI == kEpiPoly && f.poly_horner && st->mode == 1);
            if (f.split_on_polish && st->mode == 2) ti.a_split = ti.b_split = true;  // final step: 3 passes
            ti.trace = EPI == kEpiXSplit && g.d_hi != nullptr && f.gate == kGateStep && st->mode == 2;
        }
        // precision schedule: single-pass steps.  A Gram only after iteration 0's and only
        // while the last residual is large (>= kOnePassGramResid): a Gram whose test can pass
        // feeds the final polish, which nothing corrects afterwards, so it keeps its passes.
        const int k = (EPI == kEpiGram) ? st->step : st->step - 1;
        if (k >= g.one_from && k < g.one_to &&
            ((EPI == kEpiGram) ? (st->step > 0 && st->resid >= kOnePassGramResid) : st->mode == 1)) {
            ti.a_split = ti.b_split = false;
            // a single-pass Gram never feeds the polish and its polynomial reads G's hi only
            if (EPI == kEpiGram) ti.hi_only = true;
        }
        if (EPI == kEpiXSplit && f.gate == kGateStep && st->mode == 1 && st->x_hi_only) ti.hi_only = true;
        ti.ca = st->a;
        ti.cb = st->b;
        ti.cc = st->c;
        ti.xs = f.unit_scale ? 1.f : st->xscale;
    }
    const int total_kb = (g.K + BK - 1) / BK;
    ti.kb_begin = split * g.kblocks_per_split;
    ti.kb_end = min(total_kb, ti.kb_begin + g.kblocks_per_split);
    if (ti.kb_begin >= ti.kb_end) ti.run_mma = false;
    // (a step on 64-wide matrices 338 -> 330 us, one of odd widths 2.97 -> 2.93 ms; full tiles level)
    ti.n_mma = g.N - ti.n0 > BN / 2 ? BN : BN / 2;
    ti.a_sw = g.a_tri ? tm * (kTileM / BK) : 0;
    ti.b_sw = g.b_tri ? tn * (BN / BK) : 0;
}

// (Symmetric G, Y, P with only the tiles on and above the diagonal stored: mirroring each tile
// cost the Gram's epilogue, which bounds its phase, half of its 20,000 cycles per tile, and 40 %
// of the planes' writes.  A step on 12 layers of 1024 x 2816, 8 replicas: 10.01 -> 9.71 ms.)
// Calls f(from, to, a transposed, b transposed) for the runs of a tile's k-blocks that read both
// operands in one layout; stops when f returns false.
template <class F>
__device__ __forceinline__ bool for_k_runs(const TileInfo& ti, F f) {
    const int end = ti.kb_end;
    for (int k = ti.kb_begin; k < end;) {
        const bool at = k < ti.a_sw, bt = k < ti.b_sw;
        int to = end;
        if (at) to = min(to, ti.a_sw);
        if (bt) to = min(to, ti.b_sw);
        if (!f(k, to, at, bt)) return false;
        k = to;
    }
    return true;
}

// Staging of an epilogue warp: blocks of 32 x 32 16-bit values with 64-byte rows whose 16-byte
// chunks are swizzled (chunk XOR (row / 2) mod 4), the layout a TMA store with
// CU_TENSOR_MAP_SWIZZLE_64B reads.  Addresses are shared addresses.

// This lane's row: its chunk q is at row_addr ^ (q << 4).
__device__ __forceinline__ uint32_t stage_row_addr(uint32_t blk, int lane) {
    return blk + lane * 64 + (((lane >> 1) & 3) << 4);
}
__device__ __forceinline__ void stage_row(const uint32_t (&w)[16], uint32_t row_addr) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        st_shared4(row_addr ^ (q << 4), w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// The transpose of the warp's 32 x 32 block (lane = row, w = the lane's 32 values packed in
// pairs) into block `blk`: T(r, c) = value of lane c at column r.  For rows 2i and
// 2i + 1, even lanes c form (own, partner) column 2i and odd lanes (partner, own) column
// 2i + 1 from the packed pair w[i] and the partner lane's, one 32-bit store each.
__device__ __forceinline__ void stage_transposed(const uint32_t (&w)[16], uint32_t blk, int lane) {
    const uint32_t sel = (lane & 1) ? 0x3276u : 0x5410u;
    const int c = lane & ~1;
    const uint32_t at = blk + (lane & 1) * 64 + (c & 7) * 2, chunk = (c >> 3) << 4;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const uint32_t other = __shfl_xor_sync(0xffffffffu, w[i], 1);
        st_shared(at + (chunk ^ ((i & 3) << 4)) + i * 128, __byte_perm(w[i], other, sel));
    }
}

// One warp writes a 32 x 32 block of a diagonal tile (16-bit values, lane = row, w = the lane's 32
// values packed in pairs) to staging and stores it with TMA at (col0, row_base, b).  The block
// on the diagonal (diag) is made symmetric (each row takes what lies left of the diagonal from
// the transpose); another is also stored transposed at (row_base, col0, b).  `stg` is the
// warp's two blocks, taken once the store before has read them.
__device__ __forceinline__ void stage_store_block(const uint32_t (&w)[16], const CUtensorMap* map, uint32_t stg,
                                                  bool diag, int lane, int col0, int row_base, int b) {
    static_assert(kStageBlocks == 2, "a block and its transpose");
    const uint32_t sm = stg + kStageBlockBytes;  // the transpose
    if (elect_one()) bulk_wait_read0();
    __syncwarp();
    stage_transposed(w, sm, lane);
    const uint32_t row = stage_row_addr(stg, lane);
    if (diag) {
        __syncwarp();
        const uint32_t trow = stage_row_addr(sm, lane);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 t = ld_shared4(trow ^ (q << 4));
            const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
            uint32_t x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = 4 * q + k;  // columns 2i and 2i + 1 of row `lane`
                x[k] = __byte_perm(tw[k], w[i], 2 * i >= lane ? 0x7654u : 2 * i + 1 >= lane ? 0x7610u : 0x3210u);
            }
            st_shared4(row ^ (q << 4), x[0], x[1], x[2], x[3]);
        }
    } else {
        stage_row(w, row);
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (elect_one()) {
        tma_store_3d(map, stg, col0, row_base, b);
        if (!diag) tma_store_3d(map, sm, row_base, col0, b);
        bulk_commit();
    }
}

// A row's share of tr(Q^T Delta) in 32 columns from c0, added to s: Q in fp32 as stored (before
// its split into planes), Delta from its bf16 hi/lo planes.
__device__ __forceinline__ float trace_share(const GemmGroup& g, const TileInfo& ti, const float (&v)[32], int row,
                                             int c0, float s) {
    const int64_t doff = ti.b * g.bf_batch_stride + static_cast<int64_t>(row) * g.ld_bf + c0;
    const uint16_t* dh = reinterpret_cast<const uint16_t*>(g.d_hi) + doff;
    const uint16_t* dl = reinterpret_cast<const uint16_t*>(g.d_lo) + doff;
    if (g.N - c0 >= 32) {
        const uint4* h4 = reinterpret_cast<const uint4*>(dh);
        const uint4* l4 = reinterpret_cast<const uint4*>(dl);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 hh = h4[q], ll = l4[q];
            const uint32_t hw[4] = {hh.x, hh.y, hh.z, hh.w};
            const uint32_t lw[4] = {ll.x, ll.y, ll.z, ll.w};
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const float d0 = __uint_as_float(hw[w] << 16) + __uint_as_float(lw[w] << 16);
                const float d1 = __uint_as_float(hw[w] & 0xFFFF0000u) + __uint_as_float(lw[w] & 0xFFFF0000u);
                s = fmaf(v[8 * q + 2 * w], d0, s);
                s = fmaf(v[8 * q + 2 * w + 1], d1, s);
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < g.N - c0)
                s = fmaf(v[j], __uint_as_float(static_cast<uint32_t>(dh[j]) << 16) +
                                   __uint_as_float(static_cast<uint32_t>(dl[j]) << 16), s);
    }
    return s;
}

// Fixed-order warp reduction into this warp's slot of the tile (every slot of every tile of the
// matrix is written by the launch that writes its Q).
__device__ __forceinline__ void trace_store(const GemmGroup& g, const TileInfo& ti, float s, int eg, int half, int lane,
                                            uint32_t crank) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0)
        g.tf_part[(static_cast<int64_t>(ti.b) * (g.tiles_m * g.tiles_n) + ti.tile) * kPartSlots +
                  static_cast<int>(crank) * kEpiWarps + half * 4 + eg] = static_cast<double>(s);
}

// The 16-bit words of one plane of 32 values: kind 0 hi, 1 lo, 2 Y = yb I + yc G (hi plane only,
// it is the single operand of G Y), its diagonal at column d if diag.
__device__ __forceinline__ void plane_words(const float (&v)[32], int kind, bool of16, float yb, float yc, bool diag,
                                            int d, uint32_t (&w)[16]) {
    if (kind == 0) {
#pragma unroll
        for (int j = 0; j < 16; ++j) w[j] = round16x2(v[2 * j], v[2 * j + 1], of16);
    } else if (kind == 1) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            uint32_t hi;
            split16x2(v[2 * j], v[2 * j + 1], of16, hi, w[j]);
        }
    } else if (diag) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            w[j] = round16x2(yc * v[2 * j] + (2 * j == d ? yb : 0.f), yc * v[2 * j + 1] + (2 * j + 1 == d ? yb : 0.f), of16);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) w[j] = round16x2(yc * v[2 * j], yc * v[2 * j + 1], of16);
    }
}

// kEpiPoly without Horner's form: v = cc v + cb G for this lane's row and 32 columns from c0 (G past
// L1: within the polar loop other SMs rewrite it in every iteration).  Which product is rounded is
// spelled out: left to the compiler it differs between instantiations and columns, and with it
// the result's bits.  A block cut short rounds the other product than a whole one, as it always has.
__device__ __forceinline__ void add_gram(const GemmGroup& g, const TileInfo& ti, bool f16, int row, int c0,
                                         float (&v)[32]) {
    const int64_t goff = ti.b * g.bf_batch_stride + static_cast<int64_t>(row) * g.ld_bf + c0;
    const uint16_t* gh = reinterpret_cast<const uint16_t*>(g.g_hi) + goff;
    const uint16_t* gl = reinterpret_cast<const uint16_t*>(g.g_lo) + goff;
    const float cb = ti.cb, cc = ti.cc;
    if (g.N - c0 >= 32) {
        const uint4* h4 = reinterpret_cast<const uint4*>(gh);
        const uint4* l4 = reinterpret_cast<const uint4*>(gl);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 hh = __ldcg(h4 + q), ll = __ldcg(l4 + q);
            const uint32_t hw[4] = {hh.x, hh.y, hh.z, hh.w};
            const uint32_t lw[4] = {ll.x, ll.y, ll.z, ll.w};
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const float g0 = dec16(hw[w] & 0xFFFFu, f16) + dec16(lw[w] & 0xFFFFu, f16);
                const float g1 = dec16(hw[w] >> 16, f16) + dec16(lw[w] >> 16, f16);
                v[8 * q + 2 * w] = fmaf(cb, g0, cc * v[8 * q + 2 * w]);
                v[8 * q + 2 * w + 1] = fmaf(cb, g1, cc * v[8 * q + 2 * w + 1]);
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < g.N - c0) v[j] = fmaf(cc, v[j], cb * (dec16(__ldcg(gh + j), f16) + dec16(__ldcg(gl + j), f16)));
    }
}

// A Gram tile's partial sums (sum of squares, trace, squared distance from I; an entry off the
// diagonal counts for its mirror too): fixed-order warp reduction into this warp's slot.
__device__ __forceinline__ void gram_sums_store(const GemmGroup& g, const TileInfo& ti, float sq, float tr, float dev,
                                                int eg, int half, int lane, uint32_t crank) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
        tr += __shfl_xor_sync(0xffffffffu, tr, o);
        dev += __shfl_xor_sync(0xffffffffu, dev, o);
    }
    if (lane == 0) {
        const int ntiles = g.sym ? g.tiles_sym : g.tiles_m * g.tiles_n;
        float* slot = g.part + ((g.part_base + static_cast<int64_t>(ti.b) * ntiles + ti.tile) * kPartSlots +
                                static_cast<int>(crank) * kEpiWarps + half * 4 + eg) * 3;
        slot[0] = sq;
        slot[1] = tr;
        slot[2] = dev;
    }
}

// The blocks of `width` columns that a half of the epilogue's warps takes: it stores [begin, end),
// an even split of those that the tile has (one half stored all of a tile of up to 128 columns:
// steps of 64-wide matrices 373 -> 344 us).  A tile's sums (of G^2, G's trace, tr(Q^T Delta)) go by
// fixed columns instead, half 0's below BN / 2, so that their order, and with it every bit of
// the result, does not depend on how the stores are dealt: half 0 looks at [end, sums_end) for
// them alone, and half 1 sums from block sums_begin on.  (Sums dealt as the stores are: 336 us
// instead of 338 there, another order for each width.)  Of an odd number of blocks half 1
// stores one more, as half 0 has sums to add.
struct HalfBlocks {
    int begin, end, sums_begin, sums_end;
};
__device__ __forceinline__ HalfBlocks half_blocks(const GemmGroup& g, const TileInfo& ti, int half, int width, bool sums) {
    const int blocks = (min(BN, g.N - ti.n0) + width - 1) / width, mid = blocks / 2, fixed = BN / 2 / width;
    HalfBlocks r;
    r.begin = half ? mid : 0;
    r.end = half ? blocks : mid;
    r.sums_begin = half ? fixed : 0;
    r.sums_end = sums && !half ? min(blocks, fixed) : r.end;
    return r;
}

// Epilogue of an update tile (kEpiXSplit: X = xs acc) or of a tile above the diagonal of a
// symmetric output (Gram, polynomial), for one warp's 32 rows and half of the columns.  A plane leaves
// 64 columns at a time through the warp's whole staging (32 rows of 128 bytes, 128-byte
// swizzle) and one TMA store: the TMA unit, which also brings the operands, takes a row of up
// to 128 bytes every ~2 cycles, so 64-byte rows cost it twice.  The accumulator is read again
// for each plane.  (A tile alone in a launch 16.2 -> 13.6 us, 1016-wide updates 238 -> 219 us;
// 1024-wide ones are bound elsewhere and level.)
template <int EPI, bool ROLLED>
__device__ __forceinline__ void wide_epilogue(const TileFlags& p, const GemmGroup& g, const TileInfo& ti,
                                              uint32_t tacc, bool ok, int eg, int half, int lane, uint32_t crank,
                                              uint32_t stg) {
    const int b = ti.b, row_base = ti.m0 + eg * 32, row = row_base + lane;
    const bool row_ok = row < g.M, of16 = p.out_f16 != 0;
    const bool have = ti.run_mma && ok;
    const float xs = EPI == kEpiXSplit ? ti.xs : 1.f;
    const int lo_plane = (ti.horner || ti.hi_only || g.st_lo == nullptr) ? 0 : 1;
    const int nplanes = 1 + lo_plane + ((EPI == kEpiGram && p.gram_y) ? 1 : 0);
    const int st64 = EPI == kEpiXSplit ? 0 : kSt64;
    const uint32_t row_addr = stg + lane * 128 + ((lane & 7) << 4);
    float s_tq = 0.f, s_sq = 0.f;  // shares of tr(Q^T Delta) (ti.trace), of the sum of G^2
    const HalfBlocks hb = half_blocks(g, ti, half, 64, EPI == kEpiGram || (EPI == kEpiXSplit && ti.trace));
#pragma unroll 1
    for (int c64 = hb.begin; c64 < hb.sums_end; ++c64) {
        const int col0 = ti.n0 + c64 * 64;
        if (col0 >= g.N || row_base >= g.M) break;
        const bool store = c64 < hb.end, sums = c64 >= hb.sums_begin;
        // kEpiPoly keeps the lo plane's words: reading G again for it made the first polynomial of
        // 86 matrices of 1024 take 251 us, so 211
        uint32_t lo[2][16];
        constexpr bool kKeepLo = EPI == kEpiPoly;
        constexpr int kUnroll = ROLLED && !kKeepLo ? 1 : EPI == kEpiGram ? 3 : 2;
#pragma unroll kUnroll
        for (int pl = 0; pl < (store ? nplanes : 1); ++pl) {
            const int kind = pl == 0 ? 0 : pl == lo_plane ? 1 : 2;
            if (elect_one()) bulk_wait_read0();
            __syncwarp();
            constexpr int kUnrollH = ROLLED && !kKeepLo ? 1 : 2;
#pragma unroll kUnrollH
            for (int h = 0; h < 2; ++h) {
                if (kKeepLo && pl == 1) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        st_shared4(row_addr ^ ((h * 4 + q) << 4), lo[h][4 * q], lo[h][4 * q + 1], lo[h][4 * q + 2], lo[h][4 * q + 3]);
                    continue;
                }
                float v[32];
                if (have) {
                    uint32_t r[32];
                    tmem_ld32(tacc + (static_cast<uint32_t>(eg * 32) << 16) + c64 * 64 + h * 32, r);
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        v[j] = EPI == kEpiXSplit ? __uint_as_float(r[j]) * xs : __uint_as_float(r[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0.f;
                }
                const int c0 = col0 + h * 32, nvalid = g.N - c0;
                if (row_ok && nvalid > 0) {
                    if (EPI == kEpiPoly && !ti.horner) add_gram(g, ti, p.in_f16 != 0, row, c0, v);
                    if (EPI == kEpiXSplit && ti.trace && pl == 0 && sums) s_tq = trace_share(g, ti, v, row, c0, s_tq);
                    if (EPI == kEpiGram && pl == 0 && sums) {
                        // every entry counts twice, and (G - I) = G here
                        if (nvalid >= 32) {
                            float ss = 0.f;
#pragma unroll
                            for (int j = 0; j < 32; ++j) ss = fmaf(v[j], v[j], ss);
                            s_sq = fmaf(2.f, ss, s_sq);
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (j < nvalid) s_sq = fmaf(2.f * v[j], v[j], s_sq);
                        }
                    }
                }
                if (!store) continue;
                uint32_t w[16];
                plane_words(v, kind, of16, 0.f, ti.yc, false, 0, w);
                if (kKeepLo && lo_plane) plane_words(v, 1, of16, 0.f, 0.f, false, 0, lo[h]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st_shared4(row_addr ^ ((h * 4 + q) << 4), w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
            }
            if (!store) break;
            fence_proxy_async_smem();
            __syncwarp();
            if (elect_one()) {
                tma_store_3d(kind == 0 ? g.st_hi + st64 : kind == 1 ? g.st_lo + st64 : g.st_y + kStY64, stg, col0,
                             row_base, b);
                bulk_commit();
            }
        }
    }
    if (EPI == kEpiXSplit && ti.trace) trace_store(g, ti, s_tq, eg, half, lane, crank);
    if (EPI == kEpiGram) gram_sums_store(g, ti, s_sq, 0.f, s_sq, eg, half, lane, crank);
}

// Epilogue of one tile's column half, run by four warps (thread (eg, lane) owns
// output row m0 + 32 eg + lane).  `tacc` is the tensor-memory accumulator of the tile.
// Of a symmetric 16-bit output (Gram, polynomial) only the tiles on and above the diagonal are
// stored.  A diagonal tile goes one 32 x 32 block at a time: blocks below the diagonal are
// skipped, a block above it is also stored transposed, and the diagonal block is made
// symmetric in shared memory (its upper half mirrored) before its single store, so every
// entry is written once and the matrix is bitwise symmetric.
template <int EPI, bool ROLLED>
__device__ __forceinline__ void tile_epilogue(const TileFlags& p, const GemmGroup& g, const TileInfo& ti, uint32_t tacc,
                                              bool ok, int eg, int half, int lane, uint32_t crank, uint32_t stg) {
    const int b = ti.b, m0 = ti.m0, n0 = ti.n0, split = ti.split;
    // (the polar loop's tiles, ROLLED, are never split over K, and symmetric here)
    const bool f32_out = (EPI == kEpiF32) || (!ROLLED && EPI == kEpiGram && g.splits > 1);
    if (EPI == kEpiXSplit || (!f32_out && n0 != (m0 & ~(kTileM - 1)))) {
        wide_epilogue<EPI, ROLLED>(p, g, ti, tacc, ok, eg, half, lane, crank, stg);
        return;
    }
    const int row_base = m0 + eg * 32;
    const int row = row_base + lane;
    const bool row_ok = row < g.M;
    const bool sym = ROLLED || g.sym != 0;
    const bool gram_fused = EPI == kEpiGram && !f32_out;
    const bool of16 = p.out_f16 != 0;
    // planes written: hi, lo (if kept; not for a Horner-form P, whose lo plane nobody reads),
    // and for the Gram with p.gram_y the plane Y = yb I + yc G (hi only)
    const int lo_plane = (ti.horner || ti.hi_only || g.st_lo == nullptr) ? 0 : 1;
    const int nplanes = 1 + lo_plane + ((EPI == kEpiGram && p.gram_y) ? 1 : 0);
    float s_sq = 0.f, s_tr = 0.f, s_dev = 0.f;
    const HalfBlocks hb = half_blocks(g, ti, half, 32, gram_fused);
#pragma unroll 1
    for (int c32 = hb.begin; c32 < hb.sums_end; ++c32) {
        const int col0 = n0 + c32 * 32;
        if (col0 >= g.N || row_base >= g.M) break;
        if (sym && col0 < row_base) continue;  // block below the diagonal (warp-uniform)
        const bool diag = sym && col0 == row_base;
        float v[32];
        __syncwarp();
        if (ti.run_mma && ok) {
            uint32_t r[32];
            tmem_ld32(tacc + (static_cast<uint32_t>(eg * 32) << 16) + c32 * 32, r);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = 0.f;
        }
        const int nvalid = min(32, g.N - col0);
        const int d = row - col0;  // column index of this lane's diagonal entry in the block
        if (EPI == kEpiPoly) {
            if (!ti.horner && row_ok) add_gram(g, ti, p.in_f16 != 0, row, col0, v);
            const float ca = ti.ca;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (j == d) v[j] += ca;
        }
        const bool sums = gram_fused && row_ok && c32 >= hb.sums_begin;
        if (sums && sym && !diag && nvalid == 32) {
            // block strictly above the diagonal: every entry counts twice and (G - I) = G
            float ss = 0.f;
#pragma unroll
            for (int j = 0; j < 32; ++j) ss = fmaf(v[j], v[j], ss);
            s_sq = fmaf(2.f, ss, s_sq);
            s_dev = fmaf(2.f, ss, s_dev);
        } else if (sums) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                if (j < nvalid && (!sym || j >= d)) {
                    const float x = v[j];
                    const float e = (j == d) ? x - 1.f : x;
                    const float w = (sym && j > d) ? 2.f : 1.f;  // mirrored entry counts twice
                    s_sq = fmaf(w * x, x, s_sq);
                    s_dev = fmaf(w * e, e, s_dev);
                    if (j == d) s_tr += x;
                }
            }
        }
        if (c32 >= hb.end) continue;
        if (f32_out) {
            if (!row_ok) continue;
            float* base = g.out_f32 + split * g.f32_split_stride + b * g.f32_batch_stride;
            float* out = base + static_cast<int64_t>(row) * g.ld_f32 + col0;
            if (!diag && nvalid == 32 && (g.ld_f32 & 3) == 0) {
                float4* o4 = reinterpret_cast<float4*>(out);
#pragma unroll
                for (int q = 0; q < 8; ++q) o4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (j < nvalid && (!sym || j >= d)) out[j] = v[j];
            }
            if (sym) {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (j < nvalid && j > d) base[static_cast<int64_t>(col0 + j) * g.ld_f32 + row] = v[j];
            }
            continue;
        }
        // ---- 16-bit planes through shared memory and TMA stores, one after the other.  ROLLED:
        // the code of one store serves them all (the polar loop's tiles of small matrices run
        // through it once per phase, fetched at ~12 cycles per instruction)
        constexpr int kUnroll = ROLLED ? 1 : 3;
#pragma unroll kUnroll
        for (int pl = 0; pl < nplanes; ++pl) {
            const int kind = pl == 0 ? 0 : pl == lo_plane ? 1 : 2;
            uint32_t w[16];
            plane_words(v, kind, of16, ti.yb, ti.yc, diag, d, w);
            stage_store_block(w, kind == 0 ? g.st_hi : kind == 1 ? g.st_lo : g.st_y, stg, diag, lane, col0, row_base, b);
        }
    }
    if (gram_fused) gram_sums_store(g, ti, s_sq, s_tr, s_dev, eg, half, lane, crank);
}

// Position in the shared-memory ring; one pass around it flips the phase.
struct RingPos {
    int stage;
    uint32_t phase;
};

// Loads k-blocks [from, to) of a tile into the ring (one thread of each CTA of the pair): this
// CTA's rows of A and its half of B's rows, AMN / BMN their layouts, a and b their hi planes'
// maps (the lo planes' follow them).  The bytes of both CTAs complete on rank 0's `full`
// barriers (shared::cluster address fbar0 of the first).  The wait for the next stage is tested
// while this stage's loads are issued.  False on a timeout.
template <bool AMN, bool BMN>
__device__ __forceinline__ bool load_run(const CUtensorMap* a_hi, const CUtensorMap* b_hi, const TileInfo& ti, int from,
                                         int to, uint32_t sbase, uint32_t stride, int nstages, uint64_t* full,
                                         uint64_t* empty, uint32_t fbar0, uint32_t crank, RingPos& pos) {
    const CUtensorMap *a_lo = a_hi + 1, *b_lo = b_hi + 1;
    const bool as = ti.a_split, bs = ti.b_split;
    const uint32_t off_b = kTileABytes * (as ? 2u : 1u);
    const uint32_t pair_bytes = 2u * (off_b + kTileBBytes * (bs ? 2u : 1u));
    const int m0 = ti.m0, nb0 = ti.n0 + static_cast<int>(crank) * (ti.n_mma / 2), b = ti.b;
    const int k_end = to * BK;
    bool ready = mbar_test(&empty[pos.stage], pos.phase ^ 1u);
#pragma unroll 1
    for (int k0 = from * BK; k0 < k_end; k0 += BK) {
        const int s = pos.stage;
        if (!ready && !mbar_wait(&empty[s], pos.phase ^ 1u)) return false;
        if (++pos.stage == nstages) {
            pos.stage = 0;
            pos.phase ^= 1u;
        }
        ready = mbar_test(&empty[pos.stage], pos.phase ^ 1u);
        if (crank == 0) mbar_arrive_expect_tx(&full[s], pair_bytes);
        const uint32_t fbar = fbar0 + 8u * s;
        const uint32_t sa = sbase + s * stride, sb = sa + off_b;
        if (AMN) {
#pragma unroll
            for (int c = 0; c < BM / 64; ++c) {
                tma_load_3d_pair(sa + c * (BK * 128), a_hi, fbar, m0 + 64 * c, k0, b);
                if (as) tma_load_3d_pair(sa + kTileABytes + c * (BK * 128), a_lo, fbar, m0 + 64 * c, k0, b);
            }
        } else {
            tma_load_3d_pair(sa, a_hi, fbar, k0, m0, b);
            if (as) tma_load_3d_pair(sa + kTileABytes, a_lo, fbar, k0, m0, b);
        }
        if (BMN) {
#pragma unroll
            for (int c = 0; c < kBRows / 64; ++c) {
                tma_load_3d_pair(sb + c * (BK * 128), b_hi, fbar, nb0 + 64 * c, k0, b);
                if (bs) tma_load_3d_pair(sb + kTileBBytes + c * (BK * 128), b_lo, fbar, nb0 + 64 * c, k0, b);
            }
        } else {
            tma_load_3d_pair(sb, b_hi, fbar, k0, nb0, b);
            if (bs) tma_load_3d_pair(sb + kTileBBytes, b_lo, fbar, k0, nb0, b);
        }
    }
    return true;
}

// The maps of a run's operands (at / bt: read from the transposed tiles).
__device__ __forceinline__ const CUtensorMap* map_a(const GemmGroup& g, bool at) { return g.a_hi + (at ? g.a_tri : 0); }
__device__ __forceinline__ const CUtensorMap* map_b(const GemmGroup& g, bool bt) { return g.b_hi + (bt ? g.b_tri : 0); }

// All of a tile's k-blocks.
__device__ __forceinline__ bool load_tile(const GemmGroup& g, const TileInfo& ti, uint32_t sbase, uint32_t stride,
                                          int nstages, uint64_t* full, uint64_t* empty, uint32_t fbar0, uint32_t crank,
                                          RingPos& pos) {
    return for_k_runs(ti, [&](int from, int to, bool at, bool bt) {
        const CUtensorMap *a = map_a(g, at), *b = map_b(g, bt);
        if (g.a_mn || at)
            return g.b_mn || bt ? load_run<true, true>(a, b, ti, from, to, sbase, stride, nstages, full, empty, fbar0, crank, pos)
                                : load_run<true, false>(a, b, ti, from, to, sbase, stride, nstages, full, empty, fbar0, crank, pos);
        return g.b_mn || bt ? load_run<false, true>(a, b, ti, from, to, sbase, stride, nstages, full, empty, fbar0, crank, pos)
                            : load_run<false, false>(a, b, ti, from, to, sbase, stride, nstages, full, empty, fbar0, crank, pos);
    });
}

// Issues MMAs of a tile (one thread of rank 0) over nkb k-blocks of the ring, in one layout (acc 0
// before the tile's first): the passes
// hi hi (+ hi lo_B) (+ lo_A hi) of each 16-deep slice, accumulated in tensor memory at tacc.
// a_lo, b_lo: low descriptor words of the hi planes in stage 0.  A stage or slice only moves
// the start address (a 14-bit field; every shared address is below 256 KB, so the sum never
// carries out of it).  The barrier of the next stage is tested between this stage's MMAs, so
// that its latency hides behind them: a k-block's four 1-pass MMAs take 512 cycles (128 each,
// the tensor core's rate), and what the thread does between two k-blocks' MMAs has to stay
// below the few queued ones.  Measured per 64-deep k-block without loads and epilogue (114 x
// 1024^3): 390 ns -> 278 ns with one pass, 638 -> 540 with two, 806 -> 805 with three, against
// the loop that chose the passes per MMA, built 64-bit descriptors and ran under
// `lane == 0`.  With loads 360 ns: a k-block's 32 KB arrive at ~64 bytes per cycle and SM.
// False on a timeout.
template <bool AS, bool BS>
__device__ __forceinline__ bool issue_tile(uint64_t* full, uint64_t* empty, int nstages, uint32_t stride16, int nkb,
                                           uint32_t tacc, uint32_t idesc, uint32_t a_lo, uint32_t a_hi,
                                           uint32_t b_lo, uint32_t b_hi, uint32_t step_a, uint32_t step_b,
                                           RingPos& pos, uint32_t& acc) {
    constexpr uint32_t kA16 = kTileABytes >> 4, kB16 = kTileBBytes >> 4;  // hi -> lo plane
    uint32_t so = pos.stage * stride16;
    bool ready = mbar_test(&full[pos.stage], pos.phase);
#pragma unroll 1
    for (int kb = 0; kb < nkb; ++kb) {
        const int s = pos.stage;
        if (!ready && !mbar_wait(&full[s], pos.phase)) return false;
        tc_fence_after();
        const uint32_t a = a_lo + so, b = b_lo + so;
        so += stride16;
        if (++pos.stage == nstages) {
            pos.stage = 0;
            pos.phase ^= 1u;
            so = 0u;
        }
#pragma unroll
        for (int ks = 0; ks < BK / 16; ++ks) {
            const uint32_t da = a + ks * step_a, db = b + ks * step_b;
            umma_16bit_pair(tacc, da, a_hi, db, b_hi, idesc, acc);
            if (BS) umma_16bit_pair(tacc, da, a_hi, db + kB16, b_hi, idesc, 1u);
            if (AS) umma_16bit_pair(tacc, da + kA16, a_hi, db, b_hi, idesc, 1u);
            acc = 1u;
            if (ks == BK / 16 - 2) ready = mbar_test(&full[pos.stage], pos.phase);
        }
        umma_commit_pair_mc(&empty[s], 0x3);  // the stage is free in both CTAs once they have read it
    }
    return true;
}

}  // namespace isoloco
