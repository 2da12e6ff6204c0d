// rowsum.cuh -- device helpers shared by the forward and backward day kernels.
//
// Edge storage is SELL-32 (sliced ELLPACK, one slice per 32-row warp tile) in pairs of
// entries: pair q of the row in lane l of a slice sits at cw[slice_ptr[s] + 32 q + l] and
// holds {column, weight, column, weight} of entries 2q and 2q + 1.  A warp reads two
// entries of its 32 rows with one 16-byte load per lane (512 consecutive bytes), where
// separate column and weight arrays took four loads and their addresses; the day kernels
// issue about as many instructions as they wait for memory, so the count matters.  Every
// lane sums its own row in entry order.  The sum of a row therefore depends only on the
// row (the same operation sequence wherever and whenever it is computed), so a sum
// recomputed in the backward is bitwise the forward's.  Rows are laid out so that a slice
// holds rows of similar length (little padding).
#pragma once

#include "gabm_internal.cuh"

namespace gabm {

#ifndef GABM_GATHER_PAIRS
#define GABM_GATHER_PAIRS 2
#endif
#ifndef GABM_MINBLOCKS
#define GABM_MINBLOCKS 3
#endif
// Pairs of entries per lane loaded ahead of use: by the gathers (whose kernels have little
// register room left) and by the marked sums.
constexpr int kGP = GABM_GATHER_PAIRS;
constexpr int kMP = 4;

__device__ __forceinline__ void kahan_add(float &s, float &c, float x) {
    const float y = __fsub_rn(x, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

// kahan_add when `take`, else no change (selects instead of a branch).
__device__ __forceinline__ void kahan_add_if(float &s, float &c, float x, bool take) {
    const float y = __fsub_rn(x, c);
    const float t = __fadd_rn(s, y);
    const float cn = __fsub_rn(__fsub_rn(t, s), y);
    s = take ? t : s;
    c = take ? cn : c;
}

// Infectiousness of a neighbour exposed on day e_j, seen on day t: c[t - e_j] for
// 1 <= t - e_j < L, else 0 (susceptible agents, padding rows, long-recovered agents).
__device__ __forceinline__ float infectiousness(int e_j, const float *c_s, int t, int L) {
    const int k = t - e_j;
    return ((unsigned)(k - 1) < (unsigned)(L - 1)) ? c_s[k] : 0.f;
}

// A compile-time width.
template <int N>
struct Width {
    static constexpr int value = N;
};

// Whether row j is marked in a per-day bitmap of infectious rows (read-only during the launch).
__device__ __forceinline__ bool marked(const uint32_t *bits, uint32_t j) {
    return (bits[j >> 5] >> (j & 31u)) & 1u;
}

// Hands tiles to a warp in runs claimed with one atomic each from the launch's
// counter.  All warps hammering one counter with a tile per atomic serialises
// on that address, so runs hold up to 16 tiles and shrink as the counter nears
// the end (guided scheduling keeps the tail short); the next run is claimed
// one run ahead so the atomic's latency is hidden.
struct TileDispenser {
    int *ctr;
    int ntiles, nwarps, lane;
    int next, end;     // current run [next, end)
    int pend;          // lane 0: first tile of the claimed next run
    int pend_len;      // its length (warp-uniform)

    __device__ __forceinline__ int run_len(int from) const {
        const int rem = ntiles - from;
        return max(1, min(16, rem / (4 * nwarps)));
    }
    __device__ __forceinline__ void init(int *c, int nt, int nw, int ln) {
        ctr = c;
        ntiles = nt;
        nwarps = nw;
        lane = ln;
        next = end = 0;
        pend_len = run_len(0);
        pend = (lane == 0) ? atomicAdd(ctr, pend_len) : 0;
    }
    // the next tile of this warp, or a value >= ntiles when the launch's tiles are gone
    __device__ __forceinline__ int get() {
        if (next >= end) {
            const int base = __shfl_sync(0xffffffffu, pend, 0);
            if (base >= ntiles) return ntiles;
            next = base;
            end = base + pend_len;
            pend_len = run_len(end);
            if (lane == 0) pend = atomicAdd(ctr, pend_len);
        }
        return next < ntiles ? next++ : ntiles;
    }
};

// Hands each block one contiguous range of tiles; its warps take the first two rounds in
// order and the rest one at a time through a shared-memory counter.  Rows are laid out in
// groups, so the neighbours of a range's rows mostly lie in and around the same range:
// the warps of a block gather from lines their own SM has just cached, where a
// launch-wide counter would spread consecutive tiles over all SMs.  (Measured
// on the 1M-agent typed graph: 10% shorter day kernels than the launch-wide
// dispenser; handing the last eighth of the tiles out launch-wide to balance
// the tail costs more locality than it gains.  The batched kernels, whose rows
// carry up to 64 sets each, keep the launch-wide dispenser: there the ranges'
// imbalance cost 7%.)  Called by every thread of the block (init holds a barrier).
struct BlockTiles {
    int *ctr;          // the block's counter (shared memory)
    int end, ntiles, lane, pend, given, first, nw;
    __device__ __forceinline__ void init(int nt, int ln) {
        __shared__ int s_ctr;
        ntiles = nt;
        lane = ln;
        nw = (int)(blockDim.x >> 5);
        const int b0 = (int)(((long long)blockIdx.x * nt) / gridDim.x);
        end = (int)(((long long)(blockIdx.x + 1) * nt) / gridDim.x);
        first = b0 + (int)(threadIdx.x >> 5);
        given = 0;
        pend = 0;
        if (threadIdx.x == 0) s_ctr = b0 + 2 * nw;
        __syncthreads();
        ctr = &s_ctr;
    }
    // the next tile of this warp, or ntiles when the block's range is done
    __device__ __forceinline__ int get() {
        int tile;
        if (given < 2) {
            tile = first + given * nw;
            if (++given == 2 && lane == 0) pend = atomicAdd(ctr, 1);
        } else {
            tile = __shfl_sync(0xffffffffu, pend, 0);
            if (tile < end && lane == 0) pend = atomicAdd(ctr, 1);
        }
        return tile < end ? tile : ntiles;
    }
};

// Warp sums of v by age bin.  Bin b's 32 values lie in shared memory (the warp's `cells`,
// zero outside this call), even lanes' in its row 2b, odd lanes' in row 2b + 1; lane r < 2
// kAges sums row r with four 16-byte loads and the two rows' sums meet in one shuffle: lanes
// 2b and 2b + 1 return bin b's sum.  About 30 instructions for all bins, where a
// reduce-scatter over the lanes took 100 and a butterfly per bin 200.  The addition tree is
// the butterfly's (lanes 16 apart first, neighbours last), so the sums do not depend on
// anything but the inputs.  Rows are 20 words apart: eight lanes' 16-byte loads then cover
// all banks once.  Called by all 32 lanes; lanes with nothing to add pass v = 0.
constexpr int kBinStride = 20;
constexpr int kBinWords = 2 * kAges * kBinStride;   // shared-memory words per warp
__device__ __forceinline__ float warp_bin_sums(float v, int bin, int lane, float *cells) {
    float *cell = cells + (2 * bin + (lane & 1)) * kBinStride + (lane >> 1);
    *cell = v;
    __syncwarp();
    float x[16];
    if (lane < 2 * kAges) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 q = *reinterpret_cast<const float4 *>(cells + lane * kBinStride + 4 * i);
            x[4 * i] = q.x; x[4 * i + 1] = q.y; x[4 * i + 2] = q.z; x[4 * i + 3] = q.w;
        }
#pragma unroll
        for (int h = 8; h >= 1; h >>= 1)
#pragma unroll
            for (int i = 0; i < h; ++i) x[i] = __fadd_rn(x[i], x[i + h]);
    } else {
        x[0] = 0.f;
    }
    __syncwarp();
    *cell = 0.f;
    return __fadd_rn(x[0], __shfl_xor_sync(0xffffffffu, x[0], 1));
}

// Row data of one tile, loaded one tile ahead of use.
struct TileRows {
    int tile;
    int e;            // exposure day of this lane's row
    uint32_t len;     // this lane's row_len word: entries in the slice, or a long row's index (see split_len)
    uint32_t p0;      // the tile's slice
    int g;            // graph of the tile
    bool flag;        // the row has an infectious in-neighbour today (true without flags)
};

// A row_len word: entries in the slice, and the index of a long row or -1.
__device__ __forceinline__ void split_len(uint32_t v, uint32_t &len, int &lrow) {
    const bool lng = (v & kLongBit) != 0u;
    len = lng ? 0u : v;
    lrow = lng ? (int)(v & ~kLongBit) : -1;
}

// What no launch of a day loop writes (row layout), and the rest.
__device__ __forceinline__ void load_tile_layout(const Sell &m, const uint16_t *tile_graph, int ntiles, int tile,
                                                 int lane, TileRows &tr) {
    tr.tile = tile;
    tr.len = 0;
    tr.p0 = 0;
    tr.g = 0;
    if (tile < ntiles) {
        tr.len = m.row_len[tile * kTile + lane];
        tr.p0 = m.slice_ptr[tile];
        tr.g = tile_graph ? (int)tile_graph[tile] : 0;
    }
}

__device__ __forceinline__ void load_tile_state(const int16_t *e, int ntiles, int lane, TileRows &tr,
                                                const uint8_t *flags = nullptr) {
    tr.e = kPad;
    tr.flag = true;
    if (tr.tile < ntiles) {
        const int row = tr.tile * kTile + lane;
        tr.e = e[row];
        if (flags) tr.flag = flags[row] != 0;
    }
}

__device__ __forceinline__ void load_tile_rows(const Sell &m, const int16_t *e, const uint16_t *tile_graph,
                                               int ntiles, int tile, int lane, TileRows &tr,
                                               const uint8_t *flags = nullptr) {
    load_tile_layout(m, tile_graph, ntiles, tile, lane, tr);
    load_tile_state(e, ntiles, lane, tr, flags);
}

// The column and weight of entry k of the row in lane r of a slice.
__device__ __forceinline__ const uint2 *entry_ptr(const Sell &m, uint32_t p0, uint32_t k, int r) {
    return reinterpret_cast<const uint2 *>(m.cw + p0 + 32u * (k >> 1) + (uint32_t)r) + (k & 1u);
}

// Sets flags[j] = 1 for every out-neighbour j of the tile rows whose lane has `push`
// (byte stores: every writer stores the same value, so the result does not depend on
// their order).  Up to two rows: one at a time, the lanes splitting the row's entries.
// More: every lane walks its own row, kMP pairs in flight; taken one at a time, the rows
// of a tile with a dozen infectious agents would cost a dozen load round trips in a row.
// `own` is the tile's row data of the in-edges: the same as the out-edges' where the
// weights are symmetric, which spares a round trip.  Called by all 32 lanes.
__device__ __forceinline__ void push_flags(const Sell &m, const Sell &m_out, const TileRows &own, int lane, bool push,
                                           uint8_t *flags) {
    unsigned rows = __ballot_sync(0xffffffffu, push);
    if (!rows) return;
    const bool same = m.cw == m_out.cw;
    const uint32_t base = same ? own.p0 : m_out.slice_ptr[own.tile];
    uint32_t my_len = !push ? 0u : (same ? own.len : m_out.row_len[own.tile * kTile + lane]);
    if (my_len & kLongBit) my_len = 0u;   // the next day's long-row launch pushes these
    if (__popc(rows) <= 2) {
        while (rows) {
            const int r = __ffs(rows) - 1;
            rows &= rows - 1u;
            const uint32_t len = __shfl_sync(0xffffffffu, my_len, r);
            for (uint32_t k = (uint32_t)lane; k < len; k += 32u) flags[__ldg(&entry_ptr(m_out, base, k, r)->x)] = 1;
        }
        return;
    }
    const uint32_t np = (my_len + 1u) >> 1;
    const uint4 *row = m_out.cw + base + (uint32_t)lane;
    for (uint32_t q0 = 0; q0 < np; q0 += kMP) {
        uint4 v[kMP];
#pragma unroll
        for (int u = 0; u < kMP; ++u) v[u] = __ldg(row + 32u * min(q0 + (uint32_t)u, np - 1u));
#pragma unroll
        for (int u = 0; u < kMP; ++u) {
            if (q0 + (uint32_t)u < np) flags[v[u].x] = 1;
            if (2u * (q0 + (uint32_t)u) + 1u < my_len) flags[v[u].z] = 1;
        }
    }
}

// Loads that are skipped (value left at `dflt`) when pred is false, written as
// predicated PTX so that a batch of them issues without branches.
__device__ __forceinline__ uint32_t ld_cs_if(const uint32_t *p, bool pred) {
    uint32_t v = 0u;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.cs.u32 %0, [%1]; }" : "+r"(v) : "l"(p), "r"((uint32_t)pred));
    return v;
}
__device__ __forceinline__ float ld_cs_if(const float *p, bool pred) {
    float v = 0.f;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.cs.f32 %0, [%1]; }" : "+f"(v) : "l"(p), "r"((uint32_t)pred));
    return v;
}
__device__ __forceinline__ float ld_if(const float *p, bool pred) {
    float v = 0.f;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.f32 %0, [%1]; }" : "+f"(v) : "l"(p), "r"((uint32_t)pred));
    return v;
}
__device__ __forceinline__ uint32_t ld_if(const uint32_t *p, bool pred) {
    uint32_t v = 0u;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.u32 %0, [%1]; }" : "+r"(v) : "l"(p), "r"((uint32_t)pred));
    return v;
}
__device__ __forceinline__ int ld_if(const int16_t *p, bool pred, int dflt) {
    int v = dflt;
    asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.s16 %0, [%1]; }" : "+r"(v) : "l"(p), "r"((uint32_t)pred));
    return v;
}

// ---- sums over a tile's rows ------------------------------------------------
// What a tile's 32 lanes sum, worked out once per tile by all of them.
struct TileSpan {
    const uint4 *row;   // pair q of this lane's row at row[32 q]
    uint32_t len;       // entries this lane sums (0: nothing)
    uint32_t lim;       // pairs this lane loads: mostly-active slices are read whole, sparse ones row by row
    uint32_t np;        // pairs of the longest summing row (warp-uniform)
    uint32_t kfull;     // entries below this are valid in every lane (warp-uniform)
};

__device__ __forceinline__ TileSpan tile_span(const Sell &m, uint32_t p0, uint32_t len, bool act, int lane) {
    TileSpan s;
    s.row = m.cw + p0 + (uint32_t)lane;
    s.len = act && !(len & kLongBit) ? len : 0u;   // a long row is summed elsewhere
    s.np = (__reduce_max_sync(0xffffffffu, s.len) + 1u) >> 1;
    s.kfull = __reduce_min_sync(0xffffffffu, s.len);
    s.lim = __popc(__ballot_sync(0xffffffffu, act)) >= 24 ? s.np : (s.len + 1u) >> 1;
    return s;
}

// Pairs [q0, q0 + UP) of the lane's row below its limit; the others keep what they held
// (columns of some row, or 0: nothing is added for them).
template <int UP>
__device__ __forceinline__ void load_pairs(const uint4 *row, uint32_t q0, uint32_t lim, uint4 (&v)[UP]) {
#pragma unroll
    for (int u = 0; u < UP; ++u)
        if (q0 + (uint32_t)u < lim) v[u] = __ldcs(row + 32u * (q0 + (uint32_t)u));
}

// sum of w x[j] over the lane's entries, in entry order with compensated summation.  `ea`
// holds the first kGP pairs (load_pairs(row, 0, lim, ea), issued by the caller well ahead:
// before the previous tile's epilogue).  The next batch of pairs is in flight while one is
// used.  Batches in which every lane's entries are valid run without predicates; in the
// others an invalid entry adds y = 0, which leaves the sum as it is (entries are invalid
// from some k on, so the compensation it spoils is not used again).
template <int GP>
__device__ __forceinline__ float gather_sum(const TileSpan &s, const float *x, uint4 (&ea)[GP]) {
    float sum = 0.f, comp = 0.f;
    auto use = [&](uint32_t q0, const uint4 (&v)[GP]) {
        float g[2 * GP];
        if (2u * q0 + 2u * GP <= s.kfull) {
#pragma unroll
            for (int u = 0; u < GP; ++u) {
                g[2 * u] = x[v[u].x];
                g[2 * u + 1] = x[v[u].z];
            }
#pragma unroll
            for (int u = 0; u < GP; ++u) {
                kahan_add(sum, comp, __uint_as_float(v[u].y) * g[2 * u]);
                kahan_add(sum, comp, __uint_as_float(v[u].w) * g[2 * u + 1]);
            }
            return;
        }
#pragma unroll
        for (int u = 0; u < GP; ++u) {
            const uint32_t k = 2u * (q0 + (uint32_t)u);
            g[2 * u] = k < s.len ? x[v[u].x] : 0.f;
            g[2 * u + 1] = k + 1u < s.len ? x[v[u].z] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 2 * GP; ++i) {
            const float w = __uint_as_float((i & 1) ? v[i >> 1].w : v[i >> 1].y);
            const float y = (2u * q0 + (uint32_t)i < s.len) ? __fsub_rn(w * g[i], comp) : 0.f;
            const float t = __fadd_rn(sum, y);
            comp = __fsub_rn(__fsub_rn(t, sum), y);
            sum = t;
        }
    };
    uint4 eb[GP];
#pragma unroll
    for (int u = 0; u < GP; ++u) eb[u] = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t q = 0; q < s.np; q += 2 * GP) {
        if (q + GP < s.np) load_pairs(s.row, q + GP, s.lim, eb);
        use(q, ea);
        if (q + GP >= s.np) break;
        if (q + 2 * GP < s.np) load_pairs(s.row, q + 2 * GP, s.lim, ea);
        use(q + GP, eb);
    }
    return sum;
}

// gather_sum that loads its own first pairs.
__device__ __forceinline__ float gather_sum(const Sell &m, uint32_t p0, uint32_t len, bool act, int lane,
                                            const float *x) {
    const TileSpan s = tile_span(m, p0, len, act, lane);
    uint4 ea[kGP];
#pragma unroll
    for (int u = 0; u < kGP; ++u) ea[u] = make_uint4(0u, 0u, 0u, 0u);
    load_pairs(s.row, 0u, s.lim, ea);
    return gather_sum(s, x, ea);
}

// sum of w c[t - e_j] over the lane's entries whose neighbour j is infectious on day t: marked
// in `bits` and 1 <= t - e_j < L.  Only those entries are added, in entry order with
// compensated summation, so a row's value is a function of its marked entries however
// they are visited.  Entries go 32 at a time: first every entry's bit is tested (the
// bitmap is small enough for L1) and the marks collected in one word per lane; then the
// lanes walk their marks, two or four at a time, reading the entry again and the
// neighbour's exposure day.  On a typical day one entry in twenty is marked, and the
// longest lane has three or four marks, so this runs about a third of the instructions of
// a pass that carries every entry through the lookup and the compensated addition.
template <int UP = kMP>
__device__ __forceinline__ float marked_sum(const Sell &m, uint32_t p0, uint32_t len, bool act, int lane,
                                            const uint32_t *bits, const int16_t *e, const float *c_s, int t, int L) {
    const TileSpan s = tile_span(m, p0, len, act, lane);
    float sum = 0.f, comp = 0.f;
    uint4 ea[UP], eb[UP];
#pragma unroll
    for (int u = 0; u < UP; ++u) ea[u] = eb[u] = make_uint4(0u, 0u, 0u, 0u);
    load_pairs(s.row, 0u, s.lim, ea);
    uint32_t mask = 0u;
    auto word = [&](uint32_t j) { return bits[j >> 5] >> (j & 31u); };
    auto test = [&](uint32_t q0, const uint4 (&v)[UP]) {
        uint32_t w[2 * UP];
#pragma unroll
        for (int u = 0; u < UP; ++u) {
            const uint32_t k = 2u * (q0 + (uint32_t)u);
            w[2 * u] = k < s.len ? word(v[u].x) : 0u;
            w[2 * u + 1] = k + 1u < s.len ? word(v[u].z) : 0u;
        }
        const uint32_t sh = (2u * q0) & 31u;
        uint32_t mk = 0u;
#pragma unroll
        for (int i = 0; i < 2 * UP; ++i) mk |= (w[i] & 1u) << i;
        mask |= mk << sh;
    };
    auto take = [&](uint32_t k0, auto width) {
        constexpr int W = decltype(width)::value;
        uint2 v[W];
        int ej[W];
        bool ok[W];
#pragma unroll
        for (int i = 0; i < W; ++i) {
            ok[i] = mask != 0u;
            const uint32_t k = k0 + (uint32_t)(ok[i] ? __ffs(mask) - 1 : 0);
            mask &= mask - 1u;
            v[i] = make_uint2(0u, 0u);
            if (ok[i]) v[i] = __ldg(reinterpret_cast<const uint2 *>(s.row + 32u * (k >> 1)) + (k & 1u));
        }
#pragma unroll
        for (int i = 0; i < W; ++i) ej[i] = ok[i] ? (int)e[v[i].x] : kNever;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const int k = t - ej[i];
            const bool tk = (unsigned)(k - 1) < (unsigned)(L - 1);
            kahan_add_if(sum, comp, tk ? __uint_as_float(v[i].y) * c_s[k] : 0.f, tk);
        }
    };
    for (uint32_t q = 0; q < s.np; q += 2 * UP) {
        if (q + UP < s.np) load_pairs(s.row, q + UP, s.lim, eb);
        test(q, ea);
        if (q + 2 * UP < s.np) load_pairs(s.row, q + 2 * UP, s.lim, ea);
        if (q + UP < s.np) test(q + UP, eb);
        if (((q + 2 * UP) & 15u) == 0u || q + 2 * UP >= s.np) {   // 32 entries tested, or the last
            const uint32_t k0 = (2u * q) & ~31u;
            for (unsigned n = __reduce_max_sync(0xffffffffu, (unsigned)__popc(mask)); n > 0u;) {
                if (n > 2u) {
                    take(k0, Width<4>{});
                    n = n > 4u ? n - 4u : 0u;
                } else {
                    take(k0, Width<2>{});
                    n = 0u;
                }
            }
        }
    }
    return sum;
}

// marked_sum without the bitmap: every entry's exposure day is gathered and tested, which
// takes the same entries (an exposure during day t itself gives t - e_j = 0): one round trip a
// batch, where the bitmap costs one for the bits and two for the marks.  On every day of the
// base model this is the faster way (250k agents x 120 days: 2.42 ms by the bitmap below a
// quarter of the agents infected, 2.28 without it; 1M x 60: 37.3 and 35.6 us a day).  The
// first pairs loaded ahead, during the tile before, cost more registers than they gave.
template <int UP = kMP>
__device__ __forceinline__ float exposed_sum(const Sell &m, uint32_t p0, uint32_t len, bool act, int lane,
                                             const int16_t *e, const float *c_s, int t, int L) {
    const TileSpan s = tile_span(m, p0, len, act, lane);
    float sum = 0.f, comp = 0.f;
    uint4 ea[UP], eb[UP];
#pragma unroll
    for (int u = 0; u < UP; ++u) ea[u] = eb[u] = make_uint4(0u, 0u, 0u, 0u);
    load_pairs(s.row, 0u, s.lim, ea);
    auto use = [&](uint32_t q0, const uint4 (&v)[UP]) {
        int ej[2 * UP];
#pragma unroll
        for (int u = 0; u < UP; ++u) {
            const uint32_t k = 2u * (q0 + (uint32_t)u);
            ej[2 * u] = k < s.len ? (int)e[v[u].x] : kNever;
            ej[2 * u + 1] = k + 1u < s.len ? (int)e[v[u].z] : kNever;
        }
#pragma unroll
        for (int i = 0; i < 2 * UP; ++i) {
            const float w = __uint_as_float((i & 1) ? v[i >> 1].w : v[i >> 1].y);
            const int k = t - ej[i];
            const bool tk = (unsigned)(k - 1) < (unsigned)(L - 1);
            kahan_add_if(sum, comp, tk ? w * c_s[k] : 0.f, tk);
        }
    };
    for (uint32_t q = 0; q < s.np; q += 2 * UP) {
        if (q + UP < s.np) load_pairs(s.row, q + UP, s.lim, eb);
        use(q, ea);
        if (q + UP >= s.np) break;
        if (q + 2 * UP < s.np) load_pairs(s.row, q + 2 * UP, s.lim, ea);
        use(q + UP, eb);
    }
    return sum;
}

// gather_sum, and for the rows with `lam` the sum of w c[t - e_j] over the neighbours infectious on
// day t (exposed_sum), in one pass over the entries: each pair is read once and its neighbours'
// coefficients and exposure days are gathered together.  (Two passes, gather_sum and then the
// marked neighbours by the day's bitmap: 110 us a day on the 1M-agent town against 91, 50 on the
// 300k-agent power-law graph against 37; one pass that tests the bitmap before it gathers an
// exposure day: 111 and 52.)
template <int GP>
__device__ __forceinline__ float gather_and_exposed_sum(const TileSpan &s, const float *x, bool lam, const int16_t *e,
                                                        const float *c_s, int t, int L, uint4 (&ea)[GP],
                                                        float &lam_sum) {
    float sum = 0.f, comp = 0.f, ls = 0.f, lc = 0.f;
    auto use = [&](uint32_t q0, const uint4 (&v)[GP]) {
        float g[2 * GP];
        int ej[2 * GP];
#pragma unroll
        for (int u = 0; u < GP; ++u) {
            const uint32_t k = 2u * (q0 + (uint32_t)u);
            g[2 * u] = k < s.len ? x[v[u].x] : 0.f;
            g[2 * u + 1] = k + 1u < s.len ? x[v[u].z] : 0.f;
            ej[2 * u] = lam && k < s.len ? (int)e[v[u].x] : kNever;
            ej[2 * u + 1] = lam && k + 1u < s.len ? (int)e[v[u].z] : kNever;
        }
#pragma unroll
        for (int i = 0; i < 2 * GP; ++i) {
            const float w = __uint_as_float((i & 1) ? v[i >> 1].w : v[i >> 1].y);
            const float y = (2u * q0 + (uint32_t)i < s.len) ? __fsub_rn(w * g[i], comp) : 0.f;
            const float tt = __fadd_rn(sum, y);
            comp = __fsub_rn(__fsub_rn(tt, sum), y);
            sum = tt;
            const int k = t - ej[i];
            const bool tk = (unsigned)(k - 1) < (unsigned)(L - 1);
            kahan_add_if(ls, lc, tk ? w * c_s[k] : 0.f, tk);
        }
    };
    uint4 eb[GP];
#pragma unroll
    for (int u = 0; u < GP; ++u) eb[u] = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t q = 0; q < s.np; q += 2 * GP) {
        if (q + GP < s.np) load_pairs(s.row, q + GP, s.lim, eb);
        use(q, ea);
        if (q + GP >= s.np) break;
        if (q + 2 * GP < s.np) load_pairs(s.row, q + 2 * GP, s.lim, ea);
        use(q + GP, eb);
    }
    lam_sum = ls;
    return sum;
}

// Tiles with at most this many summing rows have them summed one row at a time by the
// whole warp (few_row_sums) instead of lane by lane over the tile's longest row.
#ifndef GABM_COOP_ROWS
#define GABM_COOP_ROWS 4
#endif

// The sum of one row's taken contributions by the whole warp: the row of tile lane r
// (entries [k_first, len)), the result in lane r's sum / comp.  The lanes load 32 entries at
// a time and f(j, w, valid, out, take) gives an entry's contribution and whether it is
// added; lane r then adds the taken ones in entry order with the same compensated
// addition, so the value is marked_sum's.  Called by all 32 lanes.
template <class F>
__device__ __forceinline__ void warp_row_sum_from(const Sell &m, uint32_t p0, uint32_t len, uint32_t k_first, int r,
                                                  int lane, F f, float &sum, float &comp) {
    for (uint32_t k0 = k_first; k0 < len; k0 += 32u) {
        const uint32_t k = k0 + (uint32_t)lane;
        const bool valid = k < len;
        uint2 v = make_uint2(0u, 0u);
        if (valid) v = __ldg(entry_ptr(m, p0, k, r));
        float out;
        bool take;
        f(v.x, __uint_as_float(v.y), valid, out, take);
        unsigned mm = __ballot_sync(0xffffffffu, take);
        while (mm) {
            const int src = __ffs(mm) - 1;
            mm &= mm - 1u;
            const float x = __shfl_sync(0xffffffffu, out, src);
            if (lane == r) kahan_add(sum, comp, x);
        }
    }
}

// warp_row_sum_from for up to GABM_COOP_ROWS rows of a tile at once (the rows of `amask`), so
// that their loads overlap: the first 32 entries of every row are loaded, tested and
// gathered together, then each row's lane adds its taken contributions in entry order.
// Each row's value is marked_sum's.  Lanes without a row return 0.  Called by all 32 lanes.
template <class F>
__device__ __forceinline__ float few_row_sums(const Sell &m, uint32_t p0, uint32_t my_len, unsigned amask, int lane,
                                              F f) {
    constexpr int K = GABM_COOP_ROWS;
    float sum = 0.f, comp = 0.f;
    if (my_len & kLongBit) my_len = 0u;
    int r[K];
    uint32_t len[K];
    uint2 v[K];
    float out[K];
    bool take[K];
    unsigned mm = amask;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        r[i] = mm ? __ffs(mm) - 1 : -1;
        mm &= mm - 1u;
        len[i] = __shfl_sync(0xffffffffu, my_len, r[i] < 0 ? 0 : r[i]);
        if (r[i] < 0) len[i] = 0u;
        v[i] = make_uint2(0u, 0u);
        if ((uint32_t)lane < len[i]) v[i] = __ldg(entry_ptr(m, p0, (uint32_t)lane, r[i]));
    }
#pragma unroll
    for (int i = 0; i < K; ++i) f(v[i].x, __uint_as_float(v[i].y), (uint32_t)lane < len[i], out[i], take[i]);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        unsigned tm = __ballot_sync(0xffffffffu, take[i]);
        while (tm) {
            const int src = __ffs(tm) - 1;
            tm &= tm - 1u;
            const float x = __shfl_sync(0xffffffffu, out[i], src);
            if (lane == r[i]) kahan_add(sum, comp, x);
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i)
        if (len[i] > 32u) warp_row_sum_from(m, p0, len[i], 32u, r[i], lane, f, sum, comp);   // len[i]: warp-uniform
    return sum;
}

}  // namespace gabm
