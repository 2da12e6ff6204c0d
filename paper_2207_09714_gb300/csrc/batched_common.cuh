// batched_common.cuh -- device helpers of the batched day kernels (batched.cu,
// batched_bwd.cu): per-lane vectors of SPL sets, the grouped row sums with their
// load pipeline, and the (Bp, SPL) schedules built.
#pragma once

#include <algorithm>

#include "gabm_internal.cuh"
#include "rowsum.cuh"

// Resident blocks per SM the batched day kernels are compiled for (register budget
// 65536 / (256 x blocks) per thread).
#ifndef GABM_BFWD_MINBLOCKS
#define GABM_BFWD_MINBLOCKS 3
#endif

namespace gabm {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr float kUmin = 5.9604644775390625e-8f;   // 2^-24: the smallest uniform (u < p is then impossible)

// Adds w * x (x finite).  Invalid entries carry w = 0: s + 0 * x = s exactly for the
// plain sum (s is never -0); the compensated sum skips them explicitly.
template <bool KAHAN>
__device__ __forceinline__ void acc_add(float &s, float &c, float w, float x, bool take) {
    if (KAHAN) kahan_add_if(s, c, w * x, take);
    else s = __fmaf_rn(w, x, s);
}

// ---- per-lane vectors of SPL sets ----------------------------------------
// SPL int16 exposure days travel as SPL/2 32-bit words, SPL floats as one or two
// vector accesses; the predicated forms load nothing (zeros) when !ok.
template <int SPL>
__device__ __forceinline__ void ld_words(const uint32_t *p, bool ok, uint32_t (&w)[SPL / 2]) {
    const uint32_t pr = ok;
    if constexpr (SPL == 2) {
        w[0] = 0u;
        asm("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.u32 %0, [%1]; }" : "+r"(w[0]) : "l"(p), "r"(pr));
    } else if constexpr (SPL == 4) {
        w[0] = w[1] = 0u;
        asm("{ .reg .pred q; setp.ne.u32 q, %3, 0; @q ld.global.v2.u32 {%0, %1}, [%2]; }"
                     : "+r"(w[0]), "+r"(w[1]) : "l"(p), "r"(pr));
    } else {
        w[0] = w[1] = w[2] = w[3] = 0u;
        asm("{ .reg .pred q; setp.ne.u32 q, %5, 0; @q ld.global.v4.u32 {%0, %1, %2, %3}, [%4]; }"
                     : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]) : "l"(p), "r"(pr));
    }
}

template <int SPL>
__device__ __forceinline__ void ld_floats(const float *p, bool ok, float (&v)[SPL]) {
    const uint32_t pr = ok;
#pragma unroll
    for (int h = 0; h < SPL; ++h) v[h] = 0.f;
    if constexpr (SPL == 2) {
        asm("{ .reg .pred q; setp.ne.u32 q, %3, 0; @q ld.global.v2.f32 {%0, %1}, [%2]; }"
                     : "+f"(v[0]), "+f"(v[1]) : "l"(p), "r"(pr));
    } else {
#pragma unroll
        for (int h = 0; h < SPL; h += 4)
            asm("{ .reg .pred q; setp.ne.u32 q, %5, 0; @q ld.global.v4.f32 {%0, %1, %2, %3}, [%4]; }"
                         : "+f"(v[h]), "+f"(v[h + 1]), "+f"(v[h + 2]), "+f"(v[h + 3]) : "l"(p + h), "r"(pr));
    }
}

template <int SPL>
__device__ __forceinline__ void st_floats(float *p, const float (&v)[SPL]) {
    if constexpr (SPL == 2) {
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    } else {
#pragma unroll
        for (int h = 0; h < SPL; h += 4)
            *reinterpret_cast<float4 *>(p + h) = make_float4(v[h], v[h + 1], v[h + 2], v[h + 3]);
    }
}

template <int SPL>
__device__ __forceinline__ void st_words(uint32_t *p, const uint32_t (&w)[SPL / 2]) {
    if constexpr (SPL == 2) *p = w[0];
    else if constexpr (SPL == 4) *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
    else *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ int half_of(uint32_t w, int h) { return (int16_t)(h ? (w >> 16) : (w & 0xffffu)); }

// Lane of the i-th (0-based) set bit of m; i < popc(m).
__device__ __forceinline__ int nth_set_bit(uint32_t m, int i) {
    uint32_t pos;
    asm("fns.b32 %0, %1, 0, %2;" : "=r"(pos) : "r"(m), "r"(i + 1));
    return (int)(pos & 31u);
}

// c[t - e] for 1 <= t - e < L, else 0, from a table c_s[0..kMaxL] with c_s[k] = 0 for k >= L:
// t - e is negative for susceptible agents (e = NEVER) and huge for padding (e = kPad), both
// of which clamp (as unsigned) to L, and c[0] = 0.
__device__ __forceinline__ float infect_lut(int e, const float *c_s, int t, unsigned L) {
    return c_s[min((unsigned)(t - e), L)];
}

// A group of LPR lanes holds CPL entries of its row a lane at a time (a chunk: entry i LPR + q
// is lane q's i-th).  The reverse sweep, which gathers for nearly every entry, holds at
// least eight: with one a lane and two lanes a row, a row of 22 entries was eleven rounds
// of dependent loads.  The forward keeps one: it gathers few of its entries, and the
// selection among several cost it more (53 to 65 us a day on 50k agents x 12 sets).
template <int LPR>
constexpr int chunk_per_lane() { return LPR >= 8 ? 1 : 8 / LPR; }

// Row data of one pass (one row per group), loaded a pass ahead of use: the
// lane's exposure words of its row, the row's entry range and the first chunk
// of its entries.
template <int LPR, int SPL, int CPL>
struct PassRow {
    uint32_t ew[SPL / 2];
    uint32_t p0, len;      // entries [p0, p0 + len)
    uint32_t j0[CPL];
    float w0[CPL];
};

// This lane's entries of the chunk at k0 of a row of len entries at p0 (0 past its end).
template <int LPR, int CPL>
__device__ __forceinline__ void load_chunk(const Csr &m, uint32_t p0, uint32_t len, uint32_t k0, int q,
                                           uint32_t (&j)[CPL], float (&w)[CPL]) {
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        const uint32_t k = k0 + (uint32_t)(i * LPR + q);
        j[i] = ld_cs_if(m.col + p0 + k, k < len);
        w[i] = ld_cs_if(m.w + p0 + k, k < len);
    }
}

// Loads the pass row of unit row r into pr, or an empty padding row when !ok; lane r holds the
// row bounds (rowptr of unit row r and r + 1; 0 past the unit) in rp_lo / rp_hi.  Called by all 32 lanes.
template <int LPR, int SPL, int CPL>
__device__ __forceinline__ void load_pass_row(const Csr &m, const uint32_t *ew_ptr, bool ok, uint32_t rp_lo, uint32_t rp_hi,
                                              int r, int q, PassRow<LPR, SPL, CPL> &pr) {
    pr.p0 = __shfl_sync(kFull, rp_lo, r);
    pr.len = __shfl_sync(kFull, rp_hi, r) - pr.p0;
    ld_words<SPL>(ew_ptr, ok, pr.ew);
    if (!ok) {   // no row: every set a padding one
#pragma unroll
        for (int k = 0; k < SPL / 2; ++k) pr.ew[k] = 0x80008000u;
    }
    load_chunk<LPR, CPL>(m, pr.p0, pr.len, 0u, q, pr.j0, pr.w0);
}

// V marked entries of the current chunk, taken from mm in entry order (lowest lane
// of the group first): their columns and weights broadcast from the lanes holding
// them, every lane's gathers issued before any of their values is used, then the
// sums.  Slots past the group's last marked entry carry weight 0 and load nothing.
template <int V, int LPR, int SPL, int CPL, bool KAHAN, class Raw, class Ld, class Val>
__device__ __forceinline__ void gather_batch(unsigned &mm, const uint32_t (&j)[CPL],
                                             const float (&w)[CPL], Ld &ld, Val &val,
                                             float (&sum)[SPL], float (&comp)[SPL]) {
    uint32_t jv[V];
    float wv[V];
    bool ok[V];
#pragma unroll
    for (int u = 0; u < V; ++u) {
        ok[u] = mm != 0u;
        const int src = ok[u] ? __ffs(mm) - 1 : 0;
        mm &= mm - 1u;
        uint32_t js = j[0];   // the group's lanes agree on src, so each offers its entry of that round
        float wsl = w[0];
#pragma unroll
        for (int i = 1; i < CPL; ++i)
            if (src / LPR == i) {
                js = j[i];
                wsl = w[i];
            }
        jv[u] = __shfl_sync(kFull, js, src % LPR, LPR);
        const float ws = __shfl_sync(kFull, wsl, src % LPR, LPR);
        wv[u] = ok[u] ? ws : 0.f;   // a zero weight leaves a plain sum unchanged
    }
    Raw rv[V];
#pragma unroll
    for (int u = 0; u < V; ++u) ld(jv[u], ok[u], rv[u]);
#pragma unroll
    for (int u = 0; u < V; ++u)
#pragma unroll
        for (int h = 0; h < SPL; ++h) acc_add<KAHAN>(sum[h], comp[h], wv[u], val(rv[u], h), ok[u]);
}

// For this lane's group row (entries [p0, p0 + len)), sum[h] = sum over the
// entries whose column is marked in `bits` of w * x_h(j), in entry order, where
// ld(j, ok, raw) gathers column j's values for this lane's sets (predicated by
// ok) and val(raw, h) is set h's value.  (j0, w0) are this lane's
// entries of the first chunk, loaded by the caller; each later chunk is in flight while
// the one before it is used.  A chunk's marked entries go in batches of U gathers in
// flight, and the rest (fewer than U, counted by the group with the most) in
// batches of U/2, U/4, ..., 1: where few neighbours are marked, as early in an
// epidemic, a batch no larger than needed is most of the saving.  Called by all
// 32 lanes.
template <int LPR, int SPL, int CPL, bool KAHAN, class Raw, class Ld, class Val>
__device__ __forceinline__ void group_row_sums(const Csr &m, uint32_t p0, uint32_t len,
                                               const uint32_t (&j0)[CPL],
                                               const float (&w0)[CPL],
                                               const uint32_t *__restrict__ bits, int lane, Ld ld, Val val,
                                               float (&sum)[SPL]) {
    constexpr int U = (SPL == 8) ? 4 : 8;
    const int grp = lane / LPR, q = lane % LPR;
    const unsigned gmask = (LPR == 32) ? kFull : ((1u << LPR) - 1u);
    float comp[SPL];
#pragma unroll
    for (int h = 0; h < SPL; ++h) sum[h] = comp[h] = 0.f;
    const uint32_t kmax = __reduce_max_sync(kFull, len);
    constexpr int CH = CPL * LPR;
    uint32_t jn[CPL];
    float wn[CPL];
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        jn[i] = j0[i];
        wn[i] = w0[i];
    }
    for (uint32_t k0 = 0; k0 < kmax; k0 += CH) {
        uint32_t j[CPL];
        float w[CPL];
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            j[i] = jn[i];
            w[i] = wn[i];
        }
        load_chunk<LPR, CPL>(m, p0, len, k0 + CH, q, jn, wn);
        bool mk[CPL];
#pragma unroll
        for (int i = 0; i < CPL; ++i) mk[i] = k0 + (uint32_t)(i * LPR + q) < len && marked(bits, j[i]);
        unsigned mm = 0u;   // the group's marked entries of the chunk, in entry order
#pragma unroll
        for (int i = 0; i < CPL; ++i) mm |= ((__ballot_sync(kFull, mk[i]) >> (grp * LPR)) & gmask) << (i * LPR);
        const int nmax = (int)__reduce_max_sync(kFull, (unsigned)__popc(mm));
        int i0 = 0;
        for (; i0 + U <= nmax; i0 += U) gather_batch<U, LPR, SPL, CPL, KAHAN, Raw>(mm, j, w, ld, val, sum, comp);
        const int rest = nmax - i0;   // < U, warp-uniform
        if constexpr (U >= 8)
            if (rest & 4) gather_batch<4, LPR, SPL, CPL, KAHAN, Raw>(mm, j, w, ld, val, sum, comp);
        if (rest & 2) gather_batch<2, LPR, SPL, CPL, KAHAN, Raw>(mm, j, w, ld, val, sum, comp);
        if (rest & 1) gather_batch<1, LPR, SPL, CPL, KAHAN, Raw>(mm, j, w, ld, val, sum, comp);
    }
}

// sum[h] = sum over the row's entries of w x_h(j), in entry order, with no bitmap: for
// values that are 0 where a bitmap would leave a neighbour out (the reverse sweep's
// coefficients, which are 0 from the start for rows not yet reached).  Nearly every
// neighbour counts there, so a test of each, its compaction and its round trip cost more than
// the few gathers of zeros.  U gathers a lane are in flight.  Called by all 32 lanes.
template <int LPR, int SPL, int CPL, bool KAHAN>
__device__ __forceinline__ void group_gather_sums(const Csr &m, uint32_t p0, uint32_t len,
                                                  const uint32_t (&j0)[CPL],
                                                  const float (&w0)[CPL], const float *x, int Bw,
                                                  int lane, float (&sum)[SPL]) {
    constexpr int U = (SPL == 8) ? 4 : 8;
    constexpr int CH = CPL * LPR;
    const int q = lane % LPR;
    float comp[SPL];
#pragma unroll
    for (int h = 0; h < SPL; ++h) sum[h] = comp[h] = 0.f;
    const uint32_t kmax = __reduce_max_sync(kFull, len);
    uint32_t jn[CPL];
    float wn[CPL];
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        jn[i] = j0[i];
        wn[i] = w0[i];
    }
    for (uint32_t k0 = 0; k0 < kmax; k0 += CH) {
        uint32_t j[CPL];
        float w[CPL];
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            j[i] = jn[i];
            w[i] = wn[i];
        }
        load_chunk<LPR, CPL>(m, p0, len, k0 + CH, q, jn, wn);
#pragma unroll
        for (int u0 = 0; u0 < CH; u0 += U) {
            if (k0 + (uint32_t)u0 >= kmax) break;
            float rv[U][SPL];
            float wv[U];
            bool ok[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = u0 + u;   // entry c of the chunk: lane c % LPR's (c / LPR)-th
                ok[u] = k0 + (uint32_t)c < len;
                const uint32_t jv = __shfl_sync(kFull, j[c / LPR], c % LPR, LPR);
                wv[u] = __shfl_sync(kFull, w[c / LPR], c % LPR, LPR);
                ld_floats<SPL>(x + (size_t)jv * Bw, ok[u], rv[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int h = 0; h < SPL; ++h) acc_add<KAHAN>(sum[h], comp[h], wv[u], rv[u][h], ok[u]);
        }
    }
}

// Whether any lane of each group voted, packed as one bit per group.
template <int LPR>
__device__ __forceinline__ uint32_t group_bits(unsigned ballot) {
    constexpr int RPW = 32 / LPR;
    const unsigned gmask = (LPR == 32) ? kFull : ((1u << LPR) - 1u);
    uint32_t part = 0u;
#pragma unroll
    for (int gi = 0; gi < RPW; ++gi) part |= (((ballot >> (gi * LPR)) & gmask) != 0u ? 1u : 0u) << gi;
    return part;
}

// Sum a per-lane value over the groups of the warp (lanes with the same q hold the same sets).
template <int LPR>
__device__ __forceinline__ int group_reduce(int v) {
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

template <int SPL>
struct EWords {
    uint32_t w[SPL / 2];
};

template <class K>
int blocks_of(K kernel) {
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, kBlock, 0);
    return blocks > 0 ? blocks : 1;
}

// The (Bp, SPL) pairs built: SPL in {2, 4, 8} with Bp / SPL lanes per row (1..32).
#define GABM_BATCH_CONFIGS(X) \
    X(2, 2)                   \
    X(4, 2) X(4, 4)           \
    X(8, 2) X(8, 4) X(8, 8)   \
    X(16, 2) X(16, 4) X(16, 8) \
    X(32, 2) X(32, 4) X(32, 8) \
    X(64, 2) X(64, 4) X(64, 8)

}  // namespace

}  // namespace gabm
