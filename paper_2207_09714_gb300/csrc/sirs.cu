// sirs.cu -- forward and reverse day kernels of SIRS reinfection (see sirs.cuh).
//
// Each warp holds one 32-row tile at a time.  The sums
// are those of the base model's kernels -- the same row sums over the same SELL entries,
// the same fused multiply-adds in the same order for G -- so with nobody returning
// within the horizon the results are bitwise the base model's.
#include "sirs.cuh"
#include "rowsum.cuh"

namespace gabm {

namespace {

__device__ __forceinline__ void flush_counts(int32_t *counts, int32_t *newRM, int ldP, int g, int t, int cS, int cE,
                                             int cI, int cR, int cN, int lane) {
    cS = __reduce_add_sync(0xffffffffu, cS);
    cE = __reduce_add_sync(0xffffffffu, cE);
    cI = __reduce_add_sync(0xffffffffu, cI);
    cR = __reduce_add_sync(0xffffffffu, cR);
    cN = __reduce_add_sync(0xffffffffu, cN);
    if (lane == 0) {
        int32_t *cp = counts + ((size_t)g * ldP + t) * 4;
        if (cS) atomicAdd(cp + 0, cS);
        if (cE) atomicAdd(cp + 1, cE);
        if (cI) atomicAdd(cp + 2, cI);
        if (cR) atomicAdd(cp + 3, cR);
        if (cN) atomicAdd(newRM + (size_t)g * ldP + t, cN);
    }
}

// The history of every row starts with its state after seeding (a seed's exposure day).
__global__ void k_sirs_hist_init(const int16_t *e, int64_t n_rows, int H, int16_t *hist, uint16_t *cnt) {
    for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < n_rows;
         row += (int64_t)gridDim.x * blockDim.x) {
        const int ei = e[row];
        const bool exposed = ei != kNever && ei != kPad;
        cnt[row] = exposed ? 1 : 0;
        if (exposed) hist[row * H] = (int16_t)ei;
    }
}

// Day t: rows susceptible on day t (never exposed, or at least `cycle` days past their
// last exposure) draw; an exposure is appended to the row's history.  Each block takes a
// contiguous range of tiles (neighbours stay in its SM's L1), each warp's next tile is
// read one tile ahead, and a susceptible row with no infectious in-neighbour (flag_cur)
// reads no entries: its lambda is 0 exactly.
__global__ void __launch_bounds__(kBlock, 3) k_fwd_day_sirs(SirsFwdArgs a) {
    __shared__ float c_s[kMaxL];
    __shared__ float rs_s[kBlock / 32][kAges];   // R_t S_a of the warp's graph
    float inv_D = 0.f;
    pdl_trigger();
    if (threadIdx.x < kMaxL) c_s[threadIdx.x] = a.c[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int t = a.t, L = a.L, ntiles = a.ntiles;
    const int16_t *e = a.e;
    // neighbours infectious today contribute: those whose last exposure day lies in the window
    // (one exposed again during the day gives t - e = 0, and was out of it before)
    auto contrib = [&](uint32_t j, float w, bool valid, float &out, bool &take) {
        const int k = t - ld_if(e + j, valid, kNever);
        take = valid && (unsigned)(k - 1) < (unsigned)(L - 1);
        out = take ? w * c_s[k] : 0.f;
    };
    int cur_g = -1, cS = 0, cE = 0, cI = 0, cR = 0, cN = 0;
    BlockTiles disp;
    disp.init(ntiles, lane);
    TileRows cur, nxt;
    load_tile_layout(a.m, a.gr.tile_graph, ntiles, disp.get(), lane, cur);
    load_tile_layout(a.m, a.gr.tile_graph, ntiles, disp.get(), lane, nxt);
    pdl_wait();
    load_tile_state(e, ntiles, lane, cur, a.flag_cur);
    load_tile_state(e, ntiles, lane, nxt, a.flag_cur);
    while (cur.tile < ntiles) {
        TileRows nn;
        load_tile_rows(a.m, e, a.gr.tile_graph, ntiles, disp.get(), lane, nn, a.flag_cur);
        const int g = cur.g, tile = cur.tile;
        if (g != cur_g) {
            if (cur_g >= 0) flush_counts(a.counts, a.newRM, a.ldP, cur_g, t, cS, cE, cI, cR, cN, lane);
            cur_g = g;
            cS = cE = cI = cR = cN = 0;
            const float RS_ld = lane < kAges ? a.R[(size_t)g * a.ldP + t] * a.S[g * kAges + lane] : 0.f;
            inv_D = a.gr.inv_Dbar[g];
            __syncwarp();
            if (lane < kAges) rs_s[threadIdx.x >> 5][lane] = RS_ld;
            __syncwarp();
        }
        const int row = tile * kTile + lane;
        const int ei = cur.e;
        const bool agent = ei != kPad;
        const int k = t - ei;
        const bool isS = agent && (ei == kNever || k >= a.cycle);
        if (agent && !isS) {
            if (k < a.tau_EI) ++cE; else if (k < L) ++cI; else ++cR;
            cN += (k == L);
        }
        cS += isS;
        const bool act = isS && cur.flag;
        const int age_ld = act ? (int)a.age[row] : 0;   // ahead of the sums
        const uint32_t id_ld = act ? caller_id(a.gr, row, g) : 0u;
        float sum = 0.f;
        const unsigned amask = __ballot_sync(0xffffffffu, act);
        if (a.flag_cur && __popc(amask) <= GABM_COOP_ROWS) {   // few summing rows: warp-wide, together
            if (amask) sum = few_row_sums(a.m, cur.p0, cur.len, amask, lane, contrib);
        } else {
            sum = exposed_sum(a.m, cur.p0, cur.len, act, lane, e, c_s, t, L);
        }
        if (cur.len & kLongBit) sum = a.long_sum[cur.len & ~kLongBit];
        int e_next = ei;
        if (act) {
            const float Lam = sum * inv_D;
            const float lam = rs_s[threadIdx.x >> 5][age_ld] * Lam;
            const float p = -expm1f(-lam);
            const uint32_t id = id_ld;
            const float u = uniform_from_word(philox_word(a.seed, id, (uint32_t)t, (uint32_t)g, 0u));
            if (u < p) {
                a.e[row] = (int16_t)t;
                e_next = t;
                // H covers the horizon (exposures are at least `cycle` days apart), so ci < H;
                // the count stops at H all the same, keeping every history access in bounds
                const int ci = a.cnt[row];
                if (ci < a.H) {
                    a.hist[(size_t)row * a.H + ci] = (int16_t)t;
                    a.cnt[row] = (uint16_t)(ci + 1);
                }
            }
            a.lam_out[row] = Lam;
        } else if (isS) {
            a.lam_out[row] = 0.f;
        }
        const int kn = t + 1 - e_next;
        const bool inf = (unsigned)(kn - 1) < (unsigned)(L - 1);
        const unsigned inf_next = __ballot_sync(0xffffffffu, inf);
        if (lane == 0) a.bits_next[tile] = inf_next;
        if (a.flag_cur) {   // tomorrow's flags: the out-neighbours of tomorrow's infectious rows
            push_flags(a.m, a.m_out, cur, lane, inf, a.flag_next);
            a.flag_clear[row] = 0;
        }
        cur = nxt;
        nxt = nn;
    }
    if (cur_g >= 0) flush_counts(a.counts, a.newRM, a.ldP, cur_g, t, cS, cE, cI, cR, cN, lane);
}

// The next tile's row data for the reverse sweep (one tile ahead of use).
__device__ __forceinline__ TileRows nn_next(const SirsBwdArgs &a, BlockTiles &disp, int lane) {
    TileRows nn;
    load_tile_rows(a.m, a.E, a.gr.tile_graph, a.ntiles, disp.get(), lane, nn);
    return nn;
}

// Reverse day t: gx(t+1) of every agent into the ring, then for rows susceptible on
// day t the adjoint of the draw, with the return terms B(t+1) and B(t+cycle) read from
// the G stored at the row's later exposures.
__global__ void __launch_bounds__(kBlock, 3) k_bwd_day_sirs(SirsBwdArgs a) {
    pdl_trigger();
    constexpr int NW = kBlock / 32;
    constexpr int RB = 8;   // ring slots loaded together
    __shared__ float cf_s[NW][kMaxL];    // c[k] 2^(sigma(t+k) - sigma(t)) of the days that carry adjoint,
    __shared__ int off_s[NW][kMaxL];     // and their slots' offsets, k ascending from 2
    __shared__ float rs_s[NW][kAges];    // R_t S_a of the warp's graph
    __shared__ __align__(16) float bin_s[NW][kBinWords];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int i = lane; i < kBinWords; i += 32) bin_s[wib][i] = 0.f;
    __syncwarp();
    const int t = a.t, T = a.T, L = a.L, C = a.cycle, H = a.H;
    const int slot_floats = (L - 1) * kTile;
    float cf1 = 0.f, gtail = 0.f, inv_D = 0.f;
    int nterm = 0, sig_t = 0;
    const int32_t *sg = nullptr;
    int cur_g = -1, cN = 0;
    unsigned emax_w = 0u, live_k = 0u;   // live_k bit k: day t + k carries adjoint
    bool rnz_w = false;
    BlockTiles disp;
    disp.init(a.ntiles, lane);
    TileRows cur, nxt;
    load_tile_rows(a.m, a.E, a.gr.tile_graph, a.ntiles, disp.get(), lane, cur);
    load_tile_rows(a.m, a.E, a.gr.tile_graph, a.ntiles, disp.get(), lane, nxt);
    pdl_wait();   // the layout, the final state and the histories are not written by the sweep
    for (; cur.tile < a.ntiles; cur = nxt, nxt = nn_next(a, disp, lane)) {
        const int tile = cur.tile;
        const int g = cur.g;
        if (g != cur_g) {
            if (cur_g >= 0) {
                const int sN = __reduce_add_sync(0xffffffffu, cN);
                if (lane == 0 && sN) atomicAdd(a.newRM + (size_t)cur_g * a.ldP + t, sN);
                flush_emax(a.emax + (size_t)cur_g * a.ld_sig + t, emax_w);
                flush_rnz(a.rnz + (size_t)cur_g * a.ld_sig + t, rnz_w);
                emax_w = 0u;
                rnz_w = false;
            }
            cur_g = g;
            cN = 0;
            live_k = carries_adjoint(a.rnz + (size_t)g * a.ld_sig, t, T, L);
            sg = a.sig + (size_t)g * a.ld_sig;
            sig_t = next_sigma(sg[t + 1], a.emax[(size_t)g * a.ld_sig + t + 1]);
            if (lane == 0 && tile * kTile == a.gr.row0[g]) a.sig[(size_t)g * a.ld_sig + t] = sig_t;
            const float cf = ((live_k >> lane) & 1u) ? a.c[lane] * exp2i(sg[t + lane] - sig_t) : 0.f;
            cf1 = __shfl_sync(0xffffffffu, cf, 1);
            const unsigned tm = live_k & ~3u;
            nterm = __popc(tm);
            __syncwarp();
            if ((tm >> lane) & 1u) {
                const int i = __popc(tm & ((1u << lane) - 1u));
                off_s[wib][i] = a.ring_slot[lane] * kTile;
                cf_s[wib][i] = cf;
            }
            const size_t pg = (size_t)g * a.ldP;
            if (lane < kAges) rs_s[wib][lane] = a.R[pg + t] * a.S[g * kAges + lane];
            inv_D = a.gr.inv_Dbar[g];
            gtail = (t + L < T) ? a.m_t[pg + t + L] * (float)a.gD[pg + t + L] * exp2i(-sig_t) : 0.f;
            __syncwarp();
        }

        const int row = tile * kTile + lane;
        const bool agent = cur.e != kPad;
        const int n_e = min((int)a.cnt[row], H);
        const int16_t *hr = a.hist + (size_t)row * H;
        int j_t = 0;   // exposures before day t
        while (j_t < n_e && hr[j_t] < t) ++j_t;
        const bool y = j_t < n_e && hr[j_t] == t;
        const int e_t = j_t > 0 ? hr[j_t - 1] : kNever;
        const bool isS = agent && (e_t == kNever || t - e_t >= C);
        cN += (agent && e_t != kNever && t - e_t == L);

        // gx(t+1) is used by the G of the row's susceptible days in [t + 2 - L, t]; a row
        // with none lies, the whole window, inside one exposure's stretch (e, e + C) of not
        // being susceptible, e in [t - C + 1, lo - 1], and skips the gather
        const int lo = max(0, t + 2 - L);
        bool covered = false;
        for (int j = 0; j < j_t; ++j) covered |= (hr[j] >= t - C + 1 && hr[j] <= lo - 1);
        const bool act = (live_k & 2u) && agent && !covered;
        // the row loads that do not depend on the sum go out before it
        const float Lam = isS ? a.lam_t[row] : 0.f;
        const int ai = isS ? (int)a.age[row] : 0;
        float gx1 = gather_sum(a.m, cur.p0, cur.len, act, lane, a.r_next);
        if ((cur.len & kLongBit) && act) gx1 = a.long_gx[cur.len & ~kLongBit];
        float *ring = a.ring + (size_t)tile * slot_floats + lane;
        if (act) ring[a.ring_slot[1] * kTile] = gx1;

        float v = 0.f, rc = 0.f;
        if (isS) {
            // B(t'): G at the row's first exposure on or after day t' (0 if none), at day t's scale
            auto B_at = [&](int tp) -> float {
                int j = j_t;
                while (j < n_e && hr[j] < tp) ++j;
                return j < n_e ? a.Gh[(size_t)row * H + j] * exp2i(sg[hr[j]] - sig_t) : 0.f;
            };
            // the day's own terms: the death term and the infectiousness it would cause
            float loc = __fmaf_rn(cf1, gx1, gtail);
            for (int j0 = 0; j0 < nterm; j0 += RB) {
                float rv[RB];
#pragma unroll
                for (int u = 0; u < RB; ++u)
                    if (j0 + u < nterm) rv[u] = ring[off_s[wib][j0 + u]];
#pragma unroll
                for (int u = 0; u < RB; ++u)
                    if (j0 + u < nterm) loc = __fmaf_rn(cf_s[wib][j0 + u], rv[u], loc);
            }
            const float G = loc + B_at(t + C);
            // dL/dy = G - B(t+1).  With t' the row's first exposure after t, B(t+1) = G(t'),
            // and B(t+C) = B(t'+C) when t' < t+C (the next exposure after t' is at least
            // t'+C), while B(t+C) = G(t') when t' >= t+C: so dL/dy = loc - loc(t') or loc.
            // Formed this way the return terms cancel exactly instead of in fp32, where on
            // short cycles they dwarf the difference.
            const int jn = y ? j_t + 1 : j_t;
            float dy = loc;
            if (jn < n_e && hr[jn] < t + C) dy = loc - a.Lh[(size_t)row * H + jn] * exp2i(sg[hr[jn]] - sig_t);
            if (y) {
                a.Gh[(size_t)row * H + j_t] = G;
                a.Lh[(size_t)row * H + j_t] = loc;
            }
            float stored = fmaxf(fabsf(G), fabsf(loc));
            const float RS = rs_s[wib][ai];
            const float lam = RS * Lam;
            float glam = dy;   // dy = 0 and lambda finite: the product with dy/dlambda >= 0 is dy itself
            if (!(dy == 0.f && lam >= 0.f && lam < __int_as_float(0x7f800000))) {
                const float q = expf(-lam);
                const float p = -expm1f(-lam);
                const uint32_t id = caller_id(a.gr, row, g);
                const float u = uniform_from_word(philox_word(a.seed, id, (uint32_t)t, (uint32_t)g, 0u));
                const float den = __fmaf_rn(p, 1.f - u, q * u);
                const float dydl = (u * (1.f - u)) * q / (den * den);
                glam = dy * dydl;
            }
            rc = RS * glam * inv_D;
            v = glam * Lam;
            stored = fmaxf(stored, fabsf(rc));
            rnz_w |= !(rc == 0.f);
            emax_w = max(emax_w, (unsigned)(float_exponent(stored) + 128));
        }
        a.r_cur[row] = rc;   // 0 for rows not susceptible today (r of a later day may sit there)

        float mine = 0.f;   // lanes 2b, 2b + 1: bin b (the base kernel's tree)
        if (__any_sync(0xffffffffu, !(v == 0.f))) mine = warp_bin_sums(v, ai, lane, bin_s[wib]);
        if (!(lane & 1) && (lane >> 1) < kAges) a.P_t[(size_t)tile * kAges + (lane >> 1)] = mine;
    }
    if (cur_g >= 0) {
        const int sN = __reduce_add_sync(0xffffffffu, cN);
        if (lane == 0 && sN) atomicAdd(a.newRM + (size_t)cur_g * a.ldP + t, sN);
        flush_emax(a.emax + (size_t)cur_g * a.ld_sig + t, emax_w);
        flush_rnz(a.rnz + (size_t)cur_g * a.ld_sig + t, rnz_w);
    }
}

}  // namespace

cudaError_t launch_sirs_hist_init(const int16_t *e, int64_t n_rows, int H, int16_t *hist, uint16_t *cnt,
                                  cudaStream_t s) {
    const int grid = (int)std::min<int64_t>((n_rows + 255) / 256, 65535);
    k_sirs_hist_init<<<grid > 0 ? grid : 1, 256, 0, s>>>(e, n_rows, H, hist, cnt);
    return cudaGetLastError();
}

cudaError_t launch_fwd_day_sirs(const SirsFwdArgs &a, int grid, bool overlap, cudaStream_t s) {
    return launch_day(k_fwd_day_sirs, grid, kBlock, 0, s, overlap, a);
}

cudaError_t launch_bwd_day_sirs(const SirsBwdArgs &a, int grid, bool overlap, cudaStream_t s) {
    return launch_day(k_bwd_day_sirs, grid, kBlock, 0, s, overlap, a);
}

int occupancy_sirs(bool backward) {
    int blocks = 0;
    if (backward) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_bwd_day_sirs, kBlock, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_fwd_day_sirs, kBlock, 0);
    return blocks > 0 ? blocks : 1;
}

}  // namespace gabm
