// backward.cu -- hand-written straight-through adjoint of the day loop (App. B).
//
// The reverse sweep runs one launch per day t = T-1 .. 0.  Launch t fuses two
// steps that touch the same rows:
//   (1) the transpose gather of day t+1: gx_i(t+1) = sum_{j in out(i)} w_ij r_j(t+1),
//       a pull over the source-sorted CSR (the forward CSR itself when the
//       weights are symmetric), so no atomics; written to a ring of the last
//       L-1 days;
//   (2) for every agent susceptible on day t, the adjoint of its draw:
//       G_i(t) = m_{t+L} gD_{t+L} + sum_{k=1}^{L-1} c[k] gx_i(t+k),
//       dL/dy = G (t = E_i or never infected) or G - A_i (t < E_i), A_i = G_i(E_i),
//       gl = dL/dy * dy_soft/dlambda (Gumbel-softmax, tau = 1, straight-through),
//       r_i(t) = R_t S[a_i] gl / Dbar and per-tile, per-age sums of gl * Lam.
// lambda_i(t) comes from the forward's store or is recomputed from the final
// exposure days E (no reinfection, A3/A4 of App. A, so E determines every
// day's state and no checkpoints are needed): in the same pass when in- and
// out-edges coincide, else by k_lam_day over the in-edges first.  The next tile's
// row data are loaded while the current tile is worked on.  Days no adjoint has
// reached yet (rnz) gather nothing.
#include "gabm_internal.cuh"
#include "rowsum.cuh"

namespace gabm {

namespace {

// Adds this tile's share of the table adjoint dL/dc[k] = sum_j gx_j(E_j + k): every lane
// with `has` holds gx of its row for the day that is k = kd days after the row's
// exposure, at scale 2^sigma of that day.  Rows with equal k are summed over the warp
// (fp32, fixed tree), then added in FP64 to the tile's accumulator, whose only writer
// is the warp holding the tile (days are sequential launches).  Called by all 32 lanes.
__device__ __forceinline__ void dc_accumulate(double *dc_tile, int tile, bool has, int kd, float gx, int sigma,
                                              int lane) {
    unsigned pend = __ballot_sync(0xffffffffu, has);
    if (!pend) return;
    // lane k keeps the sum for k (k < L <= 32), so the read-modify-writes of all k go out together
    float mine = 0.f;
    bool touched = false;
    while (pend) {
        const int k0 = __shfl_sync(0xffffffffu, kd, __ffs(pend) - 1);
        const bool sel = has && kd == k0;
        float v = sel ? gx : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == k0) {
            mine = v;
            touched = true;
        }
        pend &= ~__ballot_sync(0xffffffffu, sel);
    }
    if (touched) dc_tile[(size_t)tile * kMaxL + lane] += (double)mine * ldexp(1.0, sigma);
}

// One term of G_i(t): the ring slot of day t + k (an offset within the tile's slots) and
// c[k] 2^(sigma(t+k) - sigma(t)).  Only days that carry adjoint have one.
struct RingTerm {
    int off;
    float cf;
};
#ifndef GABM_RING_BATCH
#define GABM_RING_BATCH 10
#endif

// DC: accumulate the table adjoint (a.dc_tile); a separate instance, so the plain sweep
// carries none of its code.
// MINB blocks an SM, GP pairs of entries a lane ahead of their use (see bwd_kernel).
// EXIT = kExitFate (sampled R/M split, store policy): G of an exposure today takes the
// fate it would draw (window L_R or L_M; the death term gD_{t+L_M} only if M-fated), and
// the rows exposed today add H dphi/dm to day t + tau_EI's dL/dm, H = dL/dphi = sum over
// the days between the two exits of +-c[k] gx(t+k) plus gD_{t+L_M}.  Rows exposed before
// day 0 keep their gx in the ring for k_fate_seeds.
// EXIT = kExitDur (stochastic I-stage durations, store policy): G of an exposure today
// sums over the window L_i it would draw and takes the death term m gD of its own exit
// day; the exits recounted for dm are at each row's drawn L_i.
template <int MODE, bool DC, int EXIT = kExitBase, int NT = kBlock, int MINB = 3,
          int GP = kGP>
__global__ void __launch_bounds__(NT, MINB)
    k_bwd_day(BwdDayArgs a) {
    constexpr bool FATE = EXIT == kExitFate;
    constexpr bool DUR = EXIT == kExitDur;
    constexpr bool SOFT = MODE == kBwdSoft;
    constexpr int RB = GABM_RING_BATCH;   // ring slots loaded together in the epilogue
    constexpr int NW = NT / 32;
    __shared__ float c_s[kMaxL];
    __shared__ int32_t red_s[NW][4];
    __shared__ RingTerm term_s[NW][kMaxL];        // the warp's graph's ring terms, k ascending
    __shared__ int term_k[FATE || DUR ? NW : 1][kMaxL];   // their k
    __shared__ float rs_s[NW][kAges];             // R_t S_a of the warp's graph
    __shared__ __align__(16) float bin_s[NW][kBinWords];
    __shared__ double F_s[kMaxL];
    pdl_trigger();
    if (threadIdx.x < kMaxL) {
        c_s[threadIdx.x] = a.c[threadIdx.x];
        if (DUR) F_s[threadIdx.x] = a.dur.F[threadIdx.x];
    }
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int i = lane; i < kBinWords; i += 32) bin_s[wib][i] = 0.f;
    __syncthreads();

    const int t = a.t, T = a.T, L = a.L, ntiles = a.ntiles;
    const int32_t *sg = nullptr;   // scale exponents of the current graph
    int sig_t = 0;                 // sigma(t) of the current graph
    unsigned emax_w = 0u;          // largest exponent stored by this warp (+128)
    bool rnz_w = false;            // this lane stored an r other than 0
    unsigned live_k = 0u;          // bit k: day t + k carries adjoint (its gx is not all 0)
    int nterm = 0;                 // ring terms, k >= 2
    float gtail = 0.f;             // m_{t+L} gD_{t+L} at day t's scale
    float cf1 = 0.f, f1 = 0.f;     // the k = 1 term's factor, and its scale alone
    float inv_D = 0.f;
    const int16_t *E = a.E;
    const int slot_floats = (L - 1) * kTile;

    // Which of a tile's rows gather gx(t+1).  Table adjoint: rows infectious on day t+1 (k =
    // t+1-E in [1, L-1]) add gx(t+1) to dc[k]; the non-seed ones gather anyway, the seeds only
    // for this.  R/M split: rows exposed before day 0 keep gx while day t+1 is inside their
    // window.  Soft relaxation: every agent carries susceptible mass and draws every day.
    auto needs = [&](int Ei) {
        const bool agent = Ei != kPad, never = Ei == kNever, gather = (live_k & 2u) != 0u;
        if (SOFT) return gather && agent;
        return gather && ((agent && (never || (Ei >= 0 && Ei >= t + 2 - L))) ||
                          (FATE && agent && !never && Ei < 0 && t + 1 - Ei < L));
    };
    auto dc_row_of = [&](int Ei) {
        const int kd = t + 1 - Ei;
        return DC && !SOFT && (live_k & 2u) && Ei != kPad && Ei != kNever && kd >= 1 && kd <= L - 1;
    };

    int cur_g = -1, cN = 0;
    BlockTiles disp;
    disp.init(ntiles, lane);
    TileRows cur, nxt;
    load_tile_rows(a.m, E, a.gr.tile_graph, ntiles, disp.get(), lane, cur);
    uint4 ea[GP];
#pragma unroll
    for (int u = 0; u < GP; ++u) ea[u] = make_uint4(0u, 0u, 0u, 0u);
    // the first tile's first pairs before the wait, as if its rows gather (they do, but for
    // the last days of a horizon); the final exposure days are not written by the sweep
    live_k = 2u;
    {
        const TileSpan sp = tile_span(a.m, cur.p0, cur.len, needs(cur.e) || dc_row_of(cur.e), lane);
        load_pairs(sp.row, 0u, sp.lim, ea);
    }
    bool have = true;   // ea holds the current tile's first pairs
    // the first graph's scalars that no launch of the sweep writes
    float RS_ld = 0.f, gt_ld = 0.f;
    int row0_ld = 0;
    auto load_scalars = [&](int g) {
        const size_t pg = (size_t)g * a.ldP;
        RS_ld = lane < kAges ? a.R[pg + t] * a.S[g * kAges + lane] : 0.f;
        const int td = t + (FATE ? a.fate.L_M : L);   // the day today's exposures die on
        gt_ld = td < T ? (FATE ? 1.f : a.m_t[pg + td]) * (float)a.gD[pg + td] : 0.f;
        inv_D = a.gr.inv_Dbar[g];
        row0_ld = a.gr.row0[g];
    };
    if (cur.tile < ntiles) load_scalars(cur.g);
    pdl_wait();
    while (cur.tile < ntiles) {
        load_tile_rows(a.m, E, a.gr.tile_graph, ntiles, disp.get(), lane, nxt);   // a tile ahead of use

        const int g = cur.g, tile = cur.tile, Ei = cur.e;
        if (g != cur_g) {
            if (cur_g >= 0) {
                const int sN = __reduce_add_sync(0xffffffffu, cN);
                if (lane == 0 && sN) atomicAdd(a.newRM + (size_t)cur_g * a.ldP + t, sN);
                flush_emax(a.emax + (size_t)cur_g * a.ld_sig + t, emax_w);
                flush_rnz(a.rnz + (size_t)cur_g * a.ld_sig + t, rnz_w);
                emax_w = 0u;
                rnz_w = false;
            }
            const bool first = cur_g < 0;
            // every load of this block goes out before any is used
            const size_t ps = (size_t)g * a.ld_sig;
            sg = a.sig + ps;
            const bool in = lane >= 1 && lane < L && t + lane < T;
            const int32_t nz_ld = in ? a.rnz[ps + t + lane] : 0;
            const int32_t sg_ld = (lane >= 1 && lane < L && t + lane <= T) ? sg[t + lane] : 0;
            const int32_t em_ld = a.emax[ps + t + 1];
            if (!first) load_scalars(g);
            live_k = __ballot_sync(0xffffffffu, nz_ld != 0);   // days that carry adjoint (flush_rnz)
            // this day's scale for graph g (every warp computes the same value; the warp
            // holding the graph's first tile records it)
            sig_t = next_sigma(__shfl_sync(0xffffffffu, sg_ld, 1), em_ld);
            if (lane == 0 && tile * kTile == row0_ld) a.sig[ps + t] = sig_t;
            // c[k] 2^(sigma(t+k) - sigma(t)): the power of two moves no bit of the product
            const float fac = (lane >= 1 && lane < L && t + lane <= T) ? exp2i(sg_ld - sig_t) : 0.f;
            f1 = __shfl_sync(0xffffffffu, fac, 1);
            cf1 = (live_k & 2u) ? c_s[1] * f1 : 0.f;
            const unsigned tm = live_k & ~3u;
            nterm = __popc(tm);
            if ((tm >> lane) & 1u) {
                const int i = __popc(tm & ((1u << lane) - 1u));
                term_s[wib][i].off = a.ring_slot[lane] * kTile;
                term_s[wib][i].cf = c_s[lane] * fac;
                if (FATE || DUR) term_k[wib][i] = lane;
            }
            if (lane < kAges) rs_s[wib][lane] = RS_ld;
            gtail = gt_ld * exp2i(-sig_t);   // R/M split: deaths are counted, dL/d(one M entry on day t + L_M)
            __syncwarp();
            cur_g = g;
            cN = 0;
            if (!first) have = false;
        }
        const int row = tile * kTile + lane;
        const bool agent = (Ei != kPad);
        const bool never = (Ei == kNever);
        const bool live = agent && (never || Ei >= 0);           // seeds are constants
        const bool isS = SOFT ? agent : live && (never || Ei >= t);
        const bool gather = (live_k & 2u) != 0u;   // else gx(t+1) = 0 for every row
        const bool needA = needs(Ei), dc_row = dc_row_of(Ei);
        if constexpr (DUR) {
            // exits at the row's drawn L_i (its first possible day is tau_EI + 1)
            const int k = t - Ei;
            if (agent && !never && k > a.tau_EI && k <= L)
                cN += (k == dur_exit(a.dur, F_s, caller_id(a.gr, row, g), Ei, g));
        } else if (!SOFT) {
            cN += (agent && !never && t - Ei == L);
        }

        // the row loads that do not depend on the sums go out before them, so that their
        // latency overlaps the entry stream; A was stored on day E_i (soft: dL/ds on day
        // t+1) at that day's scale
        const bool readA = isS && (SOFT || (!never && Ei != t));
        const float A_ld = readA ? a.A[row] : 0.f;
        // (sigma grows towards day 0, so sigma(t) = 0 means that it is 0 on every later day)
        const int sgE_ld = (readA && !SOFT && sig_t != 0) ? sg[Ei] : 0;
        float Lam = 0.f;
        if constexpr (MODE != kBwdFused) Lam = isS ? a.lam_t[row] : 0.f;
        const int ai = isS ? (int)a.age[row] : 0;
        const bool draws = live_k != 0u || gtail != 0.f || FATE || DUR || SOFT;   // some dy is not 0
        uint32_t id = (isS && draws) ? caller_id(a.gr, row, g) : 0u;

        float gx_mine;
        {
            const TileSpan sp = tile_span(a.m, cur.p0, cur.len, needA || dc_row, lane);
            if (!have) load_pairs(sp.row, 0u, sp.lim, ea);
            if constexpr (MODE == kBwdFused) {   // lambda from the final exposure days, the forward's sum
                if (gather) {                    // rows susceptible today are among those that gather
                    gx_mine = gather_and_exposed_sum(sp, a.r_next, isS, E, c_s, t, L, ea, Lam);
                } else {
                    gx_mine = 0.f;
                    Lam = exposed_sum<2>(a.m, cur.p0, cur.len, isS, lane, E, c_s, t, L);
                }
                if (cur.len & kLongBit) Lam = a.long_lam[cur.len & ~kLongBit];
                Lam *= inv_D;
            } else {
                gx_mine = gather_sum(sp, a.r_next, ea);
            }
        }
        if ((cur.len & kLongBit) && gather) gx_mine = a.long_gx[cur.len & ~kLongBit];
        if (a.self_q && gather) gx_mine = __fmaf_rn(-a.self_q[row], a.self_r[row], gx_mine);
        // the next tile's first pairs are in flight during this tile's epilogue
        have = nxt.tile < ntiles && nxt.g == cur_g;
        if (have) {
            const TileSpan sp = tile_span(a.m, nxt.p0, nxt.len, needs(nxt.e) || dc_row_of(nxt.e), lane);
            load_pairs(sp.row, 0u, sp.lim, ea);
        }

        float *ring = a.ring + (size_t)tile * slot_floats + lane;
        if (needA) ring[a.ring_slot[1] * kTile] = gx_mine;
        if constexpr (DC && !SOFT) dc_accumulate(a.dc_tile, tile, dc_row, t + 1 - Ei, gx_mine, sg[t + 1], lane);
        if constexpr (DC && SOFT) {
            // soft: every agent's mass exposed k days before t+1 counts, n_j(d) = s_j(d) y_j(d)
            // for d >= 0 and the seeds' unit mass on their day E_j < 0 (lane k keeps k's sum)
            const bool on = gather && agent;
            if (__any_sync(0xffffffffu, on)) {
                float mine = 0.f;
                for (int k = 1; k < L; ++k) {
                    const int d = t + 1 - k;
                    float nk = 0.f;
                    if (on)
                        nk = (d >= 0) ? a.s_hist[(size_t)d * a.hist_stride + row] * a.y_hist[(size_t)d * a.hist_stride + row]
                                      : (Ei == d ? 1.f : 0.f);
                    float v = nk * gx_mine;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    if (lane == k) mine = v;
                }
                if (lane >= 1 && lane < L && mine != 0.f)
                    a.dc_tile[(size_t)tile * kMaxL + lane] += (double)mine * ldexp(1.0, sg[t + 1]);
            }
        }

        float v = 0.f, pm = 0.f;
        if (isS) {
            float Apre = 0.f;
            if (readA) Apre = A_ld * (SOFT ? f1 : exp2i(sgE_ld - sig_t));
            // R/M split: the fate an exposure today would draw on day t + tau_EI
            bool phi = false;
            float vf = 0.5f;
            int Lx = L;
            if constexpr (FATE) {
                if (t + a.tau_EI < T) {
                    vf = fate_uniform(a.fate, id, t + a.tau_EI, g);
                    phi = vf < a.m_t[(size_t)g * a.ldP + t + a.tau_EI];
                }
                Lx = phi ? a.fate.L_M : a.fate.L_R;
            }
            const int Lmin = FATE ? min(a.fate.L_R, a.fate.L_M) : L;
            const float sgn = (FATE && a.fate.L_M > a.fate.L_R) ? 1.f : -1.f;
            if constexpr (DUR) {
                // the window an exposure today would draw, and the death term of its exit day
                Lx = dur_exit(a.dur, F_s, id, t, g);
                const size_t pg = (size_t)g * a.ldP;
                gtail = (t + Lx < T) ? a.m_t[pg + t + Lx] * (float)a.gD[pg + t + Lx] * exp2i(-sig_t) : 0.f;
            }
            float G = (FATE && !phi) ? 0.f : gtail;
            float H = gtail;
            G = __fmaf_rn(cf1, gx_mine, G);
            for (int j0 = 0; j0 < nterm; j0 += RB) {
                float rv[RB];
#pragma unroll
                for (int u = 0; u < RB; ++u)
                    if (j0 + u < nterm) rv[u] = ring[term_s[wib][j0 + u].off];
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    if (j0 + u < nterm) {
                        const float cf = term_s[wib][j0 + u].cf;
                        if constexpr (FATE || DUR) {
                            const int k = term_k[wib][j0 + u];
                            if (k < Lx) G = __fmaf_rn(cf, rv[u], G);
                            if (FATE && k >= Lmin) H = __fmaf_rn(sgn * cf, rv[u], H);
                        } else {
                            G = __fmaf_rn(cf, rv[u], G);
                        }
                    }
                }
            }
            if constexpr (FATE) {
                // the fate draw of today's exposure: dphi_soft/dm = v (1-v) / (m (1-v) + (1-m) v)^2
                if (Ei == t && t + a.tau_EI < T) {
                    const float mI = a.m_t[(size_t)g * a.ldP + t + a.tau_EI];
                    const float den = __fmaf_rn(mI, 1.f - vf, (1.f - mI) * vf);
                    pm = H * ((vf * (1.f - vf)) / (den * den));
                }
            }
            float dy;
            float stored = fabsf(G);
            if (SOFT) {
                // dL/dy = s(t) (G - dL/ds(t+1));  dL/ds(t) = y G + (1 - y) dL/ds(t+1)
                const float ds = Apre;
                const float yv = a.y_hist_t[row];
                dy = a.s_hist_t[row] * (G - ds);
                const float dsn = __fmaf_rn(yv, G, (1.f - yv) * ds);
                a.A[row] = dsn;
                stored = fmaxf(stored, fabsf(dsn));
            } else if (Ei == t) { a.A[row] = G; dy = G; }
            else if (never) dy = G;
            else dy = G - Apre;
            const float RS = rs_s[wib][ai];
            const float lam = RS * Lam;
            // dy = 0 and 0 <= lambda < inf: dy/dlambda is finite and >= 0, so the product is dy
            // itself and the draw's uniform is not needed
            float glam = dy;
            if (!(dy == 0.f && lam >= 0.f && lam < __int_as_float(0x7f800000))) {
                const float q = expf(-lam);
                const float p = -expm1f(-lam);
                if (!draws) id = caller_id(a.gr, row, g);
                const float u = uniform_from_word(philox_word(a.seed, id, (uint32_t)t, (uint32_t)g, 0u));
                const float den = __fmaf_rn(p, 1.f - u, q * u);
                const float dydl = (u * (1.f - u)) * q / (den * den);
                glam = dy * dydl;
            }
            const float rc = RS * glam * inv_D;
            a.r_cur[row] = rc;
            v = glam * Lam;
            stored = fmaxf(stored, fabsf(rc));
            rnz_w |= !(rc == 0.f);
            emax_w = max(emax_w, (unsigned)(float_exponent(stored) + 128));
        }

        // per-tile sums of gl * Lam by age bin (fp32 over 32 rows, FP64 from here on)
        float mine = 0.f;   // lanes 2b, 2b + 1: bin b
        if (__any_sync(0xffffffffu, !(v == 0.f))) mine = warp_bin_sums(v, ai, lane, bin_s[wib]);
        if (!(lane & 1) && (lane >> 1) < kAges) a.P_t[(size_t)tile * kAges + (lane >> 1)] = mine;
        if constexpr (FATE) {
            // dL/dm of day t + tau_EI from this tile's exposures today (fixed tree, FP64 out)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) pm += __shfl_xor_sync(0xffffffffu, pm, o);
            if (lane == 0 && t + a.tau_EI < T) a.Pm_t[tile] = ldexp((double)pm, sig_t);
        }

        cur = nxt;
    }

    // the block's counts and flags of its warps' last graphs: one thread, without reading
    // what is there first (each warp reading, then writing, held the block's end for two
    // round trips)
    const int sN = __reduce_add_sync(0xffffffffu, cN);
    const unsigned em = __reduce_max_sync(0xffffffffu, emax_w);
    const bool nz = __any_sync(0xffffffffu, rnz_w);
    if (lane == 0) {
        red_s[wib][0] = cur_g;
        red_s[wib][1] = sN;
        red_s[wib][2] = (int)em - 128;
        red_s[wib][3] = nz;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int g = -1, acc = 0, top = 0, any = 0;
        for (int w = 0; w <= NW; ++w) {
            const int gw = (w < NW) ? red_s[w][0] : -2;
            if (gw != g) {
                if (g >= 0) {
                    if (acc) atomicAdd(a.newRM + (size_t)g * a.ldP + t, acc);
                    if (top > 0) atomicMax(a.emax + (size_t)g * a.ld_sig + t, top);   // stored maxima start at 0
                    if (any) a.rnz[(size_t)g * a.ld_sig + t] = 1;
                }
                g = gw;
                acc = top = any = 0;
            }
            if (w < NW && gw >= 0) {
                acc += red_s[w][1];
                top = max(top, red_s[w][2]);
                any |= red_s[w][3];
            }
        }
    }
}

// Normalised neighbour sums Lam_i(t) over the in-edges, recomputed from the final
// exposure days (used when the in- and out-edges differ, ahead of the backward day
// kernel of day t); the same per-row summation as the forward.
__global__ void __launch_bounds__(kBlock) k_lam_day(Sell m, const int16_t *E, const uint32_t *bits, GraphRef gr,
                                                    int t, int L, int ntiles, const float *c, const float *long_lam,
                                                    float *lam_out) {
    __shared__ float c_s[kMaxL];
    if (threadIdx.x < kMaxL) c_s[threadIdx.x] = c[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nwarps = gridDim.x * (kBlock / 32);
    for (int tile = blockIdx.x * (kBlock / 32) + wib; tile < ntiles; tile += nwarps) {
        const int row = tile * kTile + lane;
        const int Ei = E[row];
        const bool act = (Ei != kPad) && (Ei == kNever || Ei >= t);
        uint32_t len;
        int lrow;
        split_len(m.row_len[row], len, lrow);
        float sum = marked_sum(m, m.slice_ptr[tile], len, act, lane, bits, E, c_s, t, L);
        if (lrow >= 0) sum = long_lam[lrow];
        if (act) {
            const int g = gr.tile_graph ? (int)gr.tile_graph[tile] : 0;
            lam_out[row] = sum * gr.inv_Dbar[g];
        }
    }
}

// The seeds' share of the table adjoint through day 0: a seed exposed on day E < 0 is
// infectious on day 0 with k = -E, and gx(0) = sum over its out-edges of w r(0) (r(0) at
// scale 2^sigma(0)).  Only tiles holding a seed do any work.
__global__ void __launch_bounds__(kBlock) k_dc_seeds(Sell m, const int16_t *E, const float *r0, GraphRef gr,
                                                     const int32_t *sig, int ld_sig, int ntiles, int L,
                                                     const float *long_gx, double *dc_tile) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nwarps = gridDim.x * (kBlock / 32);
    for (int tile = blockIdx.x * (kBlock / 32) + wib; tile < ntiles; tile += nwarps) {
        const int row = tile * kTile + lane;
        const int Ei = E[row];
        const bool seed = Ei != kPad && Ei < 0 && -Ei <= L - 1;
        if (!__any_sync(0xffffffffu, seed)) continue;
        uint32_t len;
        int lrow;
        split_len(m.row_len[row], len, lrow);
        float sum = gather_sum(m, m.slice_ptr[tile], len, seed, lane, r0);
        if (lrow >= 0) sum = long_gx[lrow];
        const int g = gr.tile_graph ? (int)gr.tile_graph[tile] : 0;
        dc_accumulate(dc_tile, tile, seed, -Ei, sum, sig[(size_t)g * ld_sig], lane);
    }
}

// Sampled R/M split: the fate draws of agents exposed before day 0 (E < 0, drawn on day
// t_I = max(E + tau_EI, 0)).  H = gD_{E+L_M} + sum over k between the two exits of
// +-c[k] gx(E + k) over days 0..T-1: gx(0) gathered from r(0), later days from the ring
// (day d in slot d mod (L-1), written while the sweep ran).  Each tile adds its seeds'
// H dphi/dm per day t_I < tau_EI (warp tree in FP64) to Pm[t_I][tile], zeroed beforehand.
__global__ void __launch_bounds__(kBlock) k_fate_seeds(Sell m, const int16_t *E, const float *r0, const float *ring,
                                                       int Lm1, GraphRef gr, FateRef f,
                                                       const double *gD, const int32_t *sig, int ld_sig,
                                                       const int32_t *rnz, int ntiles, int T, const float *c,
                                                       const float *long_gx, double *Pm) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nwarps = gridDim.x * (kBlock / 32);
    const int L = Lm1 + 1;
    const int Lmin = min(f.L_R, f.L_M);
    const double sgn = f.L_M > f.L_R ? 1.0 : -1.0;
    for (int tile = blockIdx.x * (kBlock / 32) + wib; tile < ntiles; tile += nwarps) {
        const int row = tile * kTile + lane;
        const int Ei = E[row];
        const int tI = max(Ei + f.tau_EI, 0);
        const bool seed = Ei != kPad && Ei != kNever && Ei < 0 && tI < T;
        if (!__any_sync(0xffffffffu, seed)) continue;
        const int g = gr.tile_graph ? (int)gr.tile_graph[tile] : 0;
        const int32_t *sg = sig + (size_t)g * ld_sig;
        // gx(0), needed when day 0 lies between the two exits
        const bool at0 = seed && -Ei >= Lmin && -Ei < L;
        uint32_t len;
        int lrow;
        split_len(m.row_len[row], len, lrow);
        float gx0 = gather_sum(m, m.slice_ptr[tile], len, at0, lane, r0);
        if (lrow >= 0) gx0 = long_gx[lrow];
        double pm = 0.0;
        if (seed) {
            const size_t pg = (size_t)g * f.ldP;
            double H = (Ei + f.L_M >= 0 && Ei + f.L_M < T) ? gD[pg + Ei + f.L_M] : 0.0;
            for (int k = Lmin; k < L; ++k) {
                const int d = Ei + k;
                if (d < 0 || d >= T || rnz[(size_t)g * ld_sig + d] == 0) continue;   // no adjoint: gx(d) = 0
                const float gxs = d == 0 ? gx0 : ring[((size_t)tile * Lm1 + d % Lm1) * kTile + lane];
                H += sgn * (double)c[k] * ldexp((double)gxs, sg[d]);
            }
            const float vf = fate_uniform(f, caller_id(gr, row, g), tI, g);
            const double mI = (double)f.mort[pg + tI], v = (double)vf;
            const double den = mI * (1.0 - v) + (1.0 - mI) * v;
            pm = H * (v * (1.0 - v) / (den * den));
        }
        for (int d = 0; d < f.tau_EI && d < T; ++d) {
            double x = (seed && tI == d) ? pm : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0 && x != 0.0) Pm[(size_t)d * ntiles + tile] = x;
        }
    }
}

// dm[g][t] = sum over the graph's tiles of Pm[t][tile] (fixed order, FP64).
__global__ void __launch_bounds__(256) k_fate_dm(const double *Pm, int ntiles, const int32_t *graph_tile0,
                                                 const int32_t *graph_ntiles, int T, double *dm) {
    __shared__ double s[256];
    const int t = blockIdx.x, g = blockIdx.y;
    const int tile0 = graph_tile0[g], nt = graph_ntiles[g];
    double acc = 0.0;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) acc += Pm[(size_t)t * ntiles + tile0 + i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) dm[(size_t)g * T + t] = s[0];
}

// dc[g][k] = sum over the graph's tiles of dc_tile[tile][k] (fixed order, FP64), k < L.
__global__ void __launch_bounds__(256) k_dc_reduce(const double *dc_tile, const int32_t *graph_tile0,
                                                   const int32_t *graph_ntiles, int L, double *dc) {
    __shared__ double s[256];
    const int g = blockIdx.x, k = blockIdx.y;
    const int tile0 = graph_tile0[g], nt = graph_ntiles[g];
    double acc = 0.0;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) acc += dc_tile[(size_t)(tile0 + i) * kMaxL + k];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) dc[(size_t)g * L + k] = s[0];
}

// parts[t][inst][c][a] = sum over the c-th of gridDim.z shares of the graph's tiles of
// P[t][tile][a], fixed order, FP64.  The shares' elements are taken in a row by kReduceBlock
// threads, a multiple of nine, so a thread keeps one age bin and the loads are coalesced; one
// block of 256 threads a day with nine accumulators each took 130 us on the 1M-agent graph.
constexpr int kReduceBlock = 9 * 56;
__global__ void __launch_bounds__(kReduceBlock) k_bwd_reduce(const float *P, int ntiles, const int32_t *graph_tile0,
                                                             const int32_t *graph_ntiles, double *parts) {
    __shared__ double s[kReduceBlock];
    const int t = blockIdx.x, inst = blockIdx.y, c = blockIdx.z, tid = threadIdx.x;
    const int tile0 = graph_tile0[inst], nt = graph_ntiles[inst];
    const int np = gridDim.z, i0 = (int)((long long)nt * c / np), i1 = (int)((long long)nt * (c + 1) / np);
    const float *p = P + ((size_t)t * ntiles + tile0 + i0) * kAges;
    const int n = (i1 - i0) * kAges;
    double acc = 0.0;
    int i = tid;
    for (; i + 3 * kReduceBlock < n; i += 4 * kReduceBlock) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = p[i + u * kReduceBlock];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc += (double)v[u];
    }
    for (; i < n; i += kReduceBlock) acc += (double)p[i];
    s[tid] = acc;
    __syncthreads();
    if (tid < kAges) {   // 56 values of bin tid, in order
        double v = 0.0;
        for (int k = 0; k < kReduceBlock / kAges; ++k) v += s[k * kAges + tid];
        parts[(((size_t)t * gridDim.y + inst) * np + c) * kAges + tid] = v;
    }
}

// Q[inst][t][a] = 2^sigma(t) x the sum of the np shares, in order.
__global__ void k_bwd_reduce_parts(const double *parts, int np, int T, const int32_t *sig, int ld_sig, double *Q) {
    const int t = blockIdx.x, inst = blockIdx.y, a = threadIdx.x;
    if (a >= kAges) return;
    const double *p = parts + ((size_t)t * gridDim.y + inst) * np * kAges + a;
    double v = 0.0;
    for (int c = 0; c < np; ++c) v += p[c * kAges];
    Q[((size_t)inst * T + t) * kAges + a] = ldexp(v, sig[(size_t)inst * ld_sig + t]);
}

// dR_t = sum_a S_a Q[t][a];  dS_a = sum_t R_t Q[t][a];  dm_t = gD_t newRM(t) (not written
// when both counts are NULL: the sampled R/M split's dm comes from k_fate_dm).
__global__ void __launch_bounds__(256) k_bwd_finalize(const double *Q, const float *R, const float *S,
                                                      const double *gD, const int32_t *newRM,
                                                      const double *newRM_real, int ldP, int T, double *dR,
                                                      double *dm, double *dS) {
    const int inst = blockIdx.x;
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        const double *q = Q + ((size_t)inst * T + t) * kAges;
        double acc = 0.0;
        for (int b = 0; b < kAges; ++b) acc += (double)S[inst * kAges + b] * q[b];
        dR[(size_t)inst * T + t] = acc;
        const size_t pi = (size_t)inst * ldP + t;
        if (newRM_real || newRM) dm[(size_t)inst * T + t] = gD[pi] * (newRM_real ? newRM_real[pi] : (double)newRM[pi]);
    }
    if (threadIdx.x < kAges) {
        const int b = threadIdx.x;
        double acc = 0.0;
        for (int t = 0; t < T; ++t) acc += (double)R[(size_t)inst * ldP + t] * Q[((size_t)inst * T + t) * kAges + b];
        dS[inst * kAges + b] = acc;
    }
}

}  // namespace

// The instance of a day.  deep (deep_gather in capi.cu holds the rule): two blocks an SM with
// most of an ordinary row in flight instead of three with two pairs a lane ahead.  A row sum
// is a chain of round trips, so fewer and longer batches win wherever the fewer warps don't
// cost more waves of tiles than that saves.  Us per day, three blocks against two: 1M town
// 61.0 -> 58.9, twelve counties 29.2 -> 24.1, 300k power law 52.2 -> 37.1, deaths sampled at
// 200k 24.1 -> 23.3 (at 1M, 4, 5 and 7 pairs: 62.4, 59.9, 61.5).  The instances with the
// table's adjoint have other work between the loads: 15.5 -> 16.8 at 100k, so they stay.
using BwdKernel = void (*)(BwdDayArgs);
static BwdKernel bwd_kernel(int mode, bool dc, int exit_mode, bool deep) {
    constexpr int D = kDeepPairs;
    if (exit_mode == kExitFate)
        return deep ? k_bwd_day<kBwdStore, false, kExitFate, kBlock, 2, D> : k_bwd_day<kBwdStore, false, kExitFate>;
    if (exit_mode == kExitDur)
        return deep ? k_bwd_day<kBwdStore, false, kExitDur, kBlock, 2, D> : k_bwd_day<kBwdStore, false, kExitDur>;
    if (mode == kBwdSoft) return dc ? k_bwd_day<kBwdSoft, true> : k_bwd_day<kBwdSoft, false>;
    if (mode == kBwdFused) {
        if (dc) return k_bwd_day<kBwdFused, true>;
        return deep ? k_bwd_day<kBwdFused, false, kExitBase, kBlock, 2, D> : k_bwd_day<kBwdFused, false>;
    }
    if (dc) return k_bwd_day<kBwdStore, true>;
    return deep ? k_bwd_day<kBwdStore, false, kExitBase, kBlock, 2, D> : k_bwd_day<kBwdStore, false>;
}

cudaError_t launch_bwd_day(const BwdDayArgs &a, int grid, bool small, bool deep, bool overlap, cudaStream_t s) {
    const bool dc = a.dc_tile != nullptr;
    const int exit_mode = a.fate.L_M > 0 ? kExitFate : a.dur.n > 0 ? kExitDur : kExitBase;
    if (a.mode != kBwdStore && a.mode != kBwdFused && a.mode != kBwdSoft) return cudaErrorInvalidValue;
    // store policy, plain instance only (checked at creation)
    if (exit_mode != kExitBase && (a.mode != kBwdStore || dc)) return cudaErrorInvalidValue;
    if (small && !dc)
        return launch_day(k_bwd_day<kBwdStore, false, kExitBase, kSmallBlock, 8, kDeepPairs>,
                          (a.ntiles * 32 + kSmallBlock - 1) / kSmallBlock, kSmallBlock, 0, s, overlap, a);
    return launch_day(bwd_kernel(a.mode, dc, exit_mode, deep), grid, kBlock, 0, s, overlap, a);
}

cudaError_t launch_dc_seeds(Sell m_out, const int16_t *E, const float *r0, GraphRef gr, const int32_t *sig,
                            int ld_sig, int ntiles, int L, const float *long_gx, double *dc_tile, int grid,
                            cudaStream_t s) {
    k_dc_seeds<<<grid, kBlock, 0, s>>>(m_out, E, r0, gr, sig, ld_sig, ntiles, L, long_gx, dc_tile);
    return cudaGetLastError();
}

cudaError_t launch_fate_seeds(Sell m_out, const int16_t *E, const float *r0, const float *ring, int Lm1, GraphRef gr, FateRef f, const double *gD, const int32_t *sig, int ld_sig,
                              const int32_t *rnz, int ntiles, int T, const float *c, const float *long_gx, double *Pm,
                              int grid, cudaStream_t s) {
    k_fate_seeds<<<grid, kBlock, 0, s>>>(m_out, E, r0, ring, Lm1, gr, f, gD, sig, ld_sig, rnz, ntiles, T, c, long_gx,
                                         Pm);
    return cudaGetLastError();
}

cudaError_t launch_fate_dm(const double *Pm, int ntiles, const int32_t *graph_tile0, const int32_t *graph_ntiles,
                           int G, int T, double *dm, cudaStream_t s) {
    if (T > 0) k_fate_dm<<<dim3(T, G), 256, 0, s>>>(Pm, ntiles, graph_tile0, graph_ntiles, T, dm);
    return cudaGetLastError();
}

cudaError_t launch_dc_reduce(const double *dc_tile, const int32_t *graph_tile0, const int32_t *graph_ntiles, int G,
                             int L, double *dc, cudaStream_t s) {
    k_dc_reduce<<<dim3(G, L), 256, 0, s>>>(dc_tile, graph_tile0, graph_ntiles, L, dc);
    return cudaGetLastError();
}

cudaError_t launch_lam_day(Sell m, const int16_t *E, const uint32_t *bits, GraphRef gr, int t, int L, int ntiles,
                           const float *c, const float *long_lam, float *lam_out, int grid, cudaStream_t s) {
    k_lam_day<<<grid, kBlock, 0, s>>>(m, E, bits, gr, t, L, ntiles, c, long_lam, lam_out);
    return cudaGetLastError();
}

int occupancy_bwd(int mode, bool dc, int exit_mode, bool deep) {
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, bwd_kernel(mode, dc, exit_mode, deep), kBlock, 0);
    return blocks > 0 ? blocks : 1;
}

cudaError_t launch_bwd_reduce(const float *P, int ntiles, const int32_t *graph_tile0, const int32_t *graph_ntiles,
                              int T, int I, const int32_t *sig, int ld_sig, double *parts, int np, double *Q,
                              cudaStream_t s) {
    k_bwd_reduce<<<dim3(T, I, np), kReduceBlock, 0, s>>>(P, ntiles, graph_tile0, graph_ntiles, parts);
    k_bwd_reduce_parts<<<dim3(T, I), 32, 0, s>>>(parts, np, T, sig, ld_sig, Q);
    return cudaGetLastError();
}

cudaError_t launch_bwd_finalize(const double *Q, const float *R, const float *S, const double *gD,
                                const int32_t *newRM, const double *newRM_real, int ldP, int T, int I, double *dR,
                                double *dm, double *dS, cudaStream_t s) {
    k_bwd_finalize<<<I, 256, 0, s>>>(Q, R, S, gD, newRM, newRM_real, ldP, T, dR, dm, dS);
    return cudaGetLastError();
}

}  // namespace gabm
