// longrows.cu -- the sums of long rows (LongRows), a block each, ahead of the day kernel.
//
// What bounds it: the two dependent round trips of an entry (its column, then the
// neighbour's value) and the launch itself.  A block of 128 threads keeps four entries a
// thread in flight, so a row of 2000 entries is four rounds; one warp a row took four times
// that, and a lane of a SELL tile two thousand steps.
#include "gabm_internal.cuh"
#include "rowsum.cuh"

namespace gabm {

namespace {

constexpr int kLongBlock = 128;
constexpr int kLongUnroll = 4;

// (s, c) += (s2, c2): compensated sums (value s - c) added with the rounding of s + s2 kept in c.
__device__ __forceinline__ void add_pair(float &s, float &c, float s2, float c2) {
    const float t = __fadd_rn(s, s2);
    const float z = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(s2, z));   // s + s2 - t exactly
    c = __fsub_rn(__fadd_rn(c, c2), err);
    s = t;
}

// One block per long row: blocks [0, in.n) the in-rows, the others the out-rows.
__global__ void __launch_bounds__(kLongBlock) k_long(LongArgs a) {
    __shared__ float c_s[kMaxL];
    __shared__ float2 part[kLongBlock / 32];
    pdl_trigger();
    if (threadIdx.x < kMaxL) c_s[threadIdx.x] = a.c[threadIdx.x];
    __syncthreads();
    const bool in = (int)blockIdx.x < a.in.n;
    const LongRows &lr = in ? a.in : a.out;
    const int i = in ? (int)blockIdx.x : (int)blockIdx.x - a.in.n;
    const uint32_t row = lr.row[i], p0 = lr.ptr[i], p1 = lr.ptr[i + 1];
    pdl_wait();
    if (!in && a.flags && marked(a.bits, row))
        for (uint32_t p = p0 + threadIdx.x; p < p1; p += kLongBlock) a.flags[lr.cw[p].x] = 1;
    if (in ? !a.lam : !a.gx) return;
    const int er = a.e[row];
    if (in ? er < a.t && !(a.cycle > 0 && a.t - er >= a.cycle) : er < a.gx_from) return;
    const int g = a.tile_graph ? (int)a.tile_graph[row / kTile] : 0;
    const bool dead = !in && a.rnz && a.rnz[(size_t)g * a.ld_sig + a.t + 1] == 0;
    float s = 0.f, c = 0.f;
    for (uint32_t q = dead ? p1 : p0; q < p1; q += kLongBlock * kLongUnroll) {
        uint2 v[kLongUnroll];
        float x[kLongUnroll];
        bool ok[kLongUnroll];
#pragma unroll
        for (int u = 0; u < kLongUnroll; ++u) {
            const uint32_t p = q + threadIdx.x + (uint32_t)(u * kLongBlock);
            ok[u] = p < p1;
            v[u] = ok[u] ? lr.cw[p] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < kLongUnroll; ++u) {
            x[u] = 0.f;
            if (in) {
                const bool mk = ok[u] && marked(a.bits, v[u].x);
                const int k = mk ? a.t - (int)a.e[v[u].x] : 0;
                ok[u] = mk && (unsigned)(k - 1) < (unsigned)(a.L - 1);
                if (ok[u]) x[u] = c_s[k];
            } else if (ok[u]) {
                x[u] = a.x[v[u].x];
            }
        }
#pragma unroll
        for (int u = 0; u < kLongUnroll; ++u)
            if (ok[u]) kahan_add(s, c, __uint_as_float(v[u].y) * x[u]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        add_pair(s, c, __shfl_down_sync(0xffffffffu, s, o), __shfl_down_sync(0xffffffffu, c, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_float2(s, c);
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kLongBlock / 32; ++w) add_pair(s, c, part[w].x, part[w].y);
        (in ? a.lam : a.gx)[i] = __fsub_rn(s, c);
    }
}

}  // namespace

cudaError_t launch_long(const LongArgs &a, bool overlap, cudaStream_t s) {
    if (a.in.n + a.out.n == 0) return cudaSuccess;
    return launch_day(k_long, a.in.n + a.out.n, kLongBlock, 0, s, overlap, a);
}

}  // namespace gabm
