// k_line.cuh -- m = 1: prefix aggregation over the sorted points.
//
// With one coordinate a query's dominated set is the data before it in the
// order of that coordinate (queries first on ties): a single level whose
// records are the points themselves (Sec. 1.1).  The scan of F runs over the
// permutation directly -- per tile F over its data (k_line_sum, which also
// puts the weights in order), the tiles' prefixes in a fixed order
// (k_line_carry), then every query's F to its output (k_line_apply) -- and
// nothing is counted, written or read as a record: 3 launches of 24 bytes per
// point instead of the count scan, flat map, segmented scan and reduction
// (200 of 585 us at 6.3e6 points), bound by the random gathers of the weights
// and the random writes of the outputs.
#pragma once
#include "k_points.cuh"
#include "k_records.cuh"

namespace domagg {

constexpr int LINE_THREADS = 256, LINE_ITEMS = 16;  // a tile: POINT_TILE points

// The point at position x of the order of the last coordinate (read backwards
// for a non-strict one).
__device__ __forceinline__ u32 line_point(const u32* __restrict__ perm, const TileLoc& L, bool rev, u32 x, u32 n_total) {
    const u32 j = perm[rev ? L.seg_begin + (L.seg_end - 1u - x) : x];
    return j < n_total ? j : L.seg_begin;  // (always, for a valid permutation)
}

// Per tile F over its data, in position order; the data's weights in that order.
template <class Op, int WT>
__global__ __launch_bounds__(LINE_THREADS) void k_line_sum(const u32* __restrict__ perm,
                                                           const u32* __restrict__ seg_off,
                                                           const u32* __restrict__ tile_off, int nseg,
                                                           const Inst* __restrict__ inst,
                                                           typename Op::W* __restrict__ pw,
                                                           typename Op::Acc* __restrict__ tagg) {
    typedef typename Op::Acc Acc;
    __shared__ Acc s_w[LINE_THREADS / 32];
    const u32 t = blockIdx.x;
    if (t >= __ldg(tile_off + nseg)) return;
    const TileLoc L = locate_tile<LINE_THREADS * LINE_ITEMS>(t, seg_off, tile_off, nseg);
    const Inst& I = inst[L.seg];
    const u32 nQ = I.nQ, n_total = __ldg(seg_off + nseg);
    const bool rev = I.flags & 1u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u32 w0 = L.start + (u32)warp * 32u * LINE_ITEMS + (u32)lane;
    u32 j[LINE_ITEMS];
#pragma unroll
    for (int i = 0; i < LINE_ITEMS; ++i) {
        const u32 x = w0 + 32u * i;
        j[i] = x < L.end ? line_point(perm, L, rev, x, n_total) - L.seg_begin : 0u;
    }
    Acc acc = Op::e();
#pragma unroll
    for (int i = 0; i < LINE_ITEMS; ++i) {
        const u32 x = w0 + 32u * i;
        if (x < L.end && j[i] >= nQ) {
            if constexpr (WT == 3) {
                acc = Op::F(acc, Op::from_pay(0u));
            } else {
                const typename Op::W w = reinterpret_cast<const typename Op::W*>(I.dw)[j[i] - nQ];
                pw[x] = w;
                if constexpr (Op::GATHER) acc = Op::F(acc, Op::from_w(w));
                else acc = Op::F(acc, Op::from_pay(w));
            }
        }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc = Op::F(acc, shfl_xor_acc(acc, o));
    if (lane == 0) s_w[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < LINE_THREADS / 32; ++w) acc = Op::F(acc, s_w[w]);
        tagg[t] = acc;
    }
}

// Exclusive scan of the tiles' F per instance, in place: one block each, its
// 1024 threads take consecutive tiles (a fixed order).
template <class Op>
__global__ __launch_bounds__(1024) void k_line_carry(const u32* __restrict__ tile_off,
                                                     typename Op::Acc* __restrict__ tagg) {
    typedef typename Op::Acc Acc;
    __shared__ Acc s_w[32];
    const u32 t0 = __ldg(tile_off + blockIdx.x), n = __ldg(tile_off + blockIdx.x + 1) - t0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const u32 per = (n + 1023u) / 1024u, a = min(n, (u32)tid * per), b = min(n, a + per);
    Acc sum = Op::e();
    for (u32 t = a; t < b; ++t) sum = Op::F(sum, tagg[t0 + t]);
    Acc inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Acc x = shfl_up_acc(inc, o);
        if (lane >= o) inc = Op::F(x, inc);
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    Acc run = Op::e();
    for (int w = 0; w < warp; ++w) run = Op::F(run, s_w[w]);
    const Acc lex = shfl_up_acc(inc, 1);
    if (lane > 0) run = Op::F(run, lex);
    for (u32 t = a; t < b; ++t) {
        const Acc v = tagg[t0 + t];
        tagg[t0 + t] = run;
        run = Op::F(run, v);
    }
}

template <class Op, int WT>
constexpr size_t line_smem() {
    return (size_t)Padded<LINE_THREADS * LINE_ITEMS>::value * (4 + (WT == 3 ? 0 : sizeof(typename Op::W)));
}

// Every query's F over the data before it.
template <class Op, int WT>
__global__ __launch_bounds__(LINE_THREADS) void k_line_apply(const u32* __restrict__ perm,
                                                             const u32* __restrict__ seg_off,
                                                             const u32* __restrict__ tile_off, int nseg,
                                                             const Inst* __restrict__ inst,
                                                             const typename Op::W* __restrict__ pw,
                                                             const typename Op::Acc* __restrict__ carry) {
    typedef typename Op::Acc Acc;
    constexpr int TILE = LINE_THREADS * LINE_ITEMS;
    extern __shared__ __align__(128) unsigned char smem[];  // line_smem: weights, then points
    typename Op::W* s_p = reinterpret_cast<typename Op::W*>(smem);
    u32* s_j = reinterpret_cast<u32*>(s_p + (WT == 3 ? 0 : Padded<TILE>::value));
    __shared__ Acc s_w[LINE_THREADS / 32];
    const u32 t = blockIdx.x;
    if (t >= __ldg(tile_off + nseg)) return;
    const TileLoc L = locate_tile<TILE>(t, seg_off, tile_off, nseg);
    const Inst& I = inst[L.seg];
    const u32 nQ = I.nQ, n_total = __ldg(seg_off + nseg);
    const bool rev = I.flags & 1u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < LINE_ITEMS; ++i) {
        const u32 x = (u32)i * LINE_THREADS + threadIdx.x;
        const bool in = L.start + x < L.end;
        s_j[pidx(x)] = in ? line_point(perm, L, rev, L.start + x, n_total) - L.seg_begin : 0u;
        if constexpr (WT != 3) s_p[pidx(x)] = in ? pw[L.start + x] : typename Op::W(0);  // (a query's is not used)
    }
    __syncthreads();
    const u32 x0 = threadIdx.x * LINE_ITEMS, n = L.end - L.start;
    auto weight = [&](u32 x) -> Acc {
        if constexpr (WT == 3) return Op::from_pay(0u);
        else if constexpr (Op::GATHER) return Op::from_w(s_p[pidx(x)]);
        else return Op::from_pay(s_p[pidx(x)]);
    };
    Acc sum = Op::e();
#pragma unroll
    for (int i = 0; i < LINE_ITEMS; ++i)
        if (x0 + i < n && s_j[pidx(x0 + i)] >= nQ) sum = Op::Fc(sum, weight(x0 + i));
    sum = Op::F(sum, Op::e());
    Acc inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Acc x = shfl_up_acc(inc, o);
        if (lane >= o) inc = Op::F(x, inc);
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    Acc run = carry[t];
    for (int w = 0; w < warp; ++w) run = Op::F(run, s_w[w]);
    const Acc lex = shfl_up_acc(inc, 1);
    if (lane > 0) run = Op::F(run, lex);
#pragma unroll
    for (int i = 0; i < LINE_ITEMS; ++i) {
        if (x0 + i < n) {
            const u32 j = s_j[pidx(x0 + i)];
            if (j >= nQ) run = Op::F(run, weight(x0 + i));
            else reinterpret_cast<typename Op::Out*>(I.out)[j] = Op::to_out(run);
        }
    }
}

}  // namespace domagg
