// k_items.cuh -- m = 3: the first rank's levels above the groups as m = 2
// problems, one per node.
//
// A record of first-rank level lv is keyed by the node r0 >> (lv+1) refined by
// a node of the second rank.  The points that level lv emits (data with rank
// bit lv = 0, queries with bit lv = 1), per first-rank node in the order of
// the last coordinate, are an m = 2 problem of their own -- second rank, last
// coordinate: every datum of the node precedes every query in the first
// coordinate (Lemma 1) -- whose answers are the query's partial results at
// that level.  So instead of writing a record per second-rank digit (n log^2 n
// of them, sorted by four radix passes in HBM), a point is written once per
// level (an item), the items are sorted by node (two passes on at most ten
// bits), and all nodes of all levels go through the m = 2 pipeline as one
// batch, which forms, sorts and scans their records in shared memory.  At 2^21
// per side, the ten levels above the groups: 2.3e8 records against 2.1e7
// items.
#pragma once
#include <type_traits>

#include "k_points.cuh"

namespace domagg {

constexpr u32 ITEM_TILE = 4096;  // items of a tile of the node search

// Per 32-point chunk and level of Inst::topmask (for m = 3: the levels taken
// by items), the items and query items before the chunk within its tile, and
// the tiles' totals; laid out as k_count_scan's record counts.
static __global__ __launch_bounds__(256) void k_item_count(const u32* __restrict__ seg_off,
                                                           const u32* __restrict__ tile_off, int nseg,
                                                           const u32* __restrict__ chunk_off,
                                                           const u32* __restrict__ pr0, const Inst* __restrict__ inst,
                                                           u32* __restrict__ chunk_base,
                                                           u32* __restrict__ qchunk_base, u32* __restrict__ tile_cnt) {
    constexpr int WARPS = 8, TILE = WARPS * CS_ROUNDS * 32;
    __shared__ u32 s_w[WARPS][CS_COUNTERS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u32 t = blockIdx.x;
    if (t >= __ldg(tile_off + nseg)) return;
    const TileLoc L = locate_tile<TILE>(t, seg_off, tile_off, nseg);
    const Inst& I = inst[L.seg];
    const u32 mask = I.topmask & low_mask(I.b[0]);
    const u32 wstart = L.start + (u32)warp * CS_ROUNDS * 32u;
    u32 v[CS_ROUNDS], rc[CS_ROUNDS], qc[CS_ROUNDS];
#pragma unroll
    for (int i = 0; i < CS_ROUNDS; ++i) {
        const u32 x = wstart + (u32)i * 32u + (u32)lane;
        v[i] = x < L.end ? pr0[x] : 0u;
    }
    u32 run = 0, run_q = 0;
#pragma unroll
    for (int i = 0; i < CS_ROUNDS; ++i) {
        const bool valid = wstart + (u32)i * 32u + (u32)lane < L.end;
        const bool q = (v[i] & QUERY_BIT) != 0u;
        const u32 bits = valid ? (q ? v[i] : ~v[i]) & mask : 0u;
        rc[i] = run;
        qc[i] = run_q;
        run += (u32)__popc(warp_transpose32(bits, (u32)lane));
        run_q += (u32)__popc(warp_transpose32(q ? bits : 0u, (u32)lane));
    }
    s_w[warp][lane] = run;
    s_w[warp][LMAX + lane] = run_q;
    __syncthreads();
    if (threadIdx.x < CS_COUNTERS) {  // exclusive over the warps; the tile's totals
        u32 sum = 0;
        for (int w = 0; w < WARPS; ++w) {
            const u32 x = s_w[w][threadIdx.x];
            s_w[w][threadIdx.x] = sum;
            sum += x;
        }
        tile_cnt[(u64)t * CS_COUNTERS + threadIdx.x] = sum;
    }
    __syncthreads();
    const u32 cbase = __ldg(chunk_off + L.seg) + (wstart - L.seg_begin) / 32u;
#pragma unroll
    for (int i = 0; i < CS_ROUNDS; ++i)
        if (wstart + (u32)i * 32u < L.end) {
            chunk_base[(u64)(cbase + i) * LMAX + lane] = s_w[warp][lane] + rc[i];
            qchunk_base[(u64)(cbase + i) * LMAX + lane] = s_w[warp][LMAX + lane] + qc[i];
        }
}

// The items, level by level (as k_expand): key = node | role bit, payload =
// second rank << 32 | (a datum's position, a query's partial slot: dense per
// level, in the order of the last coordinate).
static __global__ __launch_bounds__(256) void k_item_expand(
    const u32* __restrict__ chunk_off, int k, const u32* __restrict__ pt_offs, const u32* __restrict__ pr0,
    const u32* __restrict__ pr1, const u32* __restrict__ chunk_base, const u32* __restrict__ qchunk_base,
    const u32* __restrict__ pt_tiles, const u32* __restrict__ tile_excl, const Inst* __restrict__ inst,
    const u32* __restrict__ seg_base /*[k][LMAX]*/, const u32* __restrict__ qseg_base /*[k][LMAX]*/, u32 n_items,
    u32* __restrict__ kout, u64* __restrict__ pout) {
    const int lane = threadIdx.x & 31;
    const u32 lt = lanemask_lt();
    const u32 c_end = __ldg(chunk_off + k), warps = (gridDim.x * blockDim.x) >> 5;
    for (u32 c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < c_end; c += warps) {
        const int s = upper_index(chunk_off, k + 1, c);
        const Inst& I = inst[s];
        const u32 c0 = __ldg(chunk_off + s), ps = __ldg(pt_offs + s), p = ps + (c - c0) * 32u + (u32)lane;
        const u32 tile = __ldg(pt_tiles + s) + (c - c0) / CS_CHUNKS;
        const u32 mask = I.topmask & low_mask(I.b[0]);
        const bool valid = p < __ldg(pt_offs + s + 1);
        const u32 v = valid ? pr0[p] : 0u, r1 = valid ? pr1[p] : 0u;
        const bool q = (v & QUERY_BIT) != 0u;
        const u32 a = v & ~QUERY_BIT;
        const u32 bits = valid ? (q ? v : ~v) & mask : 0u;
        // lane lv holds the bases of level lv
        const u32 my = __ldg(seg_base + (u64)s * LMAX + lane) + __ldg(chunk_base + (u64)c * LMAX + lane) +
                       __ldg(tile_excl + (u64)tile * CS_COUNTERS + lane);
        const u32 my_q = __ldg(qseg_base + (u64)s * LMAX + lane) + __ldg(qchunk_base + (u64)c * LMAX + lane) +
                         __ldg(tile_excl + (u64)tile * CS_COUNTERS + LMAX + lane);
        for (u32 m = mask; m; m &= m - 1u) {
            const u32 lv = __ffs(m) - 1;
            const bool has = (bits >> lv) & 1u;
            const u32 hb = __ballot_sync(0xffffffffu, has), qb = __ballot_sync(0xffffffffu, has && q);
            const u32 at = __shfl_sync(0xffffffffu, my, lv) + (u32)__popc(hb & lt);
            const u32 slot = __shfl_sync(0xffffffffu, my_q, lv) + (u32)__popc(qb & lt);
            if (has && domagg_check(at < n_items, SITE_EXPAND)) {
                kout[at] = (a >> (lv + 1u)) | (q ? QUERY_BIT : 0u);
                pout[at] = ((u64)r1 << 32) | (u64)(q ? slot : p);
            }
        }
    }
}

// The sort left segment `seg` in the buffer of its pass count's parity.
__device__ __forceinline__ bool item_odd(const u32* seg_bits, int seg) {
    return ((__ldg(seg_bits + seg) + RADIX_BITS - 1) / RADIX_BITS) & 1u;
}

// Per tile of sorted items: the nodes that start in it and its queries.
static __global__ __launch_bounds__(256) void k_item_heads(const u32* __restrict__ k0, const u32* __restrict__ k1,
                                                           const u32* __restrict__ seg_off,
                                                           const u32* __restrict__ tile_off, int nseg,
                                                           const u32* __restrict__ seg_bits, u32* __restrict__ cnt_h,
                                                           u32* __restrict__ cnt_q) {
    __shared__ u32 s_h[8], s_q[8];
    const u32 t = blockIdx.x;
    if (t >= __ldg(tile_off + nseg)) return;
    const TileLoc L = locate_tile<(int)ITEM_TILE>(t, seg_off, tile_off, nseg);
    const u32* __restrict__ keys = item_odd(seg_bits, L.seg) ? k1 : k0;
    u32 h = 0, q = 0;
#pragma unroll 4
    for (u32 i = 0; i < ITEM_TILE / 256u; ++i) {
        const u32 x = L.start + i * 256u + threadIdx.x;
        if (x < L.end) {
            const u32 key = keys[x];
            h += (x == L.seg_begin || ((keys[x - 1u] ^ key) & ~QUERY_BIT)) ? 1u : 0u;
            q += key >> 31;
        }
    }
    h = __reduce_add_sync(0xffffffffu, h);
    q = __reduce_add_sync(0xffffffffu, q);
    if ((threadIdx.x & 31) == 0) {
        s_h[threadIdx.x >> 5] = h;
        s_q[threadIdx.x >> 5] = q;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            h += s_h[w];
            q += s_q[w];
        }
        cnt_h[t] = h;
        cnt_q[t] = q;
    }
}

// A warp's view of its ITEM_TILE / 8 consecutive items of a tile: heads and
// queries per round of 32, and the nodes and queries before the warp (cnt_h,
// cnt_q: exclusive over the tiles).
constexpr int ITEM_ROUNDS = (int)ITEM_TILE / 256;
struct ItemWarp {
    u32 hb[ITEM_ROUNDS], qb[ITEM_ROUNDS], bh, bq;
};
__device__ __forceinline__ void item_warp(ItemWarp& I, const u32* __restrict__ keys, const TileLoc& L, u32 w0, u32 t,
                                          const u32* cnt_h, const u32* cnt_q, u32* s_h, u32* s_q) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 nh = 0, nq = 0;
#pragma unroll
    for (int i = 0; i < ITEM_ROUNDS; ++i) {
        const u32 x = w0 + 32u * i;
        bool h = false, q = false;
        if (x < L.end) {
            const u32 key = keys[x];
            h = x == L.seg_begin || ((keys[x - 1u] ^ key) & ~QUERY_BIT);
            q = key >> 31;
        }
        I.hb[i] = __ballot_sync(0xffffffffu, h);
        I.qb[i] = __ballot_sync(0xffffffffu, q);
        nh += (u32)__popc(I.hb[i]);
        nq += (u32)__popc(I.qb[i]);
    }
    if (lane == 0) {
        s_h[warp] = nh;
        s_q[warp] = nq;
    }
    __syncthreads();
    I.bh = __ldg(cnt_h + t);
    I.bq = __ldg(cnt_q + t);
    for (int w = 0; w < warp; ++w) {
        I.bh += s_h[w];
        I.bq += s_q[w];
    }
}

// Every node's first item and the queries before it, in the order of the
// sorted items; behind the last node, the totals.
static __global__ __launch_bounds__(256) void k_item_starts(
    const u32* __restrict__ k0, const u32* __restrict__ k1, const u32* __restrict__ seg_off,
    const u32* __restrict__ tile_off, int nseg, const u32* __restrict__ seg_bits, const u32* __restrict__ cnt_h,
    const u32* __restrict__ cnt_q, u32 max_nodes, u32 n_items, u32 n_queries, u32* __restrict__ node_start,
    u32* __restrict__ node_q) {
    __shared__ u32 s_h[8], s_q[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u32 lt = lanemask_lt();
    const u32 t = blockIdx.x, ntile = __ldg(tile_off + nseg);
    if (t >= ntile) return;
    const TileLoc L = locate_tile<(int)ITEM_TILE>(t, seg_off, tile_off, nseg);
    const u32* __restrict__ keys = item_odd(seg_bits, L.seg) ? k1 : k0;
    const u32 w0 = L.start + (u32)warp * 32u * ITEM_ROUNDS + (u32)lane;
    ItemWarp I;
    item_warp(I, keys, L, w0, t, cnt_h, cnt_q, s_h, s_q);
#pragma unroll
    for (int i = 0; i < ITEM_ROUNDS; ++i) {
        if ((I.hb[i] >> lane) & 1u) {
            const u32 node = I.bh + (u32)__popc(I.hb[i] & lt);
            if (domagg_check(node < max_nodes, SITE_EXPAND)) {
                node_start[node] = w0 + 32u * i;
                node_q[node] = I.bq + (u32)__popc(I.qb[i] & lt);
            }
        }
        I.bh += (u32)__popc(I.hb[i]);
        I.bq += (u32)__popc(I.qb[i]);
    }
    if (t == 0u && threadIdx.x == 0) {
        const u32 nn = min(__ldg(cnt_h + ntile), max_nodes);
        node_start[nn] = n_items;
        node_q[nn] = n_queries;
    }
}

// The m = 2 problems as their point phase has them (queries first, then data,
// node by node): the ranked keys (second ranks), the permutation that puts a
// node's points in the order of the last coordinate (the items' own order),
// the data's weights and the queries' partial slots.
template <class Op, int WT>
__global__ __launch_bounds__(256) void k_item_place(
    const u32* __restrict__ k0, const u32* __restrict__ k1, const u64* __restrict__ p0, const u64* __restrict__ p1,
    const u32* __restrict__ seg_off, const u32* __restrict__ tile_off, int nseg, const u32* __restrict__ seg_bits,
    const u32* __restrict__ cnt_h, const u32* __restrict__ cnt_q, const typename Op::W* __restrict__ pw, u32 max_nodes,
    u32 n_items, const u32* __restrict__ node_start, const u32* __restrict__ node_q, u32* __restrict__ rkey,
    u32* __restrict__ perm, u32* __restrict__ slot, typename Op::W* __restrict__ wout) {
    __shared__ u32 s_h[8], s_q[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u32 lt = lanemask_lt(), le = lt | (1u << lane);
    const u32 t = blockIdx.x;
    if (t >= __ldg(tile_off + nseg)) return;
    const TileLoc L = locate_tile<(int)ITEM_TILE>(t, seg_off, tile_off, nseg);
    const bool odd = item_odd(seg_bits, L.seg);
    const u64* __restrict__ pays = odd ? p1 : p0;
    const u32 w0 = L.start + (u32)warp * 32u * ITEM_ROUNDS + (u32)lane;
    ItemWarp I;
    item_warp(I, odd ? k1 : k0, L, w0, t, cnt_h, cnt_q, s_h, s_q);
#pragma unroll 4
    for (int i = 0; i < ITEM_ROUNDS; ++i) {
        const u32 x = w0 + 32u * i;
        if (x < L.end) {
            const u32 node = I.bh + (u32)__popc(I.hb[i] & le) - 1u, qi = I.bq + (u32)__popc(I.qb[i] & lt);
            if (domagg_check(node < max_nodes, SITE_EXPAND)) {
                const u32 start = __ldg(node_start + node), q0 = __ldg(node_q + node), nq = __ldg(node_q + node + 1) - q0;
                const u64 v = pays[x];
                const bool q = (I.qb[i] >> lane) & 1u;
                // the node's queries come first, then its data
                const u32 j = start + (q ? qi - q0 : nq + (x - start) - (qi - q0));
                if (domagg_check(j < n_items, SITE_EXPAND)) {
                    rkey[j] = (u32)(v >> 32);
                    perm[x] = j;
                    if (q) slot[qi] = (u32)v;
                    else if constexpr (WT != 3) wout[x - qi] = __ldg(pw + (u32)v);
                }
            }
        }
        I.bh += (u32)__popc(I.hb[i]);
        I.bq += (u32)__popc(I.qb[i]);
    }
}

// Every query item's answer to its partial slot.  A float32 sum comes and goes
// as a float-float pair (lo: its low halves): rounded to one float32 per level
// the query's sum was less accurate than by records, of which a level has one
// per second-rank node (outputs that are not the exact sum rounded once, 2^18
// per side, weights of one sign: 19.0 % with the rounding, 4.3 % without,
// 13.3 % by records).
template <class Op>
__global__ void k_item_out(const typename Op::Out* __restrict__ out, const float* __restrict__ lo,
                           const u32* __restrict__ slot, u32 n, typename Op::Acc* __restrict__ part) {
    const u32 i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !domagg_check(slot[i] < n, SITE_SEGSCAN_PARTIAL)) return;
    typename Op::Acc v = Op::from_out(out[i]);
    if constexpr (std::is_same<Op, OpSumF32>::value) v.lo = lo[i];
    part[slot[i]] = v;
}

}  // namespace domagg
