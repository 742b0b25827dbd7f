// k_group3.cuh -- the deep first-rank levels of m = 3, by pairs per group.
//
// For m = 3 a record of first-rank level lv is keyed by the node r0 >> (lv+1)
// of the first rank refined by a node of the second rank (Sec. 5).  As for
// m = 2 (k_group.cuh) the points, in the order of the last coordinate, are
// sorted stably by their group g = r0 >> gS, here with the role as one more
// key bit: a group's data come first, then its queries, each in the order of
// the last coordinate.  Two points of one group whose first ranks differ do so
// first at a bit below gS, so the records of the levels lv < gS reach exactly
// the pairs (datum, query) of one group with r0(d) < r0(q), r1(d) < r1(q) and
// an earlier position (Lemma 1, for each coordinate): a query's F over these
// levels is F over those pairs, and this kernel takes it from the pairs
// themselves -- three compares, a select and F per pair (PairAcc), no node, no
// split and no scan.
//
// Bound by instruction issue, on the half-rate pipe of the compares and the
// select above all (issue active 64 %); a stage of data that lies wholly before
// the tile's queries needs no third compare.
// A group of c points costs c / 8 pairs per point (half of its points are
// data, half queries, and a query meets the data before it only), so groups of
// 4096 ranks (5e3 points at 2^21 per side) cost 640 pairs per point against
// the 13-14 second-rank level walks at each of 12 first-rank levels that did
// the same in shared memory before (one CTA per group: 2.4 ms at 2^21 per
// side and 0.6 ms for a single group of 8e3 points; by pairs 1.3 ms and
// 0.06).  A wider group would double the pairs and save one level above
// (k_items.cuh, or records in HBM), about what it costs; narrower ones
// measured slower (2^21 per side 7.6 ms; groups of half the width 8.5).
#pragma once
#include "k_group.cuh"
#include "k_pairs.cuh"

namespace domagg {

constexpr u32 G3_QT = PAIR_QT;  // queries per block
// Points of a group, at most: a larger one (heavy ties) sends its levels
// through HBM (k_group_plan flags it).
constexpr u32 G3_CAP = 10240;
// Points of a group on average, at most, in a call over N points: groups of
// 4096 ranks, fewer where there are few points, so that the query tiles still
// cover the chip (1e5 per side: 677 us with N / 64, 773 with N / 512).  No
// limit of its own (8192 ranks, a level of records less) where room for
// records is short (a workspace that is capped or fixed, and calls that come
// near the limit of 2^32 records) and for a shard.
__host__ __device__ constexpr u32 g3_avg(u64 N, bool tight, bool items) {
    const u64 c = N / 64u;
    if (tight || (!items && N > (1ull << 24))) return 0xffffffffu;
    return c >= 7168u ? 7168u : (c <= 1024u ? 1024u : (u32)c);
}

// The deep levels of every group of the instances that go by pairs (see the
// file comment).  Persistent
// blocks take (query tile, group) pairs from a counter, a group's last tiles
// (the most data before them) first.  Inputs: the group-sorted points gv (per
// instance in buffer gv0 or gv1, by the parity of the group sort's passes):
// (rank | QUERY_BIT) << 32 | the point's position x in the order of the last
// coordinate; pr1 (second ranks) and pw (weights) by x.  Writes gacc[x] = F
// over the query's partial results of the levels below gS, as a partial (read
// in that order by the per-query reduction).
template <class Op, int WT>
__global__ __launch_bounds__(PAIR_THREADS, 2) void k_group3(const Inst* __restrict__ inst, int k,
                                                            const u32* __restrict__ gslot_off,
                                                            const u32* __restrict__ rstart,
                                                            const u64* __restrict__ gv0, const u64* __restrict__ gv1,
                                                            const u32* __restrict__ pr1,
                                                            const typename Op::W* __restrict__ pw,
                                                            typename Op::Part* __restrict__ gacc, Ctl* ctl,
                                                            int launch_idx) {
    typedef typename Op::Acc Acc;
    __shared__ __align__(16) u32 s_k[PAIR_STAGE][4];  // first rank, second rank, position
    __shared__ Acc s_v[PAIR_STAGE];
    __shared__ Acc s_join[PAIR_GROUPS][PAIR_QT];
    __shared__ u32 s_unit;
    const u32 tid = threadIdx.x, grp = tid / PAIR_LANES, ln = tid % PAIR_LANES;
    const u32 total = __ldg(gslot_off + k);
    constexpr u32 tiles_max = (G3_CAP + G3_QT - 1u) / G3_QT;
    for (;;) {
        __syncthreads();  // s_unit and the shared arrays of the previous unit are read
        if (tid == 0) s_unit = atomicAdd(&ctl->tile_ctr[launch_idx], 1u);
        __syncthreads();
        const u32 unit = s_unit;
        if (unit >= total * tiles_max) break;
        const u32 tile = tiles_max - 1u - unit / total, slot = unit % total;
        const int s = upper_index(gslot_off, k + 1, slot);
        const Inst& I = inst[s];
        const u32 g = I.shard + (slot - __ldg(gslot_off + s)) * max(I.nshards, 1u);
        const u32 gS = I.gS, ns = I.flags & 1u;
        const u32 us = gS - ns, Uu = ns ? I.U[0] / 2u : I.U[0];
        const u32* rs = rstart + I.pt_off + (u32)s;
        const u32 a = __ldg(rs + (g << us)), n = __ldg(rs + min((g + 1u) << us, Uu)) - a;
        const bool odd = ((I.b[0] - gS + 1u + RADIX_BITS - 1) / RADIX_BITS) & 1u;
        const u64* __restrict__ gv = (odd ? gv1 : gv0) + I.pt_off + a;
        if (n > G3_CAP) {  // too many pairs: its levels go through HBM
            if (tile == 0u) group_unit_parts<Op>(gv, n, I, gacc);
            continue;
        }
        if (n <= tile * G3_QT) continue;
        // the group's data, then its queries: where they meet, by two rounds
        // of counting the data among up to PAIR_THREADS positions
        const u32 step = (n + PAIR_THREADS - 1u) / PAIR_THREADS;
        const u32 c1 = (u32)__syncthreads_count(tid * step < n && !((u32)(gv[min(tid * step, n - 1u)] >> 32) & QUERY_BIT));
        const u32 at = (c1 ? c1 - 1u : 0u) * step;
        const u32 c2 = (u32)__syncthreads_count(c1 && tid < step && at + tid < n &&
                                                !((u32)(gv[min(at + tid, n - 1u)] >> 32) & QUERY_BIT));
        const u32 nd = at + c2, nq = n - nd;
        if (nq <= tile * G3_QT) continue;
        const u64* __restrict__ gq = gv + nd;
        const u32 b1 = I.b[1], m1 = low_mask(b1), np = I.nD + I.nQ;
        // a datum counts if every key is at most the query's bound
        u32 bound[PAIR_QPT][3];
        u32 dead = 0;
        PairQueries<Op, 3> acc;
        acc.clear();
#pragma unroll
        for (int j = 0; j < PAIR_QPT; ++j) {
            const u32 q = tile * G3_QT + (u32)j * PAIR_LANES + ln;
            u32 r = 0, x = 0, r1 = 0;
            if (q < nq) {
                const u64 v = gq[q];
                r = (u32)(v >> 32) & ~QUERY_BIT;
                x = (u32)v;
                if (domagg_check(x - I.pt_off < np, SITE_GROUP_OUT)) r1 = __ldg(pr1 + x) & m1;
            }
            if (r == 0u || r1 == 0u || x == 0u) dead |= 1u << j;
            bound[j][0] = r - 1u;
            bound[j][1] = r1 - 1u;
            bound[j][2] = x - 1u;
        }
        // the tile's first and last query
        const u32 xmin = (u32)gq[tile * G3_QT], xmax = (u32)gq[min(nq, (tile + 1u) * G3_QT) - 1u];
        for (u32 d0 = 0; d0 < nd; d0 += PAIR_STAGE) {
            const u32 m = min(PAIR_STAGE, nd - d0);
            __syncthreads();  // the previous stage is read
            if (tid < m) {
                const u64 v = gv[d0 + tid];
                const u32 x = (u32)v;
                const bool ok = domagg_check(x - I.pt_off < np, SITE_GROUP_OUT);
                s_k[tid][0] = (u32)(v >> 32) & ~QUERY_BIT;
                s_k[tid][1] = ok ? __ldg(pr1 + x) & m1 : 0xffffffffu;
                s_k[tid][2] = x;
                if constexpr (WT == 3) s_v[tid] = Op::from_pay(0u);
                else if constexpr (Op::GATHER) s_v[tid] = ok ? Op::from_w(__ldg(pw + x)) : Op::e();
                else s_v[tid] = ok ? Op::from_pay((u32)__ldg(pw + x)) : Op::e();
            }
            __syncthreads();
            if (s_k[0][2] > xmax) break;  // every datum from here on lies behind the tile's queries
            const u32 per = (m + PAIR_GROUPS - 1u) / PAIR_GROUPS, x1 = min(m, (grp + 1u) * per);
            if (s_k[m - 1u][2] < xmin) {  // the whole stage lies before the tile: no position to compare
#pragma unroll 4
                for (u32 x = grp * per; x < x1; ++x) {
                    const uint4 t = *reinterpret_cast<const uint4*>(s_k[x]);
                    const u32 kd[3] = {t.x, t.y, t.z};
                    acc.template add<2>(kd, bound, s_v[x]);
                }
            } else {
#pragma unroll 4
                for (u32 x = grp * per; x < x1; ++x) {
                    const uint4 t = *reinterpret_cast<const uint4*>(s_k[x]);
                    const u32 kd[3] = {t.x, t.y, t.z};
                    acc.template add<3>(kd, bound, s_v[x]);
                }
            }
            acc.settle();
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PAIR_QPT; ++j)
            s_join[grp][(u32)j * PAIR_LANES + ln] = (dead >> j) & 1u ? Op::e() : acc.get(j);
        __syncthreads();
        const u32 q = tile * G3_QT + tid;
        if (q < nq) {
            Acc r = s_join[0][tid];
#pragma unroll
            for (int j = 1; j < PAIR_GROUPS; ++j) r = Op::F(r, s_join[j][tid]);
            const u32 x = (u32)gq[q];
            if (domagg_check(x - I.pt_off < np, SITE_GROUP_OUT)) gacc[x] = Op::to_part(r);
        }
    }
}

}  // namespace domagg
