// k_pairs.cuh -- small problems by their definition.
//
// The pipeline of a single small call is some forty dependent launches: at
// 4096 points per side its time (0.27 ms for m = 2, 0.9 ms for m = 3, 1.5 ms
// for m = 4) is launch latency and one or two busy multiprocessors.  The
// definition out(q) = F{ w(d) : d_i < q_i for all i } evaluated over all
// (d, q) pairs needs no order, no rank and no record: m compares, one select
// and one F per pair on every multiprocessor, 10 instructions for m = 2 with
// the float-float sum (2.0e6 pairs per us at 8000 x 8000; 4096 x 4096 take 16 us
// beside the statistics), and the call is one launch plus the flat-map
// statistics beside it (k_pair_stats).
#pragma once
#include "dev_common.cuh"
#include "k_points.cuh"

namespace domagg {

constexpr int PAIR_THREADS = 512;                  // two blocks per multiprocessor
constexpr int PAIR_GROUPS = 4;                     // groups of threads, each with the block's queries
constexpr int PAIR_LANES = PAIR_THREADS / PAIR_GROUPS;
constexpr int PAIR_QPT = 4;                        // queries per thread (registers)
constexpr u32 PAIR_QT = PAIR_LANES * PAIR_QPT;     // queries per block
constexpr u32 PAIR_STAGE = PAIR_THREADS;           // data staged in shared memory at a time
static_assert(PAIR_QT == PAIR_THREADS, "a thread per query joins the groups and the chunks");

// One launch over the small problems of a call.  A block takes a tile of
// PAIR_QT queries of one instance and a chunk of `dchunk` of its data; an
// instance with several chunks leaves its blocks' partials in `scr`, and the
// last block of a query tile to finish (ctr, self-resetting) combines them in
// chunk order, so float sums repeat bit for bit.
struct PairCall {
    Inst one;             // the only instance (tab == nullptr)
    const Inst* tab;      // device: the instances
    const u32* blk_inst;  // device: per block its instance
    const u32* blk_off;   // device: per instance its first block
    const u32* ctr_off;   // device: per instance its first query-tile counter
    const u64* scr_off;   // device: per instance its first partial (in Acc units)
    u32* ctr;
    void* scr;
    u32 dchunk;
    int negate;
    Ctl* ctl;
};

// w(d) joined into a query's running F if the datum's keys are within the
// query's bounds: the compares as one chain of predicates, then the predicated
// F (written out: compiled from the conditions, every coordinate took a
// second instruction of the same half-rate pipe; 15.5 -> 12 instructions per
// pair of the m = 3 float-float sum).
template <class Op, int M>
struct PairAcc;

template <int M>
__device__ __forceinline__ float pair_select_f32(const u32 (&k)[M], const u32 (&b)[M], float v) {
    float r;
    if constexpr (M == 1)
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tselp.f32 %0, %3, 0f00000000, p;\n\t}"
            : "=f"(r) : "r"(k[0]), "r"(b[0]), "f"(v));
    else if constexpr (M == 2)
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tsetp.le.and.u32 p, %3, %4, p;\n\t"
            "selp.f32 %0, %5, 0f00000000, p;\n\t}"
            : "=f"(r) : "r"(k[0]), "r"(b[0]), "r"(k[1]), "r"(b[1]), "f"(v));
    else if constexpr (M == 3)
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tsetp.le.and.u32 p, %3, %4, p;\n\t"
            "setp.le.and.u32 p, %5, %6, p;\n\tselp.f32 %0, %7, 0f00000000, p;\n\t}"
            : "=f"(r) : "r"(k[0]), "r"(b[0]), "r"(k[1]), "r"(b[1]), "r"(k[2]), "r"(b[2]), "f"(v));
    else
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tsetp.le.and.u32 p, %3, %4, p;\n\t"
            "setp.le.and.u32 p, %5, %6, p;\n\tsetp.le.and.u32 p, %7, %8, p;\n\t"
            "selp.f32 %0, %9, 0f00000000, p;\n\t}"
            : "=f"(r) : "r"(k[0]), "r"(b[0]), "r"(k[1]), "r"(b[1]), "r"(k[2]), "r"(b[2]), "r"(k[3]), "r"(b[3]), "f"(v));
    return r;
}
// acc = F(acc, v) under the chain's predicate, for the operators that are one
// instruction OPI (two for a 64-bit sum) on registers of constraint C.
#define DOMAGG_PAIR_STEP(OPI, C, acc, v)                                                                          \
    if constexpr (M == 1)                                                                                         \
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\t@p " OPI " %0, %0, %3;\n\t}"                         \
            : "+" C(acc) : "r"(k[0]), "r"(b[0]), C(v));                                                           \
    else if constexpr (M == 2)                                                                                    \
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tsetp.le.and.u32 p, %3, %4, p;\n\t"                   \
            "@p " OPI " %0, %0, %5;\n\t}"                                                                         \
            : "+" C(acc) : "r"(k[0]), "r"(b[0]), "r"(k[1]), "r"(b[1]), C(v));                                     \
    else if constexpr (M == 3)                                                                                    \
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tsetp.le.and.u32 p, %3, %4, p;\n\t"                   \
            "setp.le.and.u32 p, %5, %6, p;\n\t@p " OPI " %0, %0, %7;\n\t}"                                        \
            : "+" C(acc) : "r"(k[0]), "r"(b[0]), "r"(k[1]), "r"(b[1]), "r"(k[2]), "r"(b[2]), C(v));               \
    else                                                                                                          \
        asm("{\n\t.reg .pred p;\n\tsetp.le.u32 p, %1, %2;\n\tsetp.le.and.u32 p, %3, %4, p;\n\t"                   \
            "setp.le.and.u32 p, %5, %6, p;\n\tsetp.le.and.u32 p, %7, %8, p;\n\t@p " OPI " %0, %0, %9;\n\t}"       \
            : "+" C(acc)                                                                                          \
            : "r"(k[0]), "r"(b[0]), "r"(k[1]), "r"(b[1]), "r"(k[2]), "r"(b[2]), "r"(k[3]), "r"(b[3]), C(v))

template <int M>
struct PairAcc<OpSumI64, M> {
    static __device__ __forceinline__ void add(long long& a, const u32 (&k)[M], const u32 (&b)[M], long long v) {
        DOMAGG_PAIR_STEP("add.s64", "l", a, v);
    }
};
template <int M>
struct PairAcc<OpMaxI32, M> {
    static __device__ __forceinline__ void add(int& a, const u32 (&k)[M], const u32 (&b)[M], int v) {
        DOMAGG_PAIR_STEP("max.s32", "r", a, v);
    }
};
template <int M>
struct PairAcc<OpMinI32, M> {
    static __device__ __forceinline__ void add(int& a, const u32 (&k)[M], const u32 (&b)[M], int v) {
        DOMAGG_PAIR_STEP("min.s32", "r", a, v);
    }
};
template <int M>
struct PairAcc<OpMaxF32, M> {  // (max.f32 and min.f32 leave a NaN weight out, as fmaxf does)
    static __device__ __forceinline__ void add(float& a, const u32 (&k)[M], const u32 (&b)[M], float v) {
        DOMAGG_PAIR_STEP("max.f32", "f", a, v);
    }
};
template <int M>
struct PairAcc<OpMinF32, M> {
    static __device__ __forceinline__ void add(float& a, const u32 (&k)[M], const u32 (&b)[M], float v) {
        DOMAGG_PAIR_STEP("min.f32", "f", a, v);
    }
};
template <int M>
struct PairAcc<OpCount, M> {
    static __device__ __forceinline__ void add(u32& a, const u32 (&k)[M], const u32 (&b)[M], u32) {
        const u32 one = 1u;
        DOMAGG_PAIR_STEP("add.u32", "r", a, one);
    }
};
#undef DOMAGG_PAIR_STEP

// The running F of a thread's PAIR_QPT queries.
template <class Op, int M>
struct PairQueries {
    typename Op::Acc a[PAIR_QPT];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < PAIR_QPT; ++j) a[j] = Op::e();
    }
    // a datum of keys k; the first C of them are compared
    template <int C>
    __device__ __forceinline__ void add(const u32 (&k)[M], const u32 (&b)[PAIR_QPT][M], typename Op::Acc v) {
        u32 kc[C];
#pragma unroll
        for (int i = 0; i < C; ++i) kc[i] = k[i];
#pragma unroll
        for (int j = 0; j < PAIR_QPT; ++j) {
            u32 bc[C];
#pragma unroll
            for (int i = 0; i < C; ++i) bc[i] = b[j][i];
            PairAcc<Op, C>::add(a[j], kc, bc, v);
        }
    }
    __device__ __forceinline__ void settle() {}
    __device__ __forceinline__ typename Op::Acc get(int j) const { return a[j]; }
};
// Float-float sums take two queries per instruction (add.rn.f32x2: the same
// roundings, half the issue slots of the seven additions: 13.3 -> 9.1 instructions per pair
// for m = 2; then the half-rate compares and the two additions' lanes bind:
// 192 planned problems 241 -> 226 us).  The exact
// error of every addition goes to the low part; settle() renormalises.
__device__ __forceinline__ u64 f2_pack(float x, float y) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void f2_unpack(u64 v, float& x, float& y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ u64 f2_add(u64 x, u64 y) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return r;
}
__device__ __forceinline__ u64 f2_sub(u64 x, u64 y) {
    u64 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return r;
}
template <int M>
struct PairQueries<OpSumF32, M> {
    static_assert(PAIR_QPT % 2 == 0, "two queries per instruction");
    u64 hi[PAIR_QPT / 2], lo[PAIR_QPT / 2];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < PAIR_QPT / 2; ++j) hi[j] = lo[j] = 0ull;
    }
    template <int C>
    __device__ __forceinline__ void add(const u32 (&k)[M], const u32 (&b)[PAIR_QPT][M], ff v) {
        u32 kc[C];
#pragma unroll
        for (int i = 0; i < C; ++i) kc[i] = k[i];
#pragma unroll
        for (int j = 0; j < PAIR_QPT / 2; ++j) {
            u32 b0[C], b1[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                b0[i] = b[2 * j][i];
                b1[i] = b[2 * j + 1][i];
            }
            const u64 x = f2_pack(pair_select_f32<C>(kc, b0, v.hi), pair_select_f32<C>(kc, b1, v.hi));
            const u64 h = hi[j], t = f2_add(h, x), z = f2_sub(t, h);  // Knuth's TwoSum, as ff_two_sum
            lo[j] = f2_add(lo[j], f2_add(f2_sub(h, f2_sub(t, z)), f2_sub(x, z)));
            hi[j] = t;
        }
    }
    __device__ __forceinline__ ff get(int j) const {
        float h[2], l[2];
        f2_unpack(hi[j / 2], h[0], h[1]);
        f2_unpack(lo[j / 2], l[0], l[1]);
        return {h[j % 2], l[j % 2]};
    }
    __device__ __forceinline__ void settle() {
#pragma unroll
        for (int j = 0; j < PAIR_QPT / 2; ++j) {
            const ff x = ff_add(get(2 * j), ff{0.f, 0.f}), y = ff_add(get(2 * j + 1), ff{0.f, 0.f});
            hi[j] = f2_pack(x.hi, y.hi);
            lo[j] = f2_pack(x.lo, y.lo);
        }
    }
};

// A partial another block wrote (through the L2).
template <typename Acc>
__device__ __forceinline__ Acc pair_load(const Acc* p) {
    Acc v;
    if constexpr (sizeof(Acc) == 8) {
        const unsigned long long b = __ldcg(reinterpret_cast<const unsigned long long*>(p));
        memcpy(&v, &b, 8);
    } else {
        const u32 b = __ldcg(reinterpret_cast<const u32*>(p));
        memcpy(&v, &b, 4);
    }
    return v;
}

template <class Op, int WT>
__device__ __forceinline__ typename Op::Acc pair_weight(const void* dw, u32 i) {
    if constexpr (WT == 3) return Op::from_pay(0u);
    else if constexpr (WT == 1) return Op::from_w(reinterpret_cast<const u64*>(dw)[i]);
    else return Op::from_pay(reinterpret_cast<const u32*>(dw)[i]);
}

// Bound by instruction issue: per pair m compares (chained predicates), a
// select and F (7 additions for a float-float sum).  Four queries per thread
// share every staged datum's two broadcast reads; the block's four groups of
// threads hold the same 512 queries and take a quarter of every stage each,
// so that one wave of two blocks per multiprocessor covers a 4096 x 4096
// problem with 38 partials per query (one block per chunk of data and 128
// threads instead left 64 to 150, whose combination took longer than the
// pairs).
template <int M, class Op, int WT, bool F32>
__global__ __launch_bounds__(PAIR_THREADS, 2) void k_pairs(const __grid_constant__ PairCall C) {
    typedef typename Op::Acc Acc;
    constexpr int KW = M <= 2 ? 2 : 4;
    __shared__ __align__(16) u32 s_k[PAIR_STAGE][KW];
    __shared__ Acc s_v[PAIR_STAGE];
    __shared__ Acc s_join[PAIR_GROUPS][PAIR_QT];
    __shared__ u32 s_last;
    const u32 tid = threadIdx.x, grp = tid / PAIR_LANES, ln = tid % PAIR_LANES;
    const u32 s = C.tab ? __ldg(C.blk_inst + blockIdx.x) : 0u;
    const Inst& I = C.tab ? C.tab[s] : C.one;
    const u32 local = blockIdx.x - (C.tab ? __ldg(C.blk_off + s) : 0u);
    const u32 nD = I.nD, nQ = I.nQ, flags = I.flags;
    const u32 nsplit = max(1u, (nD + C.dchunk - 1u) / C.dchunk);
    const u32 tile = local / nsplit, split = local - tile * nsplit;
    const bool negate = C.negate != 0;
    bool nan = false;
    // a query's bound per coordinate: a datum counts if key <= bound for all.
    // Strictly below key 0 there is nothing: such a query is dead (its F is e).
    u32 bound[PAIR_QPT][M];
    u32 dead = 0;
    PairQueries<Op, M> acc;
    acc.clear();
#pragma unroll
    for (int j = 0; j < PAIR_QPT; ++j) {
        const u32 q = tile * PAIR_QT + (u32)j * PAIR_LANES + ln;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            u32 key = 0;
            if (q < nQ) key = coord_key<F32>(I.qco, q, M, i, negate, nan);
            const u32 strict = ((flags >> i) & 1u) ^ 1u;
            if (key < strict) dead |= 1u << j;
            bound[j][i] = key - strict;
        }
    }
    const u32 d0 = split * C.dchunk, d1 = min(nD, d0 + C.dchunk);
    for (u32 a = d0; a < d1; a += PAIR_STAGE) {
        const u32 n = min(PAIR_STAGE, d1 - a);
        __syncthreads();  // the previous stage is read
        if (tid < n) {
#pragma unroll
            for (int i = 0; i < M; ++i) s_k[tid][i] = coord_key<F32>(I.dco, a + tid, M, i, negate, nan);
            s_v[tid] = pair_weight<Op, WT>(I.dw, a + tid);
        }
        __syncthreads();
        const u32 per = (n + PAIR_GROUPS - 1u) / PAIR_GROUPS, x1 = min(n, (grp + 1u) * per);
#pragma unroll 4
        for (u32 x = grp * per; x < x1; ++x) {
            u32 kd[M];
            if constexpr (M <= 2) {
                const uint2 t = *reinterpret_cast<const uint2*>(s_k[x]);
                kd[0] = t.x;
                if constexpr (M == 2) kd[1] = t.y;
            } else {
                const uint4 t = *reinterpret_cast<const uint4*>(s_k[x]);
                kd[0] = t.x;
                kd[1] = t.y;
                kd[2] = t.z;
                if constexpr (M == 4) kd[3] = t.w;
            }
            const Acc v = s_v[x];
            acc.template add<M>(kd, bound, v);
        }
        acc.settle();
    }
    if (nan) atomicOr(&C.ctl->error, ERR_NAN);
    // join the groups: from here on a thread holds one query
#pragma unroll
    for (int j = 0; j < PAIR_QPT; ++j)
        s_join[grp][(u32)j * PAIR_LANES + ln] = (dead >> j) & 1u ? Op::e() : acc.get(j);
    __syncthreads();
    const u32 q = tile * PAIR_QT + tid;
    Acc r = s_join[0][tid];
#pragma unroll
    for (int g = 1; g < PAIR_GROUPS; ++g) r = Op::F(r, s_join[g][tid]);
    bool write = nsplit == 1u;
    if (nsplit > 1u) {
        Acc* scr = reinterpret_cast<Acc*>(C.scr) + (C.tab ? __ldg(C.scr_off + s) : 0ull) + q;
        u32* ctr = C.ctr + (C.tab ? __ldg(C.ctr_off + s) : 0u) + tile;
        if (q < nQ) scr[(u64)split * nQ] = r;
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(ctr, 1u) == nsplit - 1u ? 1u : 0u;
        __syncthreads();
        write = s_last != 0u;
        if (write) {
            __threadfence();
            if (tid == 0) *ctr = 0u;  // for the next launch
            r = Op::e();
            constexpr int B = 16;  // partials in flight
            for (u32 p = 0; p < nsplit; p += B) {
                Acc v[B];
#pragma unroll
                for (int e = 0; e < B; ++e)
                    v[e] = (q < nQ && p + e < nsplit) ? pair_load(scr + (u64)(p + e) * nQ) : Op::e();
#pragma unroll
                for (int e = 0; e < B; ++e) r = Op::F(r, v[e]);
            }
        }
    }
    if (write && q < nQ) reinterpret_cast<typename Op::Out*>(I.out)[q] = Op::to_out(r);
    // launched beside k_pair_stats (programmatic dependent launch): the
    // stream's next work has to find that kernel done as well
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The flat map's statistics of a small problem: per ranked coordinate the
// number of distinct values and rank digits, and the number of records
// sum_points prod_i |P(r_i)| (Sec. 5).  A cluster of blocks per (instance,
// ranked coordinate) holds the coordinate's keys in registers and sorts them
// (stable LSD radix sort, 8-bit digits; a digit that all keys share is left
// out): the blocks exchange their digit counts and scatter the items into
// each other's shared memory, two cluster barriers per digit.  Dense ranks
// come from the key changes, and the instance's last block adds up the
// products of its points' counts.  It runs beside k_pairs, which needs none of
// it; bound by the latency of the barriers and, with one block, by the issue
// of the digit matches (106 instructions per item and digit in all).  One
// problem takes eight blocks per coordinate (one block: 26 us at 8192 points,
// 80 at 16000, 117 at 21000, longer than the pairs); a batch, whose
// instances fill the chip, takes one.
// Up to 8192 points a cluster's blocks have 256 threads (fewer warps whose
// counts are scanned: 25 -> 22 us), else 1024.
constexpr int PSTAT_THREADS = 1024, PSTAT_FEW_THREADS = 256;
constexpr u32 PSTAT_CLUSTER = 8;                // blocks per coordinate of a single problem
constexpr u32 PSTAT_MAX = 24u * PSTAT_THREADS;  // points of a problem, at most (24 registers of keys in one block)
struct PairStatCall {
    Inst one;
    const Inst* tab;
    const u64* pt_off;   // device: per instance its first point of cnt (tab != nullptr)
    unsigned char* cnt;  // [total points * (M-1)], M >= 3: |P(r_i)| of every point
    u64 total;           // points of all instances
    u32* done;           // [instances]: finished blocks (self-resetting)
    int negate;
    Ctl* ctl;
};
template <int ITEMS, int T>
constexpr size_t pstat_smem() {  // two item buffers (keys, indices) and the warps' digit counts
    return (size_t)T * ITEMS * (ITEMS <= 16 ? 12 : 6) + (size_t)(T / 32) * (RADIX + 1) * 4;
}
__device__ __forceinline__ u32 cluster_rank() {
    u32 r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ u32 cluster_size() {
    u32 r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
// The address of `p` (this block's shared memory) in block `rank` of the cluster.
__device__ __forceinline__ u32 cluster_map(const void* p, u32 rank) {
    u32 a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_st32(u32 a, u32 v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_st16(u32 a, unsigned short v) {
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(v) : "memory");
}

template <int M, bool F32, int ITEMS, int T>
__global__ __launch_bounds__(T) void k_pair_stats(const __grid_constant__ PairStatCall C) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // every block of the cluster has to have started before another stores
    // into its shared memory: arrive here, wait behind the key loads
    cluster_arrive();
    constexpr int W = T / 32, R = M - 1;
    constexpr u32 PER = T / RADIX;  // threads per digit, eight warps' counts each
    static_assert(PER * 8 == W && (PER == 1 || PER == 4), "digit scan");
    constexpr u32 CAP = (u32)T * ITEMS;  // items of a block
    // the items of the next digit go to the other buffer: no barrier between
    // a block's reads and its peers' next writes (with more than 16 items,
    // one block only: a plain barrier and one buffer)
    constexpr u32 NB = ITEMS <= 16 ? 2u : 1u;
    extern __shared__ __align__(128) unsigned char smem[];
    u32* s_key = reinterpret_cast<u32*>(smem);                                        // [NB][CAP]
    unsigned short* s_idx = reinterpret_cast<unsigned short*>(s_key + NB * CAP);      // [NB][CAP]
    u32(*s_wh)[RADIX + 1] = reinterpret_cast<u32(*)[RADIX + 1]>(s_idx + NB * CAP);    // per warp: counts, positions
    __shared__ u32 s_ct[PSTAT_CLUSTER][RADIX];  // every block's digit counts
    __shared__ u32 s_chg[PSTAT_CLUSTER];        // every block's key changes
    __shared__ u32 s_tmp[W];
    __shared__ unsigned long long s_sum[W];
    __shared__ u32 s_last, s_end;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const u32 lt = lanemask_lt();
    const u32 rank = cluster_rank(), size = cluster_size();
    const u32 job = blockIdx.x / size;
    const u32 s = C.tab ? job / R : 0u;
    const int dim = (int)(job % R);
    const Inst& I = C.tab ? C.tab[s] : C.one;
    const u32 nQ = I.nQ, n = I.nD + nQ, all_items = CAP * size;
    const u64 off = (C.tab ? __ldg(C.pt_off + s) : 0ull) + C.total * (u64)dim;
    const u32 ns = (I.flags >> dim) & 1u;
    // item j of this thread is position p0 + 32 j of the cluster's; the
    // positions from n on hold pads (the largest key, and behind every point:
    // the sort is stable)
    const u32 l0 = (u32)warp * 32u * ITEMS + (u32)lane, p0 = rank * CAP + l0;
    u32 key[ITEMS];
    unsigned short idx[ITEMS];
    bool nan = false;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const u32 i = p0 + 32u * j;
        key[j] = 0xffffffffu;
        idx[j] = (unsigned short)i;
        if (i < n) {
            const bool q = i < nQ;
            key[j] = coord_key<F32>(q ? I.qco : I.dco, q ? i : i - nQ, M, dim, C.negate != 0, nan);
        }
    }
    if (nan) atomicOr(&C.ctl->error, ERR_NAN);
    cluster_wait();  // (the arrival at the kernel's start)
    u32 buf = 0;
#pragma unroll 1
    for (int sh = 0; sh < 32; sh += 8) {
        for (int x = tid; x < W * (RADIX + 1); x += T) (&s_wh[0][0])[x] = 0u;
        __syncthreads();
        unsigned short pos[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const u32 d = (key[j] >> sh) & 255u;
            const u32 peers = match_digit8(d, 0xffffffffu);
            const int leader = __ffs(peers) - 1;
            u32 old = 0;
            if (lane == leader) old = atomicAdd(&s_wh[warp][d], (u32)__popc(peers));
            pos[j] = (unsigned short)(__shfl_sync(0xffffffffu, old, leader) + (u32)__popc(peers & lt));
        }
        __syncthreads();
        const u32 d = (u32)tid / PER, part = (u32)tid % PER;
        u32 c[8], sum = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            c[w] = s_wh[part * 8u + w][d];
            sum += c[w];
        }
        // the block's count of the digit, to every block of the cluster
        u32 quad = sum;
        if (PER == 4) {
            quad += __shfl_xor_sync(0xffffffffu, quad, 1);
            quad += __shfl_xor_sync(0xffffffffu, quad, 2);
        }
        for (u32 r = part; r < size; r += PER) cluster_st32(cluster_map(&s_ct[rank][d], r), quad);
        cluster_sync();
        // the digit's count over the blocks, and over those before this one
        u32 tot = 0, mine = 0;
        for (u32 r = 0; r < size; ++r) {
            const u32 x = s_ct[r][d];
            if (r < rank) mine += x;
            tot += x;
        }
        u32 inc = part == PER - 1u ? tot : 0u;  // over the digits, one thread of each
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += x;
        }
        if (lane == 31) s_tmp[warp] = inc;
        // (a cluster-wide decision: every block has the same counts; the
        // blocks' next counts are ordered behind this read by the barriers
        // of the next digit's matches)
        if (__syncthreads_or(tot == all_items)) {
            cluster_sync();  // s_ct read by all before it is written again
            continue;        // one digit for all: the order stays
        }
        u32 before = inc - (part == PER - 1u ? tot : 0u);  // digits below, of this warp (in the digit's last thread)
        before = __shfl_sync(0xffffffffu, before, lane | (int)(PER - 1u));
        for (int w = 0; w < warp; ++w) before += s_tmp[w];
        u32 run = before + mine;
        if (PER == 4) {  // the digit's items in this block's warps before
            u32 pre = sum + __shfl_up_sync(0xffffffffu, sum, 1) * (part >= 1u ? 1u : 0u);
            const u32 two = __shfl_up_sync(0xffffffffu, pre, 2);
            if (part >= 2u) pre += two;
            run += pre - sum;
        }
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            s_wh[part * 8u + w][d] = run;
            run += c[w];
        }
        __syncthreads();
        if (NB == 2u) buf ^= 1u;
        u32* bk = s_key + buf * CAP;
        unsigned short* bi = s_idx + buf * CAP;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const u32 at = s_wh[warp][(key[j] >> sh) & 255u] + pos[j];
            if (domagg_check(at < all_items, SITE_SORT_LOCAL)) {
                const u32 r = at / CAP, x = at - r * CAP;
                cluster_st32(cluster_map(bk + x, r), key[j]);
                cluster_st16(cluster_map(bi + x, r), idx[j]);
            }
        }
        cluster_sync();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            key[j] = bk[l0 + 32u * j];
            idx[j] = bi[l0 + 32u * j];
        }
    }
    // dense ranks: key changes up to the position.  The keys once more in
    // shared memory (the last digits may have been left out), and the last
    // one to the next block
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) s_key[l0 + 32u * j] = key[j];
    if (tid == T - 1 && rank + 1u < size) cluster_st32(cluster_map(&s_end, rank + 1u), key[ITEMS - 1]);
    cluster_sync();
    u32 flags[ITEMS], changes = 0;  // per 32 positions, as a mask
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const u32 l = l0 + 32u * j, p = p0 + 32u * j;
        const u32 prev = l > 0u ? s_key[l - 1u] : s_end;
        flags[j] = __ballot_sync(0xffffffffu, p > 0u && p < n && prev != key[j]);
        changes += (u32)__popc(flags[j]);
    }
    if (lane == 0) s_tmp[warp] = changes;
    __syncthreads();
    u32 before = 0, all = 0;
    for (int w = 0; w < W; ++w) {
        const u32 x = s_tmp[w];
        if (w < warp) before += x;
        all += x;
    }
    if ((u32)tid < size) cluster_st32(cluster_map(&s_chg[rank], (u32)tid), all);
    cluster_sync();  // (the last access to other blocks' shared memory lies before it)
    all = 0;
    for (u32 r = 0; r < size; ++r) {
        const u32 x = s_chg[r];
        if (r < rank) before += x;
        all += x;
    }
    const u32 U = (all + 1u) << ns;  // (a non-strict coordinate: 2r for data, 2r + 1 for queries)
    const u32 bits = U <= 1u ? 0u : 32u - __clz(U - 1u), mask = low_mask(bits);
    unsigned long long sum = 0, sum_q = 0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const u32 p = p0 + 32u * j;
        const u32 r = before + (u32)__popc(flags[j] & (lt | (1u << lane)));
        before += (u32)__popc(flags[j]);
        const bool q = idx[j] < nQ;
        const u32 lr = ns ? 2u * r + (q ? 1u : 0u) : r;
        const u32 c = p < n ? (u32)__popc((q ? lr : ~lr) & mask) : 0u;
        if constexpr (R == 1) sum += c;
        else if (p < n) C.cnt[off + idx[j]] = (unsigned char)c;
    }
    if (tid == 0 && rank == 0u) {
        C.ctl->pair_U[M - 1][dim] = U;
        C.ctl->pair_b[M - 1][dim] = bits;
    }
    if constexpr (R > 1) {
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(C.done + s, 1u) == (u32)R * size - 1u ? 1u : 0u;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (tid == 0) C.done[s] = 0u;
        const u64 o0 = C.tab ? __ldg(C.pt_off + s) : 0ull;
#pragma unroll 4
        for (u32 i = (u32)tid; i < n; i += T) {
            u32 c = 1u;
#pragma unroll
            for (int e = 0; e < R; ++e) c *= (u32)__ldcg(C.cnt + o0 + C.total * (u64)e + i);
            sum += c;
            if (R == 3 && i < nQ) sum_q += c;
        }
    }
    for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_sum[warp] = sum;
    __syncthreads();
    if (tid == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < W; ++w) t += s_sum[w];
        if (t) atomicAdd(&C.ctl->pair_T[M - 1], t);  // (never reset: the host takes differences)
    }
    if constexpr (R == 3) {
        for (int o = 16; o >= 1; o >>= 1) sum_q += __shfl_xor_sync(0xffffffffu, sum_q, o);
        if (lane == 0 && sum_q) atomicAdd(&C.ctl->pair_Tq, sum_q);
    }
}

}  // namespace domagg
