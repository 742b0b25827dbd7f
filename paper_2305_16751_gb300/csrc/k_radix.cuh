// k_radix.cuh -- segmented, stable LSD radix sort of (key, value) pairs.
//
// This is the sort primitive of the paper (Definition "Sort", Sec. 2.2) as a
// GPU "onesweep" sort: one histogram pass computes the digit counts of every
// pass per segment, then every pass is one kernel whose blocks take ranges of
// whole tiles and rank a tile's keys locally.  A range's global positions come
// from the histogram (first pass), from a count and a scan of their own (many
// ranges: k_range_count, k_range_bases) or from a decoupled look-back over the
// ranges before it.  Segments (problem instances of a batch) are sorted
// independently: ranges never straddle a segment and the look-back chains stop
// at the segment's first range.  Stability (items with equal
// digits keep their order) is what lets the pipeline pre-order points by the
// last coordinate and then sort records by node key only (Sec. 5).
#pragma once
#include <type_traits>

#include "dev_common.cuh"

namespace domagg {

constexpr int RADIX_BITS = 8;
constexpr int RADIX = 1 << RADIX_BITS;

template <typename K>
__device__ __forceinline__ u32 digit_of(K k, K keymask, int shift) {
    return (u32)((k & keymask) >> shift) & (u32)(RADIX - 1);
}

// Locates tile t: its segment and the half-open item range [start, end).
struct TileLoc {
    int seg;
    u32 seg_begin, seg_end, start, end;
    bool first;
};
template <int TILE>
__device__ __forceinline__ TileLoc locate_tile(u32 t, const u32* seg_off, const u32* tile_off, int nseg) {
    TileLoc L;
    L.seg = upper_index(tile_off, nseg + 1, t);
    L.seg_begin = __ldg(seg_off + L.seg);
    L.seg_end = __ldg(seg_off + L.seg + 1);
    u32 first_tile = __ldg(tile_off + L.seg);
    L.start = L.seg_begin + (t - first_tile) * (u32)TILE;
    L.end = min(L.start + (u32)TILE, L.seg_end);
    L.first = (t == first_tile);
    return L;
}

// Locates range r of `range_items` items: its segment and [start, end).
__device__ __forceinline__ TileLoc locate_range(u32 r, const u32* seg_off, const u32* range_off, int nseg,
                                                u32 range_items) {
    TileLoc L;
    L.seg = upper_index(range_off, nseg + 1, r);
    L.seg_begin = __ldg(seg_off + L.seg);
    L.seg_end = __ldg(seg_off + L.seg + 1);
    const u32 first = __ldg(range_off + L.seg);
    L.start = L.seg_begin + (r - first) * range_items;
    L.end = min(L.start + range_items, L.seg_end);
    L.first = (r == first);
    return L;
}

// Digit histograms of all passes, per segment: hist[(seg*npass + p)*RADIX + d].
// One block per range of `range_items` items (ranges never straddle a
// segment), per-warp counts in shared memory.  With seg_bits, a segment only
// counts the passes its keys have digits for (the others skip it).
template <typename K>
__global__ __launch_bounds__(256) void k_radix_hist(const K* __restrict__ keys, const u32* __restrict__ seg_off,
                                                    const u32* __restrict__ range_off, int nseg, u32 range_items,
                                                    int npass, int shift0, K keymask, u32* __restrict__ hist,
                                                    u32* __restrict__ range_cnt0,
                                                    const u32* __restrict__ seg_bits) {
    extern __shared__ u32 sh_hist[];  // [8 warps][npass][RADIX]
    const u32 r = blockIdx.x;
    if (r >= __ldg(range_off + nseg)) return;
    const u32 warp = threadIdx.x >> 5;
    for (int x = threadIdx.x; x < 8 * npass * RADIX; x += 256) sh_hist[x] = 0;
    __syncthreads();
    const TileLoc L = locate_range(r, seg_off, range_off, nseg, range_items);
    const int sbits = seg_bits ? (int)__ldg(seg_bits + L.seg) : 0;
    const int np = seg_bits ? min(npass, (sbits + RADIX_BITS - 1) / RADIX_BITS) : npass;
    u32* wh = sh_hist + warp * npass * RADIX;
    for (u32 base = L.start; base < L.end; base += 256u * 8u) {
        K kk[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const u32 x = base + (u32)j * 256u + threadIdx.x;
            kk[j] = x < L.end ? keys[x] : K(0);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (base + (u32)j * 256u + threadIdx.x < L.end)
                for (int p = 0; p < np; ++p)
                    atomicAdd(wh + p * RADIX + digit_of(kk[j], keymask, shift0 + p * RADIX_BITS), 1u);
        }
    }
    __syncthreads();
    u32* gh = hist + (u64)L.seg * npass * RADIX;
    for (int x = threadIdx.x; x < npass * RADIX; x += 256) {
        u32 c = 0;
        for (int w = 0; w < 8; ++w) c += sh_hist[w * npass * RADIX + x];
        if (c) atomicAdd(gh + x, c);
        if (range_cnt0 && x < RADIX) range_cnt0[(u64)r * RADIX + x] = c;  // this range's first-pass counts
    }
}

// Digit counts of every range for one pass (the first pass takes them from
// k_radix_hist): range_cnt[r*RADIX + d].
template <typename K>
__global__ __launch_bounds__(256) void k_range_count(const K* __restrict__ keys, const u32* __restrict__ seg_off,
                                                     const u32* __restrict__ range_off, int nseg, u32 range_items,
                                                     int shift, K keymask, u32* __restrict__ range_cnt) {
    __shared__ u32 s_wh[8][RADIX];
    const u32 r = blockIdx.x;
    if (r >= __ldg(range_off + nseg)) return;
    u32* wh = s_wh[threadIdx.x >> 5];
    for (int x = threadIdx.x; x < 8 * RADIX; x += 256) (&s_wh[0][0])[x] = 0u;
    __syncthreads();
    const TileLoc L = locate_range(r, seg_off, range_off, nseg, range_items);
    for (u32 base = L.start; base < L.end; base += 256u * 8u) {
        K kk[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const u32 x = base + (u32)j * 256u + threadIdx.x;
            kk[j] = x < L.end ? keys[x] : K(0);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (base + (u32)j * 256u + threadIdx.x < L.end) atomicAdd(wh + digit_of(kk[j], keymask, shift), 1u);
    }
    __syncthreads();
    u32 c = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) c += s_wh[w][threadIdx.x];
    range_cnt[(u64)r * RADIX + threadIdx.x] = c;
}

// Global position of every (range, digit): the digit's start in the segment
// (digit_off of the pass) plus the counts of the segment's earlier ranges.
// In place over the per-range counts.  Grid (segment, group of 32 digits);
// the WARPS warps of a block split the segment's ranges into slices (lane =
// digit): slice sums, an exclusive scan of them in shared memory, then the
// running bases.  32 warps for few segments of many ranges, one for many
// segments of few.
// With hist (the first pass) the block first scans the segment's histograms
// of all passes into digit_off, its 32 digits of each.
template <int WARPS>
__global__ __launch_bounds__(WARPS * 32) void k_range_bases(const u32* __restrict__ range_off, u32* digit_off,
                                                            int npass, u32* __restrict__ range_cnt,
                                                            const u32* __restrict__ hist,
                                                            const u32* __restrict__ seg_off) {
    __shared__ u32 s_sum[WARPS][33];
    __shared__ u32 s_d0[32];
    const int seg = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = blockIdx.y * 32 + lane;
    const u32 r0 = __ldg(range_off + seg), r1 = __ldg(range_off + seg + 1);
    const u32 n = r1 - r0, per = (n + WARPS - 1) / WARPS;
    if (hist) {
        const u32 base = __ldg(seg_off + seg);
        for (int p = warp; p < npass; p += WARPS) {
            const u32* h = hist + ((u64)seg * npass + p) * RADIX + lane * 8;
            u32 v[8], sum = 0;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                v[e] = h[e];
                sum += v[e];
            }
            u32 inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += x;
            }
            u32 ex = base + inc - sum;
            if (lane / 4 == (int)blockIdx.y) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    digit_off[((u64)seg * npass + p) * RADIX + lane * 8 + e] = ex;
                    if (p == 0) s_d0[(lane & 3) * 8 + e] = ex;
                    ex += v[e];
                }
            }
        }
        __syncthreads();
    }
    if (n == 0u) return;
    const u32 a = r0 + min(n, (u32)warp * per), b = r0 + min(n, (u32)(warp + 1) * per);
    u32 run = hist ? s_d0[lane] : digit_off[(u64)seg * npass * RADIX + d];
    if (WARPS > 1) {
        u32 sum = 0;
        for (u32 r = a; r < b; r += 16) {  // 16 loads in flight
            u32 c[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) c[i] = r + i < b ? range_cnt[(u64)(r + i) * RADIX + d] : 0u;
#pragma unroll
            for (int i = 0; i < 16; ++i) sum += c[i];
        }
        s_sum[warp][lane] = sum;
        __syncthreads();
        for (int w = 0; w < warp; ++w) run += s_sum[w][lane];
    }
    for (u32 r = a; r < b; r += 16) {
        u32 c[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) c[i] = r + i < b ? range_cnt[(u64)(r + i) * RADIX + d] : 0u;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (r + i < b) range_cnt[(u64)(r + i) * RADIX + d] = run;
            run += c[i];
        }
    }
}

// Exclusive scan of every (segment, pass) histogram plus the segment start:
// digit_off[(seg*npass + p)*RADIX + d] = global position of digit d's first item.
static __global__ __launch_bounds__(RADIX) void k_radix_offsets(const u32* __restrict__ hist, const u32* __restrict__ seg_off,
                                                         int npass, u32* __restrict__ digit_off) {
    __shared__ u32 warp_sum[RADIX / 32];
    const int sp = blockIdx.x, seg = sp / npass;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u32 v = hist[(u64)sp * RADIX + threadIdx.x];
    u32 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        u32 n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    u32 add = 0;
    for (int w = 0; w < warp; ++w) add += warp_sum[w];
    digit_off[(u64)sp * RADIX + threadIdx.x] = __ldg(seg_off + seg) + add + inc - v;
}

// Items per thread of a onesweep tile: ONESWEEP_TILE_BYTES of (key, value)
// pairs per tile.
#ifndef ONESWEEP_TILE_BYTES
#define ONESWEEP_TILE_BYTES 32768
#endif
template <typename K, typename V>
__host__ __device__ constexpr int onesweep_items() {
    return ONESWEEP_TILE_BYTES / 256 / (int)(sizeof(K) + sizeof(V));
}
constexpr int ONESWEEP_THREADS = 256;
#ifndef ONESWEEP_MIN_CTAS
#define ONESWEEP_MIN_CTAS 3
#endif

// Shared memory: the tile in digit order, the warps' digit counts (then first
// positions), per digit the global position of tile position 0 and the next
// global position.
template <typename K, typename V>
struct OnesweepSmem {
    static constexpr int WARPS = ONESWEEP_THREADS / 32;
    static constexpr int TILE = ONESWEEP_THREADS * onesweep_items<K, V>();
    static constexpr size_t KEYS = 0;
    static constexpr size_t VALS = KEYS + (size_t)TILE * sizeof(K);
    static constexpr size_t WHIST = (VALS + (size_t)TILE * sizeof(V) + 15) & ~(size_t)15;
    static constexpr size_t GDST = WHIST + (size_t)WARPS * RADIX * 4;
    static constexpr size_t RUN = GDST + RADIX * 4;
    static constexpr size_t TOTAL = RUN + RADIX * 4;
};

template <typename K, typename V>
__host__ __device__ constexpr size_t onesweep_smem() {
    return OnesweepSmem<K, V>::TOTAL;
}

// One LSD pass: stable scatter of every segment by digit `pass`.
//
// Persistent CTAs claim ranges of consecutive tiles from a global counter,
// in increasing order.  For a range the CTA
//   1. counts its digits (one read of the keys),
//   2. publishes the count and runs one decoupled look-back over the earlier
//      ranges of the segment (bounded waits), which gives the global position
//      of the range's first item of every digit,
//   3. takes the range tile by tile: keys and values into registers (warp w
//      holds consecutive items, coalesced), the rank of every item among its
//      warp's items of the same digit (8-ballot match), the tile in digit
//      order through shared memory, and coalesced stores at the running
//      global position of every digit.
// There is no inter-CTA wait inside a range; the look-back runs once per
// range (tens of thousands of items), not once per tile.
//
// Bound by instruction issue, on the half-rate pipe of the digit match above
// all (110 instructions per item without a look-back), and by the tile's
// barriers.  Keys and values wait in registers and a tile is staged in shared
// memory once, in digit order; with the ranges' positions from k_range_count
// a pass over 6.3e6 pairs of 4 + 4 bytes takes 45 us instead of 69 (with TMA
// double buffers and the look-back), over 2^25 pairs 0.22 ms instead of 0.28.
// Three CTAs of 16 items per thread: four spill (64 registers; 2.65 instead
// of 2.35 ms over the point sorts at 2^25), 12 items move more, shorter runs.
//
// IOTA: the values are the items' own global indices (first pass of a sort
// that returns a permutation); `vin` is not read.
// STABLE = false (the first pass of the dense-rank sorts, where only the
// sorted key sequence matters) ranks with one shared-memory atomic per item
// instead of the digit match: equal digits keep the order in which the
// hardware serves a warp's atomics, which nothing documents, so every later
// pass is stable (7.85 -> 8.0 ms for a forward of 2^24 points per side).
// range_base (may be null) holds every range's global position per
// digit, which replaces the range's count and look-back.
template <typename K, typename V, bool IOTA, bool STABLE>
__global__ __launch_bounds__(ONESWEEP_THREADS, ONESWEEP_MIN_CTAS) void k_onesweep(
    const K* __restrict__ kin, const V* __restrict__ vin, K* __restrict__ kout, V* __restrict__ vout,
    const u32* __restrict__ seg_off, const u32* __restrict__ range_off, int nseg, u32 range_items,
    const u32* __restrict__ seg_bits, const u32* __restrict__ range_base, const u32* __restrict__ digit_off,
    int npass, int pass, int shift, K keymask, u64* status, Ctl* ctl, int launch_idx) {
    constexpr int THREADS = ONESWEEP_THREADS, ITEMS = onesweep_items<K, V>();
    constexpr int TILE = THREADS * ITEMS, WARPS = THREADS / 32;
    typedef OnesweepSmem<K, V> SM;
    static_assert(SM::TILE == TILE && THREADS == RADIX && ITEMS % 2 == 0, "one thread per digit");
    extern __shared__ __align__(128) unsigned char smem[];
    K* s_k = reinterpret_cast<K*>(smem + SM::KEYS);
    V* s_v = reinterpret_cast<V*>(smem + SM::VALS);
    u32* s_wh = reinterpret_cast<u32*>(smem + SM::WHIST);  // [WARPS][RADIX]
    u32* s_gdst = reinterpret_cast<u32*>(smem + SM::GDST);
    u32* s_run = reinterpret_cast<u32*>(smem + SM::RUN);
    __shared__ u32 s_scan[WARPS];
    __shared__ u32 s_range;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const u32 nranges = __ldg(range_off + nseg);
    const u32 lt = lanemask_lt();
    const u32 epoch = ctl->epoch_base + (u32)launch_idx;
    u32* wh = s_wh + warp * RADIX;
    auto clear_counts = [&]() {  // the warp's own row
#pragma unroll
        for (int x = 0; x < RADIX / 32 / 4; ++x)
            reinterpret_cast<uint4*>(wh)[x * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
    };

    // one tile of n items from a (FULL: n == TILE)
    auto do_tile = [&](auto full, u32 a, u32 n, u32 seg_begin, u32 seg_len) {
        constexpr bool FULL = decltype(full)::value;
        const u32 w0 = (u32)warp * 32u * ITEMS + (u32)lane;  // item i of this lane: tile position w0 + 32 i
        K key[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const u32 x = w0 + 32u * i;
            key[i] = FULL || x < n ? kin[a + x] : K(0);
        }
        clear_counts();
        __syncwarp();
        u32 rk[ITEMS / 2];  // rank among the warp's items of the digit, two per word
#pragma unroll
        for (int i0 = 0; i0 < ITEMS; i0 += 2) {
            u32 m[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int i = i0 + e;
                const u32 d = digit_of(key[i], keymask, shift);
                const bool valid = FULL || w0 + 32u * i < n;
                if constexpr (STABLE) m[e] = match_digit8(d, FULL ? 0xffffffffu : __ballot_sync(0xffffffffu, valid));
                else m[e] = valid ? atomicAdd(wh + d, 1u) : 0u;
            }
            if constexpr (STABLE) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = i0 + e;
                    const u32 d = digit_of(key[i], keymask, shift);
                    const bool valid = FULL || w0 + 32u * i < n;
                    // every lane reads the digit's count before its first lane advances it
                    const u32 below = (u32)__popc(m[e] & lt), cnt = wh[d];
                    __syncwarp();
                    if (valid && below == 0u) wh[d] = cnt + (u32)__popc(m[e]);
                    __syncwarp();
                    m[e] = cnt + below;
                }
            }
            rk[i0 / 2] = m[0] | (m[1] << 16);
        }
        V val[ITEMS];  // (in flight over the scan of the counts)
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const u32 x = w0 + 32u * i;
            if constexpr (IOTA) val[i] = (V)(a + x);
            else val[i] = FULL || x < n ? vin[a + x] : V(0);
        }
        __syncthreads();  // the warps' counts are known; the previous tile is written out
        {
            const int d = tid;
            u32 c[WARPS], tot = 0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                c[w] = s_wh[w * RADIX + d];
                tot += c[w];
            }
            u32 inc = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 x = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += x;
            }
            if (lane == 31) s_scan[warp] = inc;
            __syncthreads();
            u32 ex = inc - tot;
#pragma unroll
            for (int w = 0; w < WARPS - 1; ++w) ex += w < warp ? s_scan[w] : 0u;
            const u32 run = s_run[d];
            s_gdst[d] = run - ex;
            s_run[d] = run + tot;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                s_wh[w * RADIX + d] = ex;
                ex += c[w];
            }
        }
        __syncthreads();  // first positions per (warp, digit)
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (FULL || w0 + 32u * i < n) {
                const u32 pos = wh[digit_of(key[i], keymask, shift)] + ((rk[i / 2] >> (16 * (i & 1))) & 0xffffu);
                if (DOMAGG_GUARD(pos < n, SITE_SORT_LOCAL)) {
                    s_k[pos] = key[i];
                    s_v[pos] = val[i];
                }
            }
        }
        __syncthreads();  // the tile in digit order
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const u32 x = (u32)tid + (u32)i * THREADS;
            if (FULL || x < n) {
                const K k = s_k[x];
                const V v = s_v[x];
                const u32 dst = s_gdst[digit_of(k, keymask, shift)] + x;
                if (domagg_check(dst - seg_begin < seg_len, SITE_SORT_SCATTER)) {  // only fails after a timed-out wait
                    kout[dst] = k;
                    vout[dst] = v;
                }
            }
        }
    };

    for (;;) {
        __syncthreads();  // the previous range is written out
        if (tid == 0) s_range = atomicAdd(&ctl->tile_ctr[launch_idx], 1u);
        __syncthreads();
        const u32 r = s_range;
        if (r >= nranges) break;
        const TileLoc L = locate_range(r, seg_off, range_off, nseg, range_items);
        // a segment whose keys have fewer digits is already in place
        if (seg_bits && (u32)pass * RADIX_BITS >= __ldg(seg_bits + L.seg)) continue;
        if (range_base) {
            s_run[tid] = __ldg(range_base + (u64)r * RADIX + tid);
        } else {
            // 1. digit counts of the range
            clear_counts();
            __syncwarp();
            for (u32 base = L.start; base < L.end; base += (u32)THREADS * 8u) {
                K kk[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const u32 x = base + (u32)j * THREADS + (u32)tid;
                    kk[j] = x < L.end ? kin[x] : K(0);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (base + (u32)j * THREADS + (u32)tid < L.end) atomicAdd(wh + digit_of(kk[j], keymask, shift), 1u);
            }
            __syncthreads();
            u32 cnt = 0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) cnt += s_wh[w * RADIX + tid];
            __syncthreads();  // read before the first tile's counts
            // 2. publish the range's counts and look back over the earlier ranges
            const u32 first_range = r - (L.start - L.seg_begin) / range_items;
            u64* st = status + (u64)r * RADIX + tid;
            u32 excl = 0;
            if (L.first) {
                st_store(st, st_pack(epoch, ST_PREFIX, cnt));
            } else {
                st_store(st, st_pack(epoch, ST_AGG, cnt));
                excl = lookback_u32(status, RADIX, tid, r, first_range, epoch, ctl, 1u);
                st_store(st, st_pack(epoch, ST_PREFIX, excl + cnt));
            }
            s_run[tid] = __ldg(digit_off + ((u64)L.seg * npass + pass) * RADIX + tid) + excl;
        }
        // 3. the tiles of the range, in order
        const u32 seg_len = L.seg_end - L.seg_begin;
        for (u32 a = L.start; a < L.end; a += (u32)TILE) {
            const u32 n = min((u32)TILE, L.end - a);
            if (n == (u32)TILE) do_tile(std::true_type(), a, n, L.seg_begin, seg_len);
            else do_tile(std::false_type(), a, n, L.seg_begin, seg_len);
        }
    }
}

}  // namespace domagg
