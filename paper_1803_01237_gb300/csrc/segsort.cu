// segsort.cu -- stable segmented radix sort (local sort of Sec. 5/6 and, over
// bucket ranges, the local merge).
//
// Design for sm_103a:
//  * A segment of at most 4096 keys is sorted by one CTA on chip (k_chip): its
//    keys (and payload) are copied from HBM once into shared memory, counted
//    into groups that follow their distribution, ordered inside the groups as
//    32-bit words in registers, and written once (16 B of HBM traffic per key).
//    CTA shapes by segment size: 128 and 256 threads, and 1024 for segments of
//    up to 14336 keys where the tuning keeps them whole or the call has no more.
//  * A larger segment takes one read pass for statistics (digit counts and the
//    OR/AND of its keys) and one stable scatter on its first-split
//    digit (its top varying byte, or an interpolation of the key range the
//    caller bounds): the statistics pass counts every 4096-key tile's digits,
//    a scan turns the counts into each tile's destination offsets, and every
//    tile ranks its keys in shared memory (ballot peer masks with a payload,
//    one shared atomic per key for keys alone) and writes them out.  The 256 sub-buckets are then sorted the same way (on chip
//    when small, recursively otherwise), so a uniform 64-bit input costs
//    8 + 16 + 16 B of HBM traffic per key instead of the 136 B of eight LSD
//    passes.  A segment whose keys are all equal is copied straight to the
//    output by its scatter pass.
#include "segsort.cuh"

#include <algorithm>
#include <atomic>

namespace hss {

__host__ __device__ static inline uint64_t ceil_div(uint64_t a, uint64_t b) { return (a + b - 1) / b; }
static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Packing that nothing asked for (pack_keys 0): packs that fill the first
// on-chip class where a level has enough of them (merge of 2^28 pairs in 4096
// buckets 4.44 -> 4.23 ms against packs of 1024), smaller and more of them
// where SMs would stand idle (2^15 keys: 71 us, with full packs 83).
constexpr uint32_t kPackAuto = 0;
constexpr uint32_t kPackDefault = 1024;
constexpr uint64_t kPackMinKeys = 1ull << 22;
static uint32_t pack_limit(uint32_t pack_keys, uint64_t keys_large) {
    if (pack_keys != kPackAuto) return pack_keys;
    return keys_large >= kPackMinKeys ? (uint32_t)kC0Cap : kPackDefault;
}

// First splits of local sorts: on the top varying byte, on sampled splitters
// where the sample calls for them, or (nothing asked for) by the call's size
// (kSplMinKeys, kSplMinSeg).
constexpr uint32_t kFirstByte = 0, kFirstSampled = 1, kFirstAuto = 2;

// Process-wide tuning (hss_set_tuning).
static std::atomic<uint32_t> g_chip_max{(uint32_t)kC1Cap};
static std::atomic<uint32_t> g_child_interp{0u};
static std::atomic<uint32_t> g_child_keys{384u};
static std::atomic<uint32_t> g_pack_keys{kPackAuto};
static std::atomic<uint32_t> g_splitters{kFirstAuto};
static std::atomic<uint32_t> g_scatter{0u};

int set_tuning(const hss_tuning* t) {
    if (!t) {
        g_chip_max = (uint32_t)kC1Cap;
        g_child_interp = 0u;
        g_child_keys = 384u;
        g_pack_keys = kPackAuto;
        g_splitters = kFirstAuto;
        g_scatter = 0u;
        return HSS_OK;
    }
    const uint32_t cm = t->chip_max_keys ? t->chip_max_keys : (uint32_t)kC1Cap;
    const uint32_t ck = t->child_bucket_keys ? t->child_bucket_keys : 384u;
    if ((cm != (uint32_t)kC1Cap && cm != (uint32_t)kSmallCap) || t->child_interp > 1u || ck < 128u || ck > 4096u ||
        t->pack_keys > 4096u || t->first_split > kFirstSampled || t->split_scatter > 1u)
        return HSS_ERR_INVALID;
    for (uint32_t r : t->reserved)
        if (r) return HSS_ERR_INVALID;
    g_chip_max = cm;
    g_child_interp = t->child_interp;
    g_child_keys = ck;
    g_pack_keys = t->pack_keys;
    g_splitters = t->first_split;
    g_scatter = t->split_scatter;
    return HSS_OK;
}
void get_tuning(hss_tuning* t) {
    *t = hss_tuning{};
    t->chip_max_keys = g_chip_max;
    t->child_interp = g_child_interp;
    t->child_bucket_keys = g_child_keys;
    const uint32_t pk = g_pack_keys;
    t->pack_keys = pk == kPackAuto ? kPackDefault : pk;
    t->first_split = g_splitters == kFirstSampled ? kFirstSampled : kFirstByte;
    t->split_scatter = g_scatter;
}

// Large segments of a level hold more than kC1Cap keys (keys alone split above
// the middle on-chip class), so a level has at most N / (kC1Cap + 1) of them.
static uint64_t max_large_of(uint64_t N) { return std::max<uint64_t>(1, N / (kC1Cap + 1)); }

struct WsDims {
    uint64_t ml, list, tiles;
};
static WsDims ws_dims(uint64_t N, uint64_t nseg) {
    WsDims d;
    d.ml = max_large_of(N);
    d.list = std::max<uint64_t>(nseg, d.ml * kRadix);
    d.tiles = ceil_div(std::max<uint64_t>(N, 1), kOsTile) + d.ml + 1;
    return d;
}

size_t segsort_ws_bytes(uint64_t N, uint64_t nseg) {
    const WsDims d = ws_dims(N, nseg);
    size_t b = 0;
    b += align_up((d.list + 1) * 4, 256) + align_up(d.list * 4, 256);  // tile_start, large_id
    b += align_up(d.tiles * 4, 256);                                  // tile_seg
    b += align_up(d.ml * 4, 256);                                     // large_seg
    b += align_up(d.tiles * 2 * kRadix * 2, 256);                     // tile_hist
    b += align_up(d.tiles, 256);                                      // tile_skew
    b += align_up(std::min(nseg, d.ml) * kRadix * 4, 256);           // spl_tab
    b += align_up(std::min(nseg, d.ml), 256);                        // spl_mode
    b += 2 * align_up(d.ml * 8, 256);                                 // vor, vand
    b += 4 * align_up(d.ml * 4, 256);                                 // msd_shift x2, spec, direct
    b += 2 * align_up(d.ml * 8, 256);                                 // msd_base, msd_mult
    b += 4 * align_up(d.ml * kRadix * 8, 256);                        // sub_lo/hi x2
    b += 6 * align_up(d.ml * kRadix * 8, 256);                        // cmin/cmax/cmult x2
    b += align_up(d.ml * 8 * 4, 256) + align_up(d.ml * 4, 256);       // large_mask, any_large
    b += align_up(d.tiles * kRadix * 4, 256);                         // tile_off
    b += align_up(64 * 4, 256);                                       // counters
    b += 3 * align_up(d.list * 4, 256);                               // class lists
    b += align_up(8 * (d.list / 1024 + 2) * 4, 256);                  // blk
    return b;
}

SegSortWs segsort_ws_carve(void* base, uint64_t N, uint64_t nseg, uint32_t* err) {
    const WsDims d = ws_dims(N, nseg);
    SegSortWs w;
    w.max_large = d.ml;
    w.max_list = d.list;
    w.max_tiles = d.tiles;
    char* p = (char*)base;
    auto take = [&](size_t bytes) { void* r = p; p += align_up(bytes, 256); return r; };
    w.tile_start = (uint32_t*)take((d.list + 1) * 4);
    w.large_id = (uint32_t*)take(d.list * 4);
    w.tile_seg = (uint32_t*)take(d.tiles * 4);
    w.large_seg = (uint32_t*)take(d.ml * 4);
    w.tile_hist = (uint16_t*)take(d.tiles * 2 * kRadix * 2);
    w.tile_skew = (uint8_t*)take(d.tiles);
    w.max_spl = std::min(nseg, d.ml);
    w.spl_tab = (uint32_t*)take(w.max_spl * kRadix * 4);
    w.spl_mode = (uint8_t*)take(w.max_spl);
    w.vor = (unsigned long long*)take(d.ml * 8);
    w.vand = (unsigned long long*)take(d.ml * 8);
    w.msd_shift[0] = (uint32_t*)take(d.ml * 4);
    w.msd_shift[1] = (uint32_t*)take(d.ml * 4);
    w.spec = (uint32_t*)take(d.ml * 4);
    w.direct = (uint32_t*)take(d.ml * 4);
    w.msd_base = (uint64_t*)take(d.ml * 8);
    w.msd_mult = (uint64_t*)take(d.ml * 8);
    for (int i = 0; i < 2; ++i) {
        w.sub_lo[i] = (uint64_t*)take(d.ml * kRadix * 8);
        w.sub_hi[i] = (uint64_t*)take(d.ml * kRadix * 8);
        w.cmin[i] = (uint64_t*)take(d.ml * kRadix * 8);
        w.cmax[i] = (uint64_t*)take(d.ml * kRadix * 8);
        w.cmult[i] = (uint64_t*)take(d.ml * kRadix * 8);
    }
    w.large_mask = (uint32_t*)take(d.ml * 8 * 4);
    w.any_large = (uint32_t*)take(d.ml * 4);
    w.tile_off = (uint32_t*)take(d.tiles * kRadix * 4);
    w.counters = (uint32_t*)take(64 * 4);
    for (int i = 0; i < 3; ++i) w.list[i] = (uint32_t*)take(d.list * 4);
    w.blk = (uint32_t*)take(8 * (d.list / 1024 + 2) * 4);
    w.err = err;
    return w;
}

// Digit of the first split of a segment: an 8-bit window of the key, or (mult
// != 0) an interpolation of the segment's key range onto 0..255 (interp_digit).
__device__ __forceinline__ uint32_t split_digit(uint64_t key, int shift, uint64_t base, uint64_t mult) {
    if (mult) return interp_digit(key - base, mult);
    return (uint32_t)((key >> shift) - base) & 255u;
}

// ---------------------------------------------------------------------------
// Exclusive scan of 256 shared values by a CTA of T threads (T >= 64).
// ---------------------------------------------------------------------------
template <int T>
__device__ __forceinline__ void scan256_smem(const uint32_t* in, uint32_t* out, uint32_t* s_warp) {
    constexpr int U = T < kRadix ? T : kRadix;
    constexpr int K = kRadix / U;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t loc[K];
    uint32_t sum = 0;
    if (tid < U) {
#pragma unroll
        for (int k = 0; k < K; ++k) { loc[k] = in[tid * K + k]; sum += loc[k]; }
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31 && tid < U) s_warp[w] = x;
    __syncthreads();
    if (tid < U) {
        uint32_t run = x - sum;
        for (int i = 0; i < w; ++i) run += s_warp[i];
#pragma unroll
        for (int k = 0; k < K; ++k) { out[tid * K + k] = run; run += loc[k]; }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Peer mask of an 8-bit digit inside a warp, from eight ballots: the lanes
// whose digit equals this lane's.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t warp_peers8(uint32_t d) {
    uint32_t peers = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < kRadixBits; ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? m : ~m;
    }
    return peers;
}

// ---------------------------------------------------------------------------
// Stable block ranking of 8-bit digits (digit_of(i): the thread's item i), in
// three steps:
//   1. counts: every warp counts its digits into its own 256 shared counters
//      (16 bits, two to a word; fire-and-forget shared atomics);
//   2. offsets: the counts become absolute bases start[d] + (earlier warps'
//      counts of d); `between` runs before the barrier that ends the step;
//   3. ranks: per item, the lanes holding the same digit (ballot peer mask)
//      take consecutive slots from the warp's base for that digit, which the
//      lowest of them moves on; body(i, rank) takes each.
// Items are warp-striped: item i of lane l in warp w is element
// w*32*ITEMS + i*32 + l, so (w, i, l) order is element order and the ranks are
// stable.  Every item takes part; empty ones carry the last digit and, being
// last in element order, rank behind all others, so nothing tests for them
// (with such tests and an atomic for the base the split of pairs took 6% more).
// ---------------------------------------------------------------------------
template <int WARPS, int ITEMS, typename DigitOf, typename Between, typename Body>
__device__ __forceinline__ void block_rank(DigitOf digit_of, uint16_t* s_cnt /*[WARPS*256]*/, uint32_t* s_total,
                                           uint32_t* s_start, uint32_t* s_warp, Between between, Body body) {
    constexpr int T = WARPS * 32;
    static_assert(T >= kRadix && T * ITEMS < 65536, "a thread per digit, 16-bit counters");
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint16_t* c = s_cnt + w * kRadix;
    *(uint4*)(c + lane * 8) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t d = digit_of(i);
        atomicAdd((uint32_t*)c + (d >> 1), 1u << ((d & 1u) * 16u));
    }
    __syncthreads();
    if (tid < kRadix) {
        uint32_t run = 0;
#pragma unroll
        for (int ww = 0; ww < WARPS; ++ww) run += s_cnt[ww * kRadix + tid];
        s_total[tid] = run;
    }
    __syncthreads();
    scan256_smem<T>(s_total, s_start, s_warp);
    if (tid < kRadix) {
        uint32_t run = s_start[tid];
#pragma unroll
        for (int ww = 0; ww < WARPS; ++ww) {
            const uint32_t x = s_cnt[ww * kRadix + tid];
            s_cnt[ww * kRadix + tid] = (uint16_t)run;
            run += x;
        }
    }
    between();
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t d = digit_of(i);
        const uint32_t peers = warp_peers8(d);
        const uint32_t base = c[d], below = __popc(peers & lt);
        __syncwarp();
        if (below == 0) c[d] = (uint16_t)(base + (uint32_t)__popc(peers));
        __syncwarp();
        body(i, base + below);
    }
}

__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4(void* sdst, const void* gsrc) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
// One arrival that also announces `bytes` of bulk copies completing on bar.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// Bounded wait for the phase of the given parity to complete; false when the
// limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < (1u << 20); ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
// Orders ordinary accesses to shared memory, seen by the calling thread, before
// the bulk copies that it issues next.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_load(void* sdst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_u32(sdst)),
                 "l"(gsrc), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// CTAs per SM the register budget must allow: what their shared memory lets
// an SM hold (with a payload; seven against six: 2^28 pairs 2.37 -> 2.30 ms.
// Keys alone would spill for a ninth: 1.47 -> 1.58 ms).
template <bool PAY, int THREADS>
constexpr int chip_min_blocks() { return THREADS <= 128 ? (PAY ? 7 : 8) : (THREADS <= 256 ? 3 : 1); }

// ---------------------------------------------------------------------------
// On-chip sort of segments with min_n < n <= max_n keys (n <= CAP), with or
// without a payload, taken from `list` (compact ids, count at *nlist) or, when
// list is null, from all nseg segments: the stable sort by (key, position).
// FEW: segments of a few values are looked for (see below).
//
// One bulk copy brings the keys (and the payload) into shared memory, where
// they stay until they are written in order; what is sorted is one 32-bit
// word per key.
//  * x, the 32 key bits below the segment's common prefix (key - min,
//    normalised), is multiplied by R / range: the high word of the product is
//    the key's group, the low word its place inside the group.  One shared
//    counter per group (16 bits, two to a word) hands out slots.
//  * A segment whose keys crowd (a group above kChipRefine keys) counts again
//    with one group per key: group g's range is cut into as many parts as it
//    holds keys, so the groups follow the keys' distribution (a piecewise
//    linear estimate of it), up to kChipRefines times.
//  * The words (group start mod 64 | place in the group | position) are
//    scattered into group order, and ordered inside the groups by windows of
//    eight in registers, two instructions per comparator: each window is
//    sorted, then windows shifted by four merge the upper half of one with the
//    lower half of the next, back and forth (an odd-even transposition of
//    sorted blocks of four).  A group of g words spans at most
//    ceil((g-1)/4) + 1 blocks and is in order after that many rounds.
//  * Neighbours that agree in group and place (equal keys, or rarely distinct
//    ones closer than the place resolves) are in position order, which is the
//    stable order of equal keys; where their keys are found out of order the
//    run is sorted by (key, position).
// A group above kChipMaxGroup words that is left holds one key value (keys
// alone): its order is free.  The refining ends after kChipRefines counts at
// most.  A count from the groups' own ranges cuts every group above kChipRefine
// keys into 25 parts or more, none wider than 2/25 of its range, so 18 of them
// use up the keys' 64 bits and 4 the 14 bits of the positions (a payload's
// equal keys).  One count takes positions over the whole segment, and the
// others, the first and those that follow where the largest group shrank to a
// quarter and is still above kChipRefine, are five.
//
// Bound by shared-memory wavefronts and issue slots together (65% and 66% of
// their peaks; about 34 wavefronts and 144 instructions per key of a warp): the
// counting atomics, the group-start and key gathers and the word scatter each
// meet random banks.  Words of 32 bits instead of the keys themselves halve
// the scatter's wavefronts and make a comparator two instructions (six for 64
// bits: a variant that ordered the keys in registers spilled and took 3.9 ms).
// 2^28 uniform keys in buckets of about 1024: 2.28 ms with an insertion sort
// per thread over 64-bit keys (60 wavefronts, 204 instructions), 1.5 ms here;
// 2^28 Morton keys with a payload in segments of 2^14, whose groups crowd:
// 57.9 ms (most of it in digit passes that took the crowded segments), 6.6 ms.
// ---------------------------------------------------------------------------
// Exclusive scan in place of 2 NW 16-bit counters packed in NW shared words
// (counter 2i in the low half of word i) by a CTA of T threads, and the
// largest counter.  The counters add up to less than 2^16.  Ends with a
// barrier.
template <int T, int NW>
__device__ __forceinline__ uint32_t scan_pairs_inplace(uint32_t* v, uint32_t* s_warp /* 64 */) {
    constexpr int K = NW / T;
    constexpr int W = T / 32;
    static_assert(NW % T == 0 && K % 4 == 0 && W <= 32, "packed scan size");
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    uint32_t loc[K];
    uint32_t sum = 0, m2 = 0;
#pragma unroll
    for (int k = 0; k < K; k += 4) {
        const uint4 q = ((const uint4*)v)[(tid * K + k) / 4];
        loc[k] = q.x; loc[k + 1] = q.y; loc[k + 2] = q.z; loc[k + 3] = q.w;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        sum += (loc[k] & 0xffffu) + (loc[k] >> 16);
        m2 = __vmaxu2(m2, loc[k]);
    }
    uint32_t mx = __reduce_max_sync(0xffffffffu, max(m2 & 0xffffu, m2 >> 16));
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) { s_warp[w] = x; s_warp[32 + w] = mx; }
    __syncthreads();
    uint32_t run = x - sum;
#pragma unroll
    for (int i = 0; i < W; ++i) {
        if (i < w) run += s_warp[i];
        mx = max(mx, s_warp[32 + i]);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t lo = loc[k] & 0xffffu, hi = loc[k] >> 16;
        loc[k] = run | ((run + lo) << 16);
        run += lo + hi;
    }
#pragma unroll
    for (int k = 0; k < K; k += 4)
        ((uint4*)v)[(tid * K + k) / 4] = make_uint4(loc[k], loc[k + 1], loc[k + 2], loc[k + 3]);
    __syncthreads();
    return mx;
}

__device__ __forceinline__ void cmp_swap(uint32_t& x, uint32_t& y) {
    const uint32_t lo = min(x, y), hi = max(x, y);
    x = lo;
    y = hi;
}
// Batcher's odd-even merge of the sorted halves k[0..3] and k[4..7], and his
// sort of eight built on it (9 and 19 comparators).
__device__ __forceinline__ void merge_4_4(uint32_t (&k)[8]) {
    cmp_swap(k[0], k[4]); cmp_swap(k[1], k[5]); cmp_swap(k[2], k[6]); cmp_swap(k[3], k[7]);
    cmp_swap(k[2], k[4]); cmp_swap(k[3], k[5]);
    cmp_swap(k[1], k[2]); cmp_swap(k[3], k[4]); cmp_swap(k[5], k[6]);
}
__device__ __forceinline__ void sort_8(uint32_t (&k)[8]) {
    cmp_swap(k[0], k[1]); cmp_swap(k[2], k[3]); cmp_swap(k[4], k[5]); cmp_swap(k[6], k[7]);
    cmp_swap(k[0], k[2]); cmp_swap(k[1], k[3]); cmp_swap(k[4], k[6]); cmp_swap(k[5], k[7]);
    cmp_swap(k[1], k[2]); cmp_swap(k[5], k[6]);
    merge_4_4(k);
}

constexpr uint32_t kChipRefine = 24;    // a larger group: count again on the refined groups
constexpr uint32_t kFewShare = 16;      // a group above this part of the segment may be one of a few values
constexpr uint32_t kChipMaxGroup = 56;  // the largest group the window rounds order (start mod 64 is unambiguous)
// Counts from a group's own range until a range of `bits` bits is one value
// (32 bits of a key are looked at: the last factor is the part cut off), and
// the bound on all counts (see above).
constexpr int range_counts(int bits) {
    int c = 0;
    for (double r = (double)(1ull << (bits - 1)) * 2.0; r >= 1.0; r *= 2.0 / (kChipRefine + 1) * (1.0 + 0x1p-26)) ++c;
    return c;
}
constexpr int other_counts() {
    int c = 1;
    for (uint32_t most = kSmallCap / 4; most > kChipRefine; most /= 4) ++c;
    return c;
}
constexpr int kChipRefines = range_counts(64) + range_counts(14) + 1 + other_counts();
static_assert(range_counts(64) == 18 && range_counts(14) == 4 && other_counts() == 5, "as the comment above counts them");
constexpr uint32_t kChipRounds = (kChipMaxGroup + 2) / 4 + 3;  // rounds that order the largest group, and the one that finds it so
constexpr int kStartBits = 6;

// Position bits of a word (a segment of at most CAP keys).
template <int CAP>
constexpr int chip_pos_bits() { return CAP <= 2048 ? 11 : (CAP <= 4096 ? 12 : 14); }
// Counters: R groups of the first pass, one group per key of a refined one.
template <int THREADS, int CAP, int R>
constexpr int chip_counters() {
    constexpr int unit = 8 * THREADS;  // whole 16-byte vectors per thread
    return ((CAP > R ? CAP : R) + unit - 1) / unit * unit;
}
template <int THREADS, int CAP>
constexpr int chip_windows() { return (CAP / 8 + THREADS - 1) / THREADS; }
// The payload is staged on chip beside the keys, but for the largest class
// (its keys and words leave no room: gathered from its place in the input).
template <bool PAY, int CAP>
constexpr bool chip_stage_pay() { return PAY && CAP <= 4096; }

template <bool PAY, int THREADS, int CAP, int R>
constexpr size_t chip_smem() {
    return (size_t)(CAP + 2) * 8 + (size_t)(CAP + 16) * 4 + (chip_stage_pay<PAY, CAP>() ? (size_t)(CAP + 8) * 4 : 0) +
           (size_t)(chip_counters<THREADS, CAP, R>() / 2 + 4 + 32) * 4 + 64 * 4 +
           2 * (size_t)chip_windows<THREADS, CAP>() * (THREADS / 32) * 4 * 4 + 4 * 4 + 8 + 16;
}

template <bool PAY, int THREADS, int CAP, int R, bool FEW>
__global__ __launch_bounds__(THREADS, chip_min_blocks<PAY, THREADS>()) void k_chip(
    const uint64_t* kin, uint64_t* kout, const uint32_t* pin, uint32_t* pout, const uint64_t* __restrict__ seg_lo,
    const uint64_t* __restrict__ seg_hi, const uint32_t* __restrict__ list, const uint32_t* __restrict__ nlist,
    uint64_t nseg, uint32_t min_n, uint32_t max_n, uint64_t flip_in, uint64_t flip_out,
    uint32_t* __restrict__ err) {
    constexpr int ITEMS = CAP / THREADS;
    constexpr int WARPS = THREADS / 32;
    constexpr int WIN = chip_windows<THREADS, CAP>();
    constexpr int IDX = chip_pos_bits<CAP>();
    constexpr int FR = 32 - IDX - kStartBits;  // bits of the place inside the group
    constexpr int SH = FR + IDX;
    constexpr int NC = chip_counters<THREADS, CAP, R>();
    constexpr bool SPAY = chip_stage_pay<PAY, CAP>();
    constexpr uint32_t kPosMask = (1u << IDX) - 1u;
    constexpr int kVote = PAY ? 0 : IDX;  // keys alone: the order of equal keys is free
    constexpr uint32_t kSlotShift = 15, kGroupMask = (1u << kSlotShift) - 1u;
    static_assert(CAP % THREADS == 0 && CAP <= (1 << IDX) && NC + 66 < (1 << kSlotShift) && R % (8 * THREADS) == 0 &&
                      CAP < 16384 + 1,
                  "on-chip sort shape");
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t* s_key = (uint64_t*)smem;                                  // CAP + 2: the keys as read, key j at [j + sh]
    uint32_t* s_w = (uint32_t*)(s_key + (CAP + 2));                     // CAP + 16
    uint32_t* s_pay = s_w + (CAP + 16);                                 // CAP + 8 (SPAY)
    uint32_t* s_cnt = s_pay + (SPAY ? CAP + 8 : 0);                     // NC/2 words, the end, 32 words for empty items
    const uint16_t* s_start = (const uint16_t*)s_cnt;                   // after the scan: group starts, [groups] = n
    uint32_t* s_warp = s_cnt + (NC / 2 + 4 + 32);                       // 64
    uint32_t* s_edge = s_warp + 64;                                     // 2 x WIN * WARPS * 4
    uint32_t* s_first = s_edge + 2 * WIN * WARPS * 4;                   // 4
    uint64_t* s_bar = (uint64_t*)(((uintptr_t)(s_first + 4) + 7) & ~(uintptr_t)7);  // the keys have landed

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint64_t count = list ? (uint64_t)*nlist : nseg;
    const uint32_t hflip = (uint32_t)(flip_in >> 32);  // the sign bit, or nothing
    const uint64_t flip = flip_in ^ flip_out;          // from the input's key bits to the output's
    if (tid == 0) mbar_init(s_bar, 1u);
    __syncthreads();
    struct Desc {
        uint64_t base;
        uint32_t n;
        bool ok;  // exists and belongs to this class
    };
    auto load_desc = [&](uint64_t k) -> Desc {
        Desc d{0ull, 0u, false};
        if (k < count) {
            const uint64_t s = list ? (uint64_t)list[k] : k;
            const uint64_t b = seg_lo[s], n = seg_hi[s] - b;
            d.base = b;
            d.n = (uint32_t)n;
            d.ok = n > min_n && n <= max_n && n > 0;
        }
        return d;
    };
    // A bulk copy needs 16-byte aligned addresses: the elements in front of
    // the first boundary and behind the last one travel by small copies, and
    // everything sits in shared memory at the same offset mod 16 bytes.
    auto fetch = [&](const Desc& d) {
        const uint64_t* g = kin + d.base;
        const uint32_t hd = (uint32_t)(((uintptr_t)g >> 3) & 1u), m = ((d.n - hd) >> 1) << 1;
        uint32_t ph = 0, pm = 0, po = 0;
        const uint32_t* gp = nullptr;
        if (SPAY) {
            gp = pin + d.base;
            po = (uint32_t)(((uintptr_t)gp >> 2) & 3u);
            ph = min(d.n, (4u - po) & 3u);
            pm = ((d.n - ph) >> 2) << 2;
        }
        if (tid == 0) {
            fence_proxy_async();  // the last segment was read, and its ends written, where the next one goes
            mbar_arrive_expect_tx(s_bar, m * 8u + pm * 4u);
            if (m) bulk_load(s_key + 2 * hd, g + hd, m * 8u, s_bar);
            if (SPAY && pm) bulk_load(s_pay + po + ph, gp + ph, pm * 4u, s_bar);
        }
        if (hd && tid == 32) cp_async8(&s_key[1], g);
        if (hd + m < d.n && tid == 33) cp_async8(&s_key[d.n - 1 + hd], g + d.n - 1);
        if (SPAY) {
            if (tid >= 40 && (uint32_t)(tid - 40) < ph) cp_async4(&s_pay[po + tid - 40], gp + tid - 40);
            if (tid >= 44 && tid < 48 && ph + pm + (uint32_t)(tid - 44) < d.n)
                cp_async4(&s_pay[po + ph + pm + tid - 44], gp + ph + pm + tid - 44);
        }
        cp_async_commit();
    };
    // Slot of a key among the keys of group d counted so far.
    auto take_slot = [&](uint32_t d) -> uint32_t {
        const uint32_t sft = (d & 1u) * 16u;
        return (atomicAdd(&s_cnt[d >> 1], 1u << sft) >> sft) & 0xffffu;
    };
    uint32_t phase = 0;
    Desc cur = load_desc(blockIdx.x);
    if (cur.ok) fetch(cur);
    for (uint64_t k = blockIdx.x; k < count; k += gridDim.x) {
        const Desc nxt = load_desc(k + gridDim.x);
        if (!cur.ok) {  // uniform per CTA; such a segment was never fetched
            cur = nxt;
            if (cur.ok) fetch(cur);
            continue;
        }
        const uint64_t base = cur.base;
        const uint32_t n = cur.n;
        const uint32_t sh = (uint32_t)(((uintptr_t)(kin + base) >> 3) & 1u);
        const uint64_t* key = s_key + sh;
        cp_async_wait_all();
        const bool late = !mbar_wait(s_bar, phase);
        phase ^= 1u;
        if (__syncthreads_or(late)) {  // uniform; not expected: a bulk copy that never landed
            if (tid == 0) {
                atomicOr(err, kDevErrTimeout);
                mbar_wait(s_bar, phase ^ 1u);  // the CTA's memory stays until the copy is done, or once more the limit
            }
            break;
        }
        // Range of the high words (of the low words when those are all equal).
        uint32_t vmin = ~0u, vmax = 0u;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if ((uint32_t)(i * THREADS) >= n) break;
            const uint32_t e = min((uint32_t)(tid + i * THREADS), n - 1);
            const uint32_t h = (uint32_t)(key[e] >> 32) ^ hflip;
            vmin = min(vmin, h);
            vmax = max(vmax, h);
        }
        vmin = __reduce_min_sync(0xffffffffu, vmin);
        vmax = __reduce_max_sync(0xffffffffu, vmax);
        if (lane == 0) { s_warp[w] = vmin; s_warp[32 + w] = vmax; }
        for (int d = tid; d < R / 8; d += THREADS) ((uint4*)s_cnt)[d] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < WARPS; ++i) { vmin = min(vmin, s_warp[i]); vmax = max(vmax, s_warp[32 + i]); }
        const bool by_hi = vmin != vmax;  // uniform
        if (!by_hi) {
            __syncthreads();  // s_warp is written again
            vmin = ~0u; vmax = 0u;
            for (uint32_t e = tid; e < n; e += THREADS) {
                const uint32_t l = (uint32_t)key[e];
                vmin = min(vmin, l);
                vmax = max(vmax, l);
            }
            vmin = __reduce_min_sync(0xffffffffu, vmin);
            vmax = __reduce_max_sync(0xffffffffu, vmax);
            if (lane == 0) { s_warp[w] = vmin; s_warp[32 + w] = vmax; }
            __syncthreads();
            for (int i = 0; i < WARPS; ++i) { vmin = min(vmin, s_warp[i]); vmax = max(vmax, s_warp[32 + i]); }
        }
        uint64_t* dst = kout + base;
        const uint32_t po = SPAY ? (uint32_t)(((uintptr_t)(pin + base) >> 2) & 3u) : 0u;
        bool done = false;
        if (vmin == vmax) {  // all keys equal: already in order
            for (uint32_t j = tid; j < n; j += THREADS) {
                dst[j] = key[j] ^ flip;
                if (PAY) pout[base + j] = SPAY ? s_pay[po + j] : pin[base + j];
            }
            done = true;
        }
        if (!done) {
            // x: the 32 bits below the common prefix of key - min; the largest
            // one, top, has its high bit set, and the multiplier stays a
            // little below R 2^32 / top so that no group number reaches R.
            const int norm = __clz((int)(vmax - vmin));
            const uint32_t top = (vmax - vmin) << norm | (norm ? (by_hi ? ~0u >> (32 - norm) : 0u) : 0u);
            const uint32_t mult = __float2uint_rz(__fdividef((float)R * 4294967296.0f, (float)top) * (1.0f - 0x1p-20f));
            uint32_t fr[ITEMS], dp[ITEMS];  // place in the group; group and slot
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                if ((uint32_t)(i * THREADS) >= n) break;
                const uint32_t e = tid + i * THREADS;
                const uint64_t kk = key[min(e, n - 1)];
                const uint32_t lo = (uint32_t)kk, hi = (uint32_t)(kk >> 32) ^ hflip;
                const uint32_t x = by_hi ? __funnelshift_l(lo, hi - vmin, norm) : (lo - vmin) << norm;
                const uint64_t prod = (uint64_t)x * mult;
                const uint32_t d = e < n ? (uint32_t)(prod >> 32) : (uint32_t)(NC + 8 + 2 * lane);
                fr[i] = (uint32_t)prod;
                dp[i] = d | take_slot(d) << kSlotShift;
            }
            if (tid == 0) s_cnt[R / 2] = n;  // the end of the last group
            __syncthreads();
            uint32_t mx = scan_pairs_inplace<THREADS, R / 2>(s_cnt, s_warp);
            // Crowded groups: every group cut into as many parts as it holds
            // keys, and counted again.  Where that did not bring the largest
            // group to a quarter, the place of a key in a group above
            // kChipRefine keys is first taken again from the group's own key
            // range (or, with a payload, its range of positions where it holds
            // one key value), so that clusters inside clusters resolve
            // whatever their widths.
            bool tried_pos = false;
            uint32_t before = 0;
            for (int it = 0; mx > kChipRefine; ++it) {  // uniform
                auto each_key = [&](auto body) {
#pragma unroll
                    for (int i = 0; i < ITEMS; ++i) {
                        if ((uint32_t)(i * THREADS) >= n) break;
                        if (tid + i * THREADS < n) body(i, (uint32_t)(tid + i * THREADS));
                    }
                };
                if (it == kChipRefines) {
                    if (tid == 0) atomicOr(err, kDevErrBounds);
                    break;
                }
                // body(item, position, the group's part of s_w)
                auto each_crowded = [&](auto body) {
                    each_key([&](int i, uint32_t e) {
                        const uint32_t d = dp[i] & kGroupMask, a = s_start[d];
                        if (s_start[d + 1] - a > kChipRefine) body(i, e, s_w + a);
                    });
                };
                bool look = it > 0 && 4u * mx > before;
                if (FEW && it == 0 && kFewShare * mx > n) {
                    // A few values make groups of one value each, which another
                    // count leaves as they are, every key at the same counter.
                    // Where no two neighbouring items of a thread share a group
                    // and not their place, look first (4096 segments of 4096
                    // keys, 2 or 16 values: 236 -> 201, 218 -> 192 us).
                    bool spread = false;
#pragma unroll
                    for (int i = 0; i + 1 < ITEMS; ++i)
                        if ((uint32_t)(tid + (i + 1) * THREADS) < n)
                            spread = spread || (((dp[i] ^ dp[i + 1]) & kGroupMask) == 0u && fr[i] != fr[i + 1]);
                    look = __syncthreads_or(spread) == 0;
                }
                if (look) {
                    // Crowded groups of one key value each are in order (keys
                    // alone), or the window rounds put them in order.
                    each_crowded([&](int i, uint32_t e, uint32_t* r) {
                        if (dp[i] >> kSlotShift == 0u) r[0] = e;
                    });
                    __syncthreads();
                    bool open = false;
                    each_crowded([&](int, uint32_t e, uint32_t* r) { open = open || key[r[0]] != key[e]; });
                    open = __syncthreads_or(open) != 0;
                    if (!open && (!PAY || mx <= kChipMaxGroup)) break;
                    if (!open && !tried_pos) {
                        // one value per group: by position over the whole segment
                        const uint32_t unit = 0xffffffffu / n;
                        tried_pos = true;
                        each_crowded([&](int i, uint32_t e, uint32_t*) { fr[i] = e * unit; });
                    } else if (!FEW || it > 0) {
                        // the group's key range (high words, then the low
                        // words at its ends) and positions
                        each_crowded([&](int i, uint32_t, uint32_t* r) {
                            if (dp[i] >> kSlotShift == 0u) {
                                r[0] = r[2] = r[4] = ~0u;
                                r[1] = r[3] = r[5] = 0u;
                            }
                        });
                        __syncthreads();
                        each_crowded([&](int, uint32_t e, uint32_t* r) {
                            const uint32_t h = (uint32_t)(key[e] >> 32) ^ hflip;
                            atomicMin(r, h);
                            atomicMax(r + 1, h);
                        });
                        __syncthreads();
                        each_crowded([&](int, uint32_t e, uint32_t* r) {
                            const uint64_t kk = key[e];
                            const uint32_t h = (uint32_t)(kk >> 32) ^ hflip, l = (uint32_t)kk;
                            if (h == r[0]) atomicMin(r + 2, l);
                            if (h == r[1]) atomicMax(r + 3, l);
                            if (PAY && r[0] == r[1]) { atomicMin(r + 4, e); atomicMax(r + 5, e); }
                        });
                        __syncthreads();
                        each_crowded([&](int i, uint32_t e, uint32_t* r) {
                            const uint64_t lo = (uint64_t)r[0] << 32 | r[2], range = ((uint64_t)r[1] << 32 | r[3]) - lo;
                            const uint64_t kk = key[e] ^ ((uint64_t)hflip << 32);
                            if (range != 0ull)
                                fr[i] = (uint32_t)(((kk - lo) << __clzll((long long)range)) >> 32);
                            else if (PAY)
                                fr[i] = (e - r[4]) << __clz((int)(r[5] - r[4]));
                        });
                    }
                }
                before = mx;
                each_key([&](int i, uint32_t) {
                    const uint32_t d = dp[i] & kGroupMask, a = s_start[d];
                    const uint64_t prod = (uint64_t)fr[i] * (s_start[d + 1] - a);
                    dp[i] = a + (uint32_t)(prod >> 32);
                    fr[i] = (uint32_t)prod;
                });
                __syncthreads();
                for (int d = tid; d < NC / 8; d += THREADS) ((uint4*)s_cnt)[d] = make_uint4(0u, 0u, 0u, 0u);
                __syncthreads();
                each_key([&](int i, uint32_t) { dp[i] |= take_slot(dp[i]) << kSlotShift; });
                if (tid == 0) s_cnt[NC / 2] = n;
                __syncthreads();
                mx = scan_pairs_inplace<THREADS, NC / 2>(s_cnt, s_warp);
            }
            {
                const uint32_t W = (n + 7) / 8;  // windows of eight words
#pragma unroll
                for (int i = 0; i < ITEMS; ++i) {
                    if ((uint32_t)(i * THREADS) >= n) break;
                    const uint32_t e = tid + i * THREADS;
                    const uint32_t a = s_start[dp[i] & kGroupMask];
                    const uint32_t word = a << SH | (fr[i] >> (32 - FR)) << IDX | e;
                    if (e < n) s_w[a + (dp[i] >> kSlotShift)] = word;
                }
                if (tid < 8 && n + tid < 8 * W) s_w[n + tid] = (n + tid) << SH | ((1u << SH) - 1u);
                if (!PAY && mx > kChipMaxGroup) {
                    // keys alone: the words of a large group (one key value)
                    // stay where they are, their own index as group start
#pragma unroll
                    for (int i = 0; i < ITEMS; ++i) {
                        if ((uint32_t)(i * THREADS) >= n) break;
                        const uint32_t e = tid + i * THREADS, d = dp[i] & kGroupMask;
                        const uint32_t a = s_start[d], at = a + (dp[i] >> kSlotShift);
                        if (e < n && s_start[d + 1] - a > kChipMaxGroup) s_w[at] = at << SH | e;
                    }
                }
                __syncthreads();
                {
                    // Words relative to their window: start - window + 56 in the top bits.
                    uint32_t q[WIN][8];
#pragma unroll
                    for (int v = 0; v < WIN; ++v) {
                        const uint32_t b = tid + v * THREADS;
                        if (b < W) {
                            const uint4* src4 = (const uint4*)(s_w + 8 * b);
                            const uint4 x = src4[(tid >> 2) & 1], y = src4[((tid >> 2) & 1) ^ 1];  // no bank met twice
                            const uint32_t rel = (8 * b + 8) << SH;  // 8 b - 56 mod 64
                            q[v][0] = x.x - rel; q[v][1] = x.y - rel; q[v][2] = x.z - rel; q[v][3] = x.w - rel;
                            q[v][4] = y.x - rel; q[v][5] = y.y - rel; q[v][6] = y.z - rel; q[v][7] = y.w - rel;
                            sort_8(q[v]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 8; ++i) q[v][i] = ~0u;
                        }
                    }
                    if (tid == 0) *(uint4*)s_first = make_uint4(q[0][0], q[0][1], q[0][2], q[0][3]);
                    constexpr uint32_t kStep = 4u << SH;
                    // Round 2 and every even one: window b takes the lower half
                    // of window b + 1; odd rounds: back.  s_first: the lower
                    // half of window 0 meanwhile.
                    auto round_up = [&](uint32_t* edge, bool moved_before) -> int {
#pragma unroll
                        for (int v = 0; v < WIN; ++v)
                            if (lane == 0)
                                *(uint4*)(edge + (v * WARPS + w) * 4) = make_uint4(q[v][0], q[v][1], q[v][2], q[v][3]);
                        return __syncthreads_or(moved_before);
                    };
                    auto merge_up = [&](const uint32_t* edge) -> bool {
                        bool moved = false;
#pragma unroll
                        for (int v = 0; v < WIN; ++v) {
                            if ((uint32_t)(v * THREADS + w * 32) >= W) break;  // uniform per warp
                            uint32_t o[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) o[i] = __shfl_down_sync(0xffffffffu, q[v][i], 1);
                            const uint32_t b = tid + v * THREADS;
                            if (lane == 31) {
                                const uint4 x = b + 1 < W ? *(const uint4*)(edge + (v * WARPS + w + 1) * 4)
                                                          : make_uint4(~0u, ~0u, ~0u, ~0u);
                                o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w;
                            }
                            const bool last = b + 1 >= W;
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                q[v][i] = q[v][4 + i] - kStep;
                                q[v][4 + i] = last ? ~0u : o[i] + kStep;
                            }
                            moved = moved || (b < W && q[v][4] >> kVote < q[v][3] >> kVote);
                            merge_4_4(q[v]);
                        }
                        return moved;
                    };
                    round_up(s_edge, false);
                    merge_up(s_edge);
                    uint32_t off = 4;
                    if (mx > 5u) {  // uniform
                        bool moved = false;
                        for (uint32_t round = 3; round <= kChipRounds; ++round) {
                            uint32_t* edge = s_edge + (round & 1u) * (WIN * WARPS * 4);
                            if (off) {
#pragma unroll
                                for (int v = 0; v < WIN; ++v)
                                    if (lane == 31)
                                        *(uint4*)(edge + (v * WARPS + w) * 4) =
                                            make_uint4(q[v][4], q[v][5], q[v][6], q[v][7]);
                                if (!__syncthreads_or(moved) && round > 3) break;  // the last round changed nothing
                                moved = false;
#pragma unroll
                                for (int v = 0; v < WIN; ++v) {
                                    if ((uint32_t)(v * THREADS + w * 32) >= W) break;
                                    uint32_t o[4];
#pragma unroll
                                    for (int i = 0; i < 4; ++i) o[i] = __shfl_up_sync(0xffffffffu, q[v][4 + i], 1);
                                    const uint32_t b = tid + v * THREADS;
                                    if (lane == 0) {
                                        const uint4 x = b > 0 ? *(const uint4*)(edge + (v * WARPS + w - 1) * 4)
                                                              : *(const uint4*)s_first;
                                        o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w;
                                    }
#pragma unroll
                                    for (int i = 0; i < 4; ++i) {
                                        q[v][4 + i] = q[v][i] + kStep;
                                        q[v][i] = b > 0 ? o[i] - kStep : o[i];
                                    }
                                    moved = moved || (b < W && q[v][4] >> kVote < q[v][3] >> kVote);
                                    merge_4_4(q[v]);
                                }
                                if (tid == 0) *(uint4*)s_first = make_uint4(q[0][0], q[0][1], q[0][2], q[0][3]);
                            } else {
                                if (!round_up(edge, moved)) break;
                                moved = merge_up(edge);
                            }
                            off ^= 4u;
                            if (mx <= 9u) break;  // three rounds order groups of nine
                        }
                    }
                    // The words in order, as they were scattered.
                    if (off && tid == 0) {
                        const uint4 x = *(const uint4*)s_first;
                        constexpr uint32_t rel = 8u << SH;
                        *(uint4*)s_w = make_uint4(x.x + rel, x.y + rel, x.z + rel, x.w + rel);
                    }
#pragma unroll
                    for (int v = 0; v < WIN; ++v) {
                        const uint32_t b = tid + v * THREADS;
                        if (b < W) {
                            const uint32_t rel = (8 * b + off + 8) << SH;
                            uint4* o = (uint4*)(s_w + 8 * b + off);
                            o[0] = make_uint4(q[v][0] + rel, q[v][1] + rel, q[v][2] + rel, q[v][3] + rel);
                            o[1] = make_uint4(q[v][4] + rel, q[v][5] + rel, q[v][6] + rel, q[v][7] + rel);
                        }
                    }
                    __syncthreads();
                    bool wrong = false;
                    auto put = [&](uint32_t j, uint32_t wj) {
                        const uint32_t e = wj & kPosMask;
                        dst[j] = key[e] ^ flip;
                        if (SPAY) pout[base + j] = s_pay[po + e];
                    };
#pragma unroll 4
                    for (uint32_t j = tid; j < n; j += THREADS) {
                        const uint32_t wj = s_w[j], w1 = s_w[j + 1];
                        if (((wj ^ w1) >> IDX) == 0u && j + 1 < n) {
                            const uint64_t f = (uint64_t)hflip << 32;
                            wrong = wrong || (key[wj & kPosMask] ^ f) > (key[w1 & kPosMask] ^ f);
                        }
                        put(j, wj);
                    }
                    if (__syncthreads_or(wrong)) {
                        // Distinct keys that the words do not tell apart: each
                        // run of equal (group, place) by (key, position).
                        const uint64_t f = (uint64_t)hflip << 32;
                        for (uint32_t j = tid; j + 1 < n; j += THREADS) {
                            if (j > 0 && ((s_w[j - 1] ^ s_w[j]) >> IDX) == 0u) continue;  // not the start of a run
                            const uint32_t head = s_w[j] >> IDX;
                            uint32_t z = j + 1;
                            for (; z < n && s_w[z] >> IDX == head; ++z) {
                                const uint32_t wz = s_w[z], ez = wz & kPosMask;
                                const uint64_t kz = key[ez] ^ f;
                                uint32_t i = z;
                                for (; i > j; --i) {
                                    const uint32_t wy = s_w[i - 1], ey = wy & kPosMask;
                                    const uint64_t ky = key[ey] ^ f;
                                    if (ky < kz || (ky == kz && ey < ez)) break;
                                    s_w[i] = wy;
                                }
                                s_w[i] = wz;
                            }
                        }
                        __syncthreads();
                        for (uint32_t j = tid; j < n; j += THREADS) put(j, s_w[j]);
                    }
                    if (PAY && !SPAY) {  // the output may be the input: gather every payload first
                        uint32_t pv[ITEMS];
#pragma unroll
                        for (int i = 0; i < ITEMS; ++i) {
                            const uint32_t j = tid + i * THREADS;
                            pv[i] = j < n ? pin[base + (s_w[j] & kPosMask)] : 0u;
                        }
                        __syncthreads();
#pragma unroll
                        for (int i = 0; i < ITEMS; ++i) {
                            const uint32_t j = tid + i * THREADS;
                            if (j < n) pout[base + j] = pv[i];
                        }
                    }
                }
            }
        }
        __syncthreads();  // the staged keys have been read
        cur = nxt;
        if (cur.ok) fetch(cur);
    }
    cp_async_wait_all();
}

// ---------------------------------------------------------------------------
// Planning of one level, as a three-step scan over chunks of 1024 segments:
// compact lists of the segments of each on-chip size class, compact ids and
// tiles of the segments above the on-chip capacity.
// counters[16..18] = class sizes, [19] = #large, [20] = #tiles,
// [22..23] = keys in large segments.
// ---------------------------------------------------------------------------
struct PlanV {
    uint32_t c[5];  // classes 0..2, large, tiles
    unsigned long long keys;
};

// chip_max: the largest segment sorted on chip at this level (kSmallCap, or
// kC1Cap to split larger ones again instead of the largest on-chip class).
__device__ __forceinline__ PlanV plan_item(const uint64_t* seg_lo, const uint64_t* seg_hi, uint64_t nseg, uint64_t s,
                                           uint32_t chip_max) {
    PlanV v = {{0, 0, 0, 0, 0}, 0ull};
    if (s < nseg) {
        const uint64_t n = seg_hi[s] - seg_lo[s];
        if (n == 0) {
        } else if (n <= (uint64_t)kC0Cap) {
            v.c[0] = 1;
        } else if (n <= (uint64_t)kC1Cap) {
            v.c[1] = 1;
        } else if (n <= (uint64_t)chip_max) {
            v.c[2] = 1;
        } else if (n >= kMaxSegKeys) {
            // above the limit on a segment: left unsorted, reported where the entries are written
        } else {
            v.c[3] = 1;
            v.c[4] = (uint32_t)ceil_div(n, kOsTile);
            v.keys = n;
        }
    }
    return v;
}

// From inclusive sums inside each warp (keys: the warp's sum, in lane 31) to
// sums over the CTA's warps so far, and the CTA's totals in tot.  The keys are
// only totalled.  Each warp adds up the others' sums with reductions (a loop
// over the warps by every thread, and shuffles for the flags, took most of the
// time: 4.2 million segments counted in 112 us, now 28, and written in 83, now
// 32; one CTA of 1024 segments 7, now 4).
__device__ __forceinline__ void plan_cross(PlanV& v, PlanV& tot) {
    __shared__ uint32_t s_c[5][32];
    __shared__ unsigned long long s_k[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 31) {
#pragma unroll
        for (int i = 0; i < 5; ++i) s_c[i][w] = v.c[i];
        s_k[w] = v.keys;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const uint32_t x = lane < nw ? s_c[i][lane] : 0u;
        v.c[i] += __reduce_add_sync(0xffffffffu, lane < w ? x : 0u);
        tot.c[i] = __reduce_add_sync(0xffffffffu, x);
    }
    unsigned long long k = lane < nw ? s_k[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    tot.keys = k;
    __syncthreads();
}
// Inclusive scan of the CTA's items: flags by ballots, tiles and keys only in
// warps that hold a large segment.
__device__ __forceinline__ void plan_scan_items(PlanV& v, PlanV& tot) {
    const uint32_t lane = threadIdx.x & 31, upto = 0xffffffffu >> (31 - lane);
    uint32_t large = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        large = __ballot_sync(0xffffffffu, v.c[i] != 0u);
        v.c[i] = __popc(large & upto);
    }
    if (large) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v.c[4], o);
            const unsigned long long yk = __shfl_up_sync(0xffffffffu, v.keys, o);
            if (lane >= (uint32_t)o) { v.c[4] += y; v.keys += yk; }
        }
    }
    plan_cross(v, tot);
}
// The same for the chunks' totals.
__device__ __forceinline__ void plan_scan(PlanV& v, PlanV& tot) {
    const uint32_t lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v.c[i], o);
            if (lane >= (uint32_t)o) v.c[i] += y;
        }
        const unsigned long long yk = __shfl_up_sync(0xffffffffu, v.keys, o);
        if (lane >= (uint32_t)o) v.keys += yk;
    }
    plan_cross(v, tot);
}

__device__ __forceinline__ void blk_store(uint32_t* blk, uint32_t i, const PlanV& v) {
    uint32_t* b = blk + 8 * (uint64_t)i;
#pragma unroll
    for (int k = 0; k < 5; ++k) b[k] = v.c[k];
    *(unsigned long long*)(b + 6) = v.keys;
}
__device__ __forceinline__ PlanV blk_load(const uint32_t* blk, uint32_t i) {
    const uint32_t* b = blk + 8 * (uint64_t)i;
    PlanV v;
#pragma unroll
    for (int k = 0; k < 5; ++k) v.c[k] = b[k];
    v.keys = *(const unsigned long long*)(b + 6);
    return v;
}

__global__ __launch_bounds__(1024) void k_plan_count(const uint64_t* __restrict__ seg_lo, const uint64_t* __restrict__ seg_hi,
                                                     uint64_t nseg, uint32_t* __restrict__ blk, uint32_t chip_max) {
    PlanV v = plan_item(seg_lo, seg_hi, nseg, (uint64_t)blockIdx.x * 1024 + threadIdx.x, chip_max), tot;
    plan_scan_items(v, tot);
    if (threadIdx.x == 0) blk_store(blk, blockIdx.x, tot);
}

// The level's totals into counters (and for the host).
__device__ __forceinline__ void plan_totals(const PlanV& carry, uint32_t* counters, volatile uint32_t* host_counts) {
    for (int k = 0; k < 5; ++k) counters[16 + k] = carry.c[k];
    *(unsigned long long*)(counters + 22) = carry.keys;
    if (host_counts) {  // the same eight words for the host, in mapped pinned memory
        for (int k = 0; k < 5; ++k) host_counts[k] = carry.c[k];
        host_counts[5] = 0;
        host_counts[6] = (uint32_t)carry.keys;
        host_counts[7] = (uint32_t)(carry.keys >> 32);
    }
}

// Exclusive scan of the chunk totals (one CTA), totals into counters.
__global__ __launch_bounds__(1024) void k_plan_scan(uint32_t nblk, uint32_t* __restrict__ blk, uint32_t* __restrict__ counters,
                                                    volatile uint32_t* host_counts) {
    PlanV carry = {{0, 0, 0, 0, 0}, 0ull};
    for (uint32_t base = 0; base < nblk; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        PlanV v = i < nblk ? blk_load(blk, i) : PlanV{{0, 0, 0, 0, 0}, 0ull};
        const PlanV v0 = v;
        PlanV tot;
        plan_scan(v, tot);
        if (i < nblk) {
            PlanV ex;
#pragma unroll
            for (int k = 0; k < 5; ++k) ex.c[k] = carry.c[k] + v.c[k] - v0.c[k];
            ex.keys = 0ull;  // not used
            blk_store(blk, i, ex);
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) carry.c[k] += tot.c[k];
        carry.keys += tot.keys;
    }
    if (threadIdx.x == 0) plan_totals(carry, counters, host_counts);
}

// The entries of segment s, given the totals of the segments before its chunk
// (off) and its inclusive scan inside the chunk (v).
struct PlanOut {
    uint32_t* tile_start;
    uint32_t* large_id;
    uint32_t* large_seg;
    uint32_t* list0;
    uint32_t* list1;
    uint32_t* list2;
    uint32_t* err;
    uint32_t* tile_seg;
};
__device__ __forceinline__ void plan_entries(uint64_t s, const PlanV& item, const PlanV& v, const PlanV& off,
                                             const PlanOut& P) {
    P.tile_start[s] = off.c[4] + v.c[4] - item.c[4];
    P.large_id[s] = 0xffffffffu;
    if (item.c[0]) P.list0[off.c[0] + v.c[0] - 1] = (uint32_t)s;
    if (item.c[1]) P.list1[off.c[1] + v.c[1] - 1] = (uint32_t)s;
    if (item.c[2]) P.list2[off.c[2] + v.c[2] - 1] = (uint32_t)s;
    if (item.c[3]) {
        const uint32_t id = off.c[3] + v.c[3] - 1;
        P.large_id[s] = id;
        P.large_seg[id] = (uint32_t)s;
    }
}
// The tiles of the warp's segments (t0: the first tile of the lane's, c: their
// number).  Long rows by the whole warp, one after the other: a lane writing
// its own row alone took 39 us for 1024 segments of 64 tiles.
__device__ __forceinline__ void plan_tiles(uint32_t s, uint32_t t0, uint32_t c, uint32_t* __restrict__ tile_seg) {
    if (__reduce_max_sync(0xffffffffu, c) <= 4u) {
        for (uint32_t u = 0; u < c; ++u) tile_seg[t0 + u] = s;
        return;
    }
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t left = __ballot_sync(0xffffffffu, c > 0u); left; left &= left - 1) {
        const int from = __ffs(left) - 1;
        const uint32_t cs = __shfl_sync(0xffffffffu, s, from), ct = __shfl_sync(0xffffffffu, t0, from),
                       cc = __shfl_sync(0xffffffffu, c, from);
        for (uint32_t u = lane; u < cc; u += 32) tile_seg[ct + u] = cs;
    }
}

__global__ __launch_bounds__(1024) void k_plan_write(const uint64_t* __restrict__ seg_lo, const uint64_t* __restrict__ seg_hi,
                                                     uint64_t nseg, const uint32_t* __restrict__ blk,
                                                     const uint32_t* __restrict__ counters, const PlanOut P,
                                                     uint32_t chip_max) {
    const uint64_t s = (uint64_t)blockIdx.x * 1024 + threadIdx.x;
    const PlanV item = plan_item(seg_lo, seg_hi, nseg, s, chip_max);
    if (s < nseg && seg_hi[s] - seg_lo[s] >= kMaxSegKeys) atomicOr(P.err, kDevErrSize);
    PlanV v = item, tot;
    plan_scan_items(v, tot);
    const PlanV off = blk_load(blk, blockIdx.x);
    if (s < nseg) plan_entries(s, item, v, off, P);
    plan_tiles((uint32_t)s, off.c[4] + v.c[4] - item.c[4], item.c[4], P.tile_seg);
    if (s == nseg) P.tile_start[nseg] = counters[20];
}

// The three steps in one launch by one CTA that carries the totals from chunk
// to chunk: for a few chunks (kPlanOneChunks) that is faster than two more
// launches (6 us each; about 2 us a chunk).
constexpr uint32_t kPlanOneChunks = 4;
__global__ __launch_bounds__(1024) void k_plan_one(const uint64_t* __restrict__ seg_lo, const uint64_t* __restrict__ seg_hi,
                                                   uint64_t nseg, uint32_t* __restrict__ counters,
                                                   volatile uint32_t* host_counts, const PlanOut P, uint32_t chip_max) {
    PlanV carry = {{0, 0, 0, 0, 0}, 0ull};
    for (uint64_t s0 = 0; s0 < nseg; s0 += 1024) {
        const uint64_t s = s0 + threadIdx.x;
        const PlanV item = plan_item(seg_lo, seg_hi, nseg, s, chip_max);
        if (s < nseg && seg_hi[s] - seg_lo[s] >= kMaxSegKeys) atomicOr(P.err, kDevErrSize);
        PlanV v = item, tot;
        plan_scan_items(v, tot);
        if (s < nseg) plan_entries(s, item, v, carry, P);
        plan_tiles((uint32_t)s, carry.c[4] + v.c[4] - item.c[4], item.c[4], P.tile_seg);
#pragma unroll
        for (int k = 0; k < 5; ++k) carry.c[k] += tot.c[k];
        carry.keys += tot.keys;
    }
    if (threadIdx.x == 0) {
        P.tile_start[nseg] = carry.c[4];
        plan_totals(carry, counters, host_counts);
    }
}

// ---------------------------------------------------------------------------
// Statistics of the large segments, per tile of kOsTile keys: the digit
// histogram of the tile (on a speculative window, or on the interpolating
// hint) and the OR/AND of the segment's keys, in one read.  One CTA per tile.
// From these the split pass gets every tile's destination offsets by a scan
// (k_msd_prep) instead of a look-back across the tiles of its segment.
// ---------------------------------------------------------------------------
// msd_shift flag: the split interpolated the key range (no byte is fixed in
// its sub-buckets).
constexpr uint32_t kShiftInterp = 0x100u;
// msd_shift flag: the split's digit is the bucket among 255 sampled splitters.
constexpr uint32_t kShiftSplit = 0x200u;

// Bucket of key k among the 255 splitters of its segment: the number of
// splitters <= x, x the 32 bits of the key from the sample's highest set bit
// down (saturated above it).  spl[0]: the shift to x; spl[1..255]: the
// splitters as a search tree in level order (children of i at 2i, 2i + 1), so
// that the first six of the eight steps meet no bank twice.  Monotone in the
// key, so it serves as a digit of the split.
__device__ __forceinline__ uint32_t splitter_digit(const uint32_t* spl, uint64_t k) {
    const uint64_t y = k >> spl[0];
    const uint32_t x = (y >> 32) != 0ull ? ~0u : (uint32_t)y;
    uint32_t i = 1;
#pragma unroll
    for (int step = 0; step < 8; ++step) i = 2 * i + (spl[i] <= x ? 1u : 0u);
    return i - 256u;
}

// Splitters of the first split of a segment with clustered keys (Gaussian
// clusters, Morton codes), whose top varying byte would leave most of it in sub-buckets too
// large for the chip: one CTA per segment split at this level draws 2048 keys
// at evenly spaced places (four neighbours each, a sector) and weighs, by the sample, the keys in such
// sub-buckets of the byte split against those in runs of one value too long
// for the chip (which no split on splitters divides).  Where a quarter of the
// keys would be spared a second level, every 8th key of the sorted sample is
// a splitter (spl_mode 1), else the byte split stays (spl_mode 0).  The
// search costs the statistics pass about 0.4 ms per 2^28 keys (its digits are
// kept for the split), a second level of keys alone 2.3 ms.  Segments above kSplMax keys
// take the byte split: 256 sub-buckets of theirs are too large anyway.
constexpr int kSplSample = 2048;
constexpr uint64_t kSplMax = 1ull << 19;
// By default only calls of 4 Mi keys and more, whose segments hold 2^15 keys
// and more on average, are sampled: below that the sample (11 us, and a
// sixteenth of a segment's keys) costs more than a uniform input's call can
// hide, and the 256 byte sub-buckets of a clustered one mostly fit the chip.
constexpr uint64_t kSplMinKeys = 1ull << 22;
constexpr uint64_t kSplMinSeg = 1ull << 15;
// Sort of the sample by the CTA, eight words per thread in, s[0 .. 2047] out: a
// bitonic network on rows of eight in registers, whose steps between threads of
// a warp are shuffles; only the six steps between warps meet shared memory
// (all 66 did: 4096 segments took 242 us, now 100).  Ends with a barrier.
__device__ __forceinline__ void sort_sample(uint32_t (&v)[8], uint32_t* s) {
    static_assert(kSplSample == 8 * 256, "eight words per thread");
    const uint32_t tid = threadIdx.x;
    sort_8(v);
    if (tid & 1u) {  // descending
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t a = v[i];
            v[i] = v[7 - i];
            v[7 - i] = a;
        }
    }
#pragma unroll
    for (uint32_t k = 2; k <= 256; k *= 2) {  // runs of 8 k words from pairs of 4 k
        const bool up = (tid & k) == 0u;
#pragma unroll
        for (uint32_t j = k / 2; j >= 1; j /= 2) {
            const bool low = ((tid & j) == 0u) == up;
            uint32_t o[8];
            if (j >= 32) {
#pragma unroll
                for (int i = 0; i < 8; ++i) s[i * 256 + tid] = v[i];
                __syncthreads();
#pragma unroll
                for (int i = 0; i < 8; ++i) o[i] = s[i * 256 + (tid ^ j)];
                __syncthreads();
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) o[i] = __shfl_xor_sync(0xffffffffu, v[i], j);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = low ? min(v[i], o[i]) : max(v[i], o[i]);
        }
#pragma unroll
        for (int j = 4; j >= 1; j /= 2)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (!(i & j)) {
                    const uint32_t a = min(v[i], v[i | j]), b = max(v[i], v[i | j]);
                    v[i] = up ? a : b;
                    v[i | j] = up ? b : a;
                }
    }
    ((uint4*)s)[2 * tid] = make_uint4(v[0], v[1], v[2], v[3]);
    ((uint4*)s)[2 * tid + 1] = make_uint4(v[4], v[5], v[6], v[7]);
    __syncthreads();
}

__global__ __launch_bounds__(256) void k_seg_sample(const uint64_t* __restrict__ kin, const uint64_t* __restrict__ seg_lo,
                                                    const uint64_t* __restrict__ seg_hi,
                                                    const uint32_t* __restrict__ large_seg,
                                                    const uint32_t* __restrict__ counters, uint64_t flip_in,
                                                    uint32_t chip_max, uint32_t* __restrict__ spl_tab,
                                                    uint8_t* __restrict__ spl_mode) {
    constexpr int kPer = kSplSample / 256;
    __shared__ __align__(16) uint32_t s_x[kSplSample];
    __shared__ uint32_t s_h[kRadix];
    __shared__ unsigned long long s_or[8], s_and[8];
    __shared__ uint32_t s_sum[2];
    const uint32_t id = blockIdx.x;
    if (id >= counters[19]) return;  // uniform
    const uint32_t s = large_seg[id];
    const uint64_t lo = seg_lo[s], n = seg_hi[s] - lo;
    const int tid = threadIdx.x;
    if (tid == 0) spl_mode[id] = 0u;
    if (n > kSplMax) return;  // uniform
    s_h[tid] = 0;
    if (tid < 2) s_sum[tid] = 0;
    uint64_t key[kPer];
    unsigned long long o = 0, an = ~0ull;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const uint32_t q = (uint32_t)(tid + i * 256);  // runs of four neighbours (n > 4096)
        key[i] = kin[lo + (uint64_t)(q >> 2) * (n - 3) / (kSplSample / 4) + (q & 3u)] ^ flip_in;
        o |= key[i];
        an &= key[i];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        o |= __shfl_xor_sync(0xffffffffu, o, off);
        an &= __shfl_xor_sync(0xffffffffu, an, off);
    }
    if ((tid & 31) == 0) { s_or[tid >> 5] = o; s_and[tid >> 5] = an; }
    __syncthreads();
    o = 0; an = ~0ull;
    for (int i = 0; i < 8; ++i) { o |= s_or[i]; an &= s_and[i]; }
    const unsigned long long vary = o ^ an;
    if (vary == 0ull) return;  // uniform: a single value in the sample
    const int sh = 8 * (int)((uint32_t)(63 - __clzll((long long)vary)) >> 3);
#pragma unroll
    for (int i = 0; i < kPer; ++i) atomicAdd(&s_h[(uint32_t)(key[i] >> sh) & 255u], 1u);
    __syncthreads();
    // more sampled keys than this: a sub-bucket above the on-chip size
    const uint32_t thr = (uint32_t)((uint64_t)kSplSample * chip_max / n);
    if (s_h[tid] > thr) atomicAdd(&s_sum[0], s_h[tid]);
    __syncthreads();
    const uint32_t crowded = s_sum[0];
    if (crowded < kSplSample / 4) return;  // uniform
    const int sft = max(0, 32 - __clzll((long long)o));
    uint32_t x[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) x[i] = (uint32_t)(key[i] >> sft);
    sort_sample(x, s_x);
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const uint32_t j = tid + i * 256;
        if (j + thr < (uint32_t)kSplSample && s_x[j] == s_x[j + thr])  // inside a run longer than thr
            atomicAdd(&s_sum[1], j == 0 || s_x[j - 1] != s_x[j] ? thr + 1u : 1u);
    }
    __syncthreads();
    if (crowded < s_sum[1] + kSplSample / 4) return;  // uniform
    uint32_t* spl = spl_tab + (uint64_t)id * kRadix;
    if (tid == 0) {
        spl[0] = (uint32_t)sft;
        spl_mode[id] = 1u;
    } else {
        const int level = 31 - __clz(tid), j = tid - (1 << level);  // node tid of the search tree
        spl[tid] = s_x[(((2 * j + 1) << (7 - level))) * (kSplSample / kRadix) - 1];
    }
}

__device__ __forceinline__ int spec_window(const uint32_t* __restrict__ prev_shift, uint32_t s) {
    // the byte below the parent split's window (a sub-bucket's keys agree on
    // that window and above); the top byte at the first level
    if (!prev_shift) return 7;
    const uint32_t ps = prev_shift[s >> 8];
    return (ps & (kShiftInterp | kShiftSplit)) ? 7 : (ps >= 8 ? (int)(ps >> 3) - 1 : 0);
}

// A tile is skewed when one digit holds more than an eighth of it: the
// split then gives the lanes of a warp that share lane 0's digit their slots
// with one atomic (sorted runs of equal keys hit one counter otherwise).
// Called by all 256 threads with their digit's count.
__device__ __forceinline__ void tile_skew_flag(uint32_t count, uint8_t* __restrict__ tile_skew, uint32_t t) {
    const bool big = count > (uint32_t)(kOsTile / 8);
    const int any = __syncthreads_or(big);
    if (threadIdx.x == 0) tile_skew[t] = any ? 1u : 0u;
}

template <bool SPL>
__global__ __launch_bounds__(256) void k_tile_stats(const uint64_t* __restrict__ kin, const uint64_t* __restrict__ seg_lo,
                                                    const uint64_t* __restrict__ seg_hi, uint64_t nseg,
                                                    const uint32_t* __restrict__ tile_start,
                                                    const uint32_t* __restrict__ tile_seg,
                                                    const uint32_t* __restrict__ large_id, uint16_t* __restrict__ tile_hist,
                                                    uint8_t* __restrict__ tile_skew,
                                                    unsigned long long* __restrict__ vor, unsigned long long* __restrict__ vand,
                                                    const uint64_t* __restrict__ hint_lo, const uint64_t* __restrict__ hint_mult,
                                                    const uint64_t* __restrict__ hint_hi,
                                                    const uint32_t* __restrict__ prev_shift, uint32_t* __restrict__ spec_out,
                                                    uint64_t flip_in, const uint32_t* __restrict__ spl_tab,
                                                    const uint8_t* __restrict__ spl_mode, uint64_t* __restrict__ digits,
                                                    uint32_t pay) {
    __shared__ uint32_t s_h[kRadix];
    __shared__ unsigned long long s_or[8], s_and[8];
    __shared__ uint32_t s_spl[kRadix];
    const uint32_t t = blockIdx.x;
    if (t >= tile_start[nseg]) return;  // uniform
    s_h[threadIdx.x] = 0;
    const uint32_t s = tile_seg[t], id = large_id[s];
    const bool bysplit = SPL && spl_mode[id];  // uniform per CTA
    if (bysplit) s_spl[threadIdx.x] = spl_tab[(uint64_t)id * kRadix + threadIdx.x];
    __syncthreads();
    const uint64_t lo = seg_lo[s], n = seg_hi[s] - lo;
    const uint32_t ti = t - tile_start[s];
    const uint64_t a = (uint64_t)ti * kOsTile, b = min(n, a + kOsTile);
    const bool win = hint_lo != nullptr;
    const int spec = spec_window(prev_shift, s);
    if (ti == 0 && threadIdx.x == 0) spec_out[id] = (uint32_t)spec;
    if (win && hint_hi && hint_hi[s] == hint_lo[s]) {
        // every key of the segment equals the one the parent's split saw: no read
        if (threadIdx.x == 0) {
            atomicOr(&vor[id], (unsigned long long)hint_lo[s]);
            atomicAnd(&vand[id], (unsigned long long)hint_lo[s]);
        }
        tile_hist[(uint64_t)t * (2 * kRadix) + threadIdx.x] = (uint16_t)(threadIdx.x == 0 ? b - a : 0);
        if (threadIdx.x == 0) tile_skew[t] = 1u;
        return;
    }
    const uint64_t hb = win ? hint_lo[s] : 0ull;
    const uint64_t hm = win ? hint_mult[s] : 0ull;
    const int sh = 8 * spec;
    unsigned long long o = 0, an = ~0ull;
    auto count = [&](auto digit) {
#pragma unroll 4
        for (uint64_t e = a + threadIdx.x; e < b; e += 256) {
            const uint64_t k = kin[lo + e] ^ flip_in;
            o |= k;
            an &= k;
            atomicAdd(&s_h[digit(k)], 1u);
        }
    };
    if (SPL && bysplit && digits) {
        // The digits, a search each, are kept for the split: 16 bytes of a
        // thread (8 and 8 with a payload), in the order of the split's threads.
        // Per 2^28 keys this pass takes 80 us more, the split 370 less alone
        // (1342 -> 972) and 480 with a payload (2125 -> 1646).
        const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        static_assert(kOsTile == 16 * 256, "four words of digits per thread");
        const uint64_t* g = kin + lo + a;
        const uint32_t m = (uint32_t)(b - a), e0 = pay ? 2 * w * 256 + lane : threadIdx.x, step = pay ? 32u : 256u;
        uint32_t q[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint64_t k[4];
            uint32_t d[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t e = e0 + (4 * c + i) * step;
                k[i] = (e < m ? g[e] : g[m - 1]) ^ flip_in;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                o |= k[i];
                an &= k[i];
                d[i] = splitter_digit(s_spl, k[i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (e0 + (4 * c + i) * step < m) atomicAdd(&s_h[d[i]], 1u);
                else d[i] = kRadix - 1;  // behind all others
            }
            q[c] = d[0] | d[1] << 8 | d[2] << 16 | d[3] << 24;
        }
        uint2* out = (uint2*)((uint8_t*)(digits + lo) + a);
        out[pay ? 2 * w * 32 + lane : 2 * threadIdx.x] = make_uint2(q[0], q[1]);
        out[pay ? (2 * w + 1) * 32 + lane : 2 * threadIdx.x + 1] = make_uint2(q[2], q[3]);
    } else if (SPL && bysplit)
        count([&](uint64_t k) { return splitter_digit(s_spl, k); });
    else if (win)
        count([&](uint64_t k) { return split_digit(k, 0, hb, hm); });
    else
        count([&](uint64_t k) { return (uint32_t)(k >> sh) & 255u; });
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        o |= __shfl_xor_sync(0xffffffffu, o, off);
        an &= __shfl_xor_sync(0xffffffffu, an, off);
    }
    if ((threadIdx.x & 31) == 0) { s_or[threadIdx.x >> 5] = o; s_and[threadIdx.x >> 5] = an; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long x = 0, y = ~0ull;
        for (int i = 0; i < 8; ++i) { x |= s_or[i]; y &= s_and[i]; }
        atomicOr(&vor[id], x);
        atomicAnd(&vand[id], y);
    }
    tile_hist[(uint64_t)t * (2 * kRadix) + threadIdx.x] = (uint16_t)s_h[threadIdx.x];
    tile_skew_flag(s_h[threadIdx.x], tile_skew, t);
}

// Recount of the tiles of segments whose top varying byte (from the OR/AND of
// the statistics pass) is not the speculative one: the histogram of that byte
// into the tile's second row.  CTA b owns tiles b, b + gridDim.x, ...; its 256
// threads look at one each, so a level that needs none costs one chain of loads
// (2^28 keys in 1024 segments: 63 us by a tile per step of a CTA, 6.4 here),
// and a segment that needs one is spread over all CTAs however few segments
// there are (keys below 2^40, 2^27 of them in one segment: the sort takes
// 5.6 ms, 16.5 with eight CTAs per segment).
__global__ __launch_bounds__(256) void k_tile_recount(
    const uint64_t* __restrict__ kin, const uint64_t* __restrict__ seg_lo, const uint64_t* __restrict__ seg_hi,
    uint32_t tiles, const uint32_t* __restrict__ tile_start, const uint32_t* __restrict__ tile_seg,
    const uint32_t* __restrict__ large_id, uint16_t* __restrict__ tile_hist, uint8_t* __restrict__ tile_skew,
    const uint8_t* __restrict__ spl_mode, const unsigned long long* __restrict__ vor,
    const unsigned long long* __restrict__ vand, const uint32_t* __restrict__ spec, uint64_t flip_in) {
    __shared__ uint32_t s_h[kRadix];
    __shared__ uint32_t s_todo[8];  // the CTA's tiles to count again, a bit each
    __shared__ uint64_t s_at[256];   // their first keys
    __shared__ uint16_t s_cnt[256];  // and numbers of them
    __shared__ uint8_t s_byte[256];
    for (uint64_t first = blockIdx.x; first < tiles; first += (uint64_t)256 * gridDim.x) {  // uniform per CTA
        const uint64_t mine = first + (uint64_t)threadIdx.x * gridDim.x;
        bool again = false;
        if (mine < tiles) {
            const uint32_t s = tile_seg[mine], id = large_id[s];
            const unsigned long long vary = vor[id] ^ vand[id];
            // on sampled splitters the statistics pass has counted the buckets
            if (vary != 0ull && !(spl_mode && spl_mode[id])) {
                const uint32_t w = (uint32_t)(63 - __clzll((long long)vary)) >> 3;
                again = w != spec[id];
                if (again) {
                    const uint64_t a = seg_lo[s] + (mine - tile_start[s]) * kOsTile;
                    s_at[threadIdx.x] = a;
                    s_cnt[threadIdx.x] = (uint16_t)min((uint64_t)kOsTile, seg_hi[s] - a);
                    s_byte[threadIdx.x] = (uint8_t)w;
                }
            }
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, again);
        if ((threadIdx.x & 31) == 0) s_todo[threadIdx.x >> 5] = bal;
        __syncthreads();
        for (uint32_t v = 0; v < 8; ++v) {
            for (uint32_t left = s_todo[v]; left; left &= left - 1) {
                const uint32_t i = 32 * v + (uint32_t)(__ffs(left) - 1);
                const uint32_t t = (uint32_t)(first + (uint64_t)i * gridDim.x), m = s_cnt[i];
                const uint64_t* g = kin + s_at[i];
                const int sh = 8 * (int)s_byte[i];
                s_h[threadIdx.x] = 0;
                __syncthreads();
#pragma unroll 4
                for (uint32_t e = threadIdx.x; e < m; e += 256)
                    atomicAdd(&s_h[(uint32_t)((g[e] ^ flip_in) >> sh) & 255u], 1u);
                __syncthreads();
                tile_hist[(uint64_t)t * (2 * kRadix) + kRadix + threadIdx.x] = (uint16_t)s_h[threadIdx.x];
                tile_skew_flag(s_h[threadIdx.x], tile_skew, t);  // ends with a barrier
            }
        }
        __syncthreads();  // s_todo is written again
    }
}

// Per large segment (thread d = digit d): the split window, the digit totals
// (summed over the segment's tile histograms), their exclusive offsets, the
// bounds of the 256 sub-buckets (empty when the keys are all equal), and the
// destination of every tile's digit-d keys: the digit's offset plus the
// digit-d keys of the segment's earlier tiles.
__global__ __launch_bounds__(256) void k_msd_prep(const uint64_t* __restrict__ seg_lo, const uint32_t* __restrict__ large_seg,
                                                  const uint32_t* __restrict__ counters,
                                                  const uint32_t* __restrict__ tile_start,
                                                  const uint16_t* __restrict__ tile_hist,
                                                  const unsigned long long* __restrict__ vor,
                                                  const unsigned long long* __restrict__ vand, const uint64_t* __restrict__ hint_lo,
                                                  const uint64_t* __restrict__ hint_mult, uint64_t* __restrict__ msd_base,
                                                  uint64_t* __restrict__ msd_mult, uint32_t* __restrict__ msd_shift,
                                                  const uint32_t* __restrict__ spec, uint32_t* __restrict__ direct,
                                                  uint64_t* __restrict__ sub_lo, uint64_t* __restrict__ sub_hi,
                                                  uint32_t* __restrict__ tile_off, uint32_t chip_max,
                                                  uint32_t* __restrict__ large_mask, uint32_t* __restrict__ any_large,
                                                  uint64_t* __restrict__ cmin, uint64_t* __restrict__ cmax,
                                                  uint32_t level_chip_max, uint32_t pack_keys,
                                                  const uint8_t* __restrict__ spl_mode) {
    __shared__ uint32_t s_c[kRadix], s_x[kRadix + 1], s_warp[32], s_end[kRadix];
    __shared__ uint16_t s_jump[8][kRadix + 1];  // packing: 2^i packs ahead of each sub-bucket
    __shared__ uint32_t s_big[8];               // packing: sub-buckets split again, one bit each
    __shared__ uint8_t s_first[kRadix];         // packing: the sub-bucket starts a pack
    const uint32_t id = blockIdx.x;
    if (id >= counters[19]) return;
    const uint32_t s = large_seg[id];
    const uint64_t lo = seg_lo[s];
    const unsigned long long vary = vor[id] ^ vand[id];
    uint32_t shift = 0, row;
    uint64_t base = 0, mult = 0;
    if (hint_lo) {
        base = hint_lo[s];
        mult = hint_mult[s];
        row = 0;
    } else {
        const uint32_t w = vary ? (uint32_t)(63 - __clzll((long long)vary)) >> 3 : spec[id];
        shift = 8 * w;
        row = w == spec[id] ? 0u : 1u;
    }
    const bool bysplit = spl_mode && spl_mode[id];
    if (bysplit) row = 0;
    const bool dir = vary == 0ull;
    const uint32_t d = threadIdx.x;
    const uint32_t t0 = tile_start[s], t1 = tile_start[s + 1];
    const uint16_t* h = tile_hist + row * kRadix + d;
    uint32_t total = 0;
    for (uint32_t t = t0; t < t1; ++t) total += h[(uint64_t)t * (2 * kRadix)];
    s_c[d] = total;
    __syncthreads();
    scan256_smem<256>(s_c, s_x, s_warp);
    const uint32_t x = s_x[d];
    // Packing: runs of consecutive sub-buckets sorted on chip (each at most
    // level_chip_max keys) are merged greedily into packs of at most
    // pack_keys keys; the keys of consecutive sub-buckets are in order
    // between them, so the next level sorting a pack as one segment sorts
    // each.  s_end[d]: end offset of the pack that starts at sub-bucket d,
    // or ~0 when d belongs to an earlier pack (it becomes empty).  Sub-buckets
    // split again stand alone.
    // Nothing to pack unless two neighbouring sub-buckets fit one pack
    // (uniform keys: none do, and the serial walk below is skipped).
    const bool pair_fits = d + 1 < (uint32_t)kRadix && total + s_c[d + 1] <= pack_keys && total + s_c[d + 1] > 0u;
    const bool packable = __syncthreads_or(pair_fits) != 0;
    if (packable) {  // uniform per CTA
        // The greedy walk over the sub-buckets in order (a sub-bucket split
        // again stands alone; otherwise a pack takes sub-buckets while they
        // add up to at most pack_keys), computed in parallel: next[d], the
        // sub-bucket after the pack that would start at d, by a bit search
        // and a binary search; the packs reachable from sub-bucket 0 by
        // pointer doubling (thread m finds the m-th pack's start).
        const bool big = total > level_chip_max;
        const uint32_t bal = __ballot_sync(0xffffffffu, big);
        if ((d & 31) == 0) s_big[d >> 5] = bal;
        if (d == 0) s_x[kRadix] = s_x[kRadix - 1] + s_c[kRadix - 1];
        __syncthreads();
        uint32_t nxt;
        if (big) {
            nxt = d + 1;
        } else {
            uint32_t fb = kRadix;  // the first sub-bucket after d split again
            for (uint32_t wd = (d + 1) >> 5; wd < 8; ++wd) {
                const uint32_t m = s_big[wd] & (wd == ((d + 1) >> 5) ? ~0u << ((d + 1) & 31) : ~0u);
                if ((d + 1) < (uint32_t)kRadix && m) { fb = wd * 32 + (uint32_t)(__ffs(m) - 1); break; }
            }
            // the first j > d whose keys would take the pack past pack_keys:
            // the first m >= d + 2 with s_x[m] > s_x[d] + pack_keys, j = m - 1
            const uint32_t lim = x + pack_keys;
            uint32_t lo = d + 2, hi = kRadix + 1;  // search m in [lo, hi)
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (s_x[mid] > lim) hi = mid; else lo = mid + 1;
            }
            const uint32_t fs = lo <= (uint32_t)kRadix ? lo - 1 : (uint32_t)kRadix;
            nxt = min(fb, fs);
        }
        s_jump[0][d] = (uint16_t)nxt;
        if (d == 0) s_jump[0][kRadix] = (uint16_t)kRadix;
        s_first[d] = 0;
        __syncthreads();
        for (int i = 1; i < 8; ++i) {
            const uint32_t a = s_jump[i - 1][d];
            s_jump[i][d] = a < (uint32_t)kRadix ? s_jump[i - 1][a] : (uint16_t)kRadix;
            if (d == 0) s_jump[i][kRadix] = (uint16_t)kRadix;
            __syncthreads();
        }
        uint32_t pos = 0;  // start of pack number d
        for (int i = 0; i < 8 && pos < (uint32_t)kRadix; ++i)
            if ((d >> i) & 1u) pos = s_jump[i][pos];
        if (pos < (uint32_t)kRadix) s_first[pos] = 1;
        __syncthreads();
        s_end[d] = s_first[d] ? s_x[nxt] : ~0u;
    }
    if (!packable) s_end[d] = x + total;
    __syncthreads();
    const uint32_t pend = s_end[d];
    sub_lo[(uint64_t)id * kRadix + d] = dir ? lo : lo + x;
    sub_hi[(uint64_t)id * kRadix + d] = dir ? lo : lo + (pend == ~0u ? x : pend);
    // sub-buckets that the next level splits again: the split pass gathers
    // their smallest and largest key
    const bool large = !dir && total > chip_max;  // chip_max = ~0: nothing gathered
    const uint32_t bal = __ballot_sync(0xffffffffu, large);
    if ((d & 31) == 0) large_mask[(uint64_t)id * 8 + (d >> 5)] = bal;
    if (d == 0) any_large[id] = 0u;
    if (chip_max != ~0u) {  // key ranges are gathered at this level
        cmin[(uint64_t)id * kRadix + d] = ~0ull;
        cmax[(uint64_t)id * kRadix + d] = 0ull;
    }
    __syncthreads();
    if (bal && (d & 31) == 0) atomicOr(&any_large[id], 1u);
    uint32_t run = x;
    for (uint32_t t = t0; t < t1; ++t) {
        tile_off[(uint64_t)t * kRadix + d] = run;
        run += h[(uint64_t)t * (2 * kRadix)];
    }
    if (d == 0) {
        msd_shift[id] = shift | (hint_lo ? kShiftInterp : 0u) | (bysplit ? kShiftSplit : 0u);
        msd_base[id] = base;
        msd_mult[id] = mult;
        direct[id] = dir ? 1u : 0u;
    }
}

// ---------------------------------------------------------------------------
// The split pass: stable scatter of every large segment on its window, one
// CTA per tile of every large segment, each tile to the offsets k_msd_prep
// assigned it.
// ---------------------------------------------------------------------------
struct SplitArgs {
    const uint64_t* kin;
    uint64_t* kout;      // next level
    uint64_t* kfinal;    // output (segments whose keys are all equal)
    const uint32_t* pin;
    uint32_t* pout;
    uint32_t* pfinal;
    const uint64_t* seg_lo;
    const uint64_t* seg_hi;
    uint64_t nseg;
    const uint32_t* tile_start;
    const uint32_t* tile_seg;
    const uint32_t* large_id;
    const uint32_t* tile_off;  // [tile][256] destination of the tile's digit-d keys, relative to the segment
    const uint8_t* tile_skew;  // [tile] one digit holds more than an eighth of the tile
    const uint64_t* digits;    // splitter digits kept by the statistics pass, a byte per key from the segment's start (or null)
    const uint32_t* spl_tab;   // [large id][256] sampled splitters (segments split with kShiftSplit)
    const uint32_t* msd_shift;
    const uint64_t* msd_base;
    const uint64_t* msd_mult;
    const uint32_t* direct;
    const uint32_t* large_mask;  // [large id][8] sub-buckets that the next level splits again
    const uint32_t* any_large;
    uint64_t* cmin;              // their smallest and largest key (atomics)
    uint64_t* cmax;
    uint32_t* err;
    uint64_t flip_in;
    uint64_t flip_out;
    uint32_t scatter;  // 1: tiles that gather no key ranges write each key straight to its run
};

// The tile's shape: keys alone 256 threads x 16 keys, with a payload 512 x 8.
template <bool PAY>
constexpr int split_threads() { return PAY ? 512 : 256; }

constexpr int kCellShift = 4;  // splitter digits, keys alone: a cell of the digit order is 16 keys
template <bool PAY, bool SPL>
constexpr size_t split_smem(bool gather) {
    return (size_t)(kOsTile + 2) * 8 + (PAY ? (size_t)(kOsTile + 8) * 4 : 0) + (size_t)kOsTile * 2 +
           (SPL && PAY ? (size_t)kOsTile : 0) + (PAY ? (size_t)(split_threads<PAY>() / 32) * kRadix * 2 : 0) +
           (gather ? 2 * (size_t)kRadix * 8 : 0);
}

// One bulk copy brings the tile's keys (and payload) into shared memory, where
// they stay; what is put into digit order is a 16-bit index per key, and the
// tile is then written run by run through it.  So no thread holds its keys in
// registers across the ranking (64 registers and half the warps of an SM
// before), and shared memory sees 2 bytes per key scattered instead of 9 (13).
// Bound by shared-memory wavefronts (87% of their peak keys alone, 74% with a
// payload: the counting atomics, the index scatter and the key gather meet
// random banks).  2^28 keys, 256-way: keys alone 1.10 -> 0.90 ms, with a
// payload 2.50 -> 1.95 ms.  Keys alone with 512 threads: 6% slower.
template <bool PAY, bool SPL>
__global__ __launch_bounds__(split_threads<PAY>(), PAY ? 3 : 5) void k_split(const SplitArgs A) {
    constexpr int kThreads = split_threads<PAY>();
    constexpr int kWarps = kThreads / 32;
    constexpr int kItems = kOsTile / kThreads;
    extern __shared__ __align__(16) unsigned char os_smem[];
    uint64_t* s_keys = (uint64_t*)os_smem;                         // kOsTile + 2: key e at [e + hd]
    uint32_t* s_pay = (uint32_t*)(s_keys + kOsTile + 2);           // kOsTile + 8 (PAY): payload e at [e + po]
    uint16_t* s_hist = (uint16_t*)(s_pay + (PAY ? kOsTile + 8 : 0));  // kWarps * 256 (PAY)
    uint16_t* s_idx = s_hist + (PAY ? kWarps * kRadix : 0);        // kOsTile: the keys in digit order
    uint8_t* s_dg = (uint8_t*)(s_idx + kOsTile);                   // kOsTile (SPL, PAY): their digits
    uint64_t* s_mn = (uint64_t*)(s_dg + (SPL && PAY ? kOsTile : 0));  // 2 x 256 (gather): key ranges of sub-buckets
    uint64_t* s_mx = s_mn + kRadix;
    __shared__ uint32_t s_total[kRadix], s_start[kRadix];
    __shared__ uint32_t s_gbase[kRadix];  // start of the digit's run in the segment, less its start in the tile
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_spl[SPL ? kRadix : 1];
    __shared__ uint8_t s_cell[SPL && !PAY ? kRadix : 1];  // digit of the cell's first key in digit order
    static_assert((kOsTile >> kCellShift) == kRadix, "a cell per thread");
    __shared__ uint32_t s_mask[8];
    __shared__ uint64_t s_bar;

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t total_tiles = A.tile_start[A.nseg];
    const uint32_t t = blockIdx.x;
    if (t >= total_tiles) return;  // uniform
    const uint32_t s = A.tile_seg[t];
    const uint32_t id = A.large_id[s];
    const uint64_t seg_base = A.seg_lo[s];
    const uint32_t seg_n = (uint32_t)(A.seg_hi[s] - seg_base);  // below 2^30
    const uint32_t tile_lo = (t - A.tile_start[s]) * (uint32_t)kOsTile;
    const uint32_t count = min((uint32_t)kOsTile, seg_n - tile_lo);
    const int shift = (int)(A.msd_shift[id] & 0xffu);
    const uint64_t dbase = A.msd_base[id];
    const uint64_t dmult = A.msd_mult[id];
    // SPL: this level's segments may split on sampled splitters (uniform per CTA)
    const bool bysplit = SPL && (A.msd_shift[id] & kShiftSplit) != 0u;
    const bool dir = A.direct[id] != 0u;
    const uint64_t flip_out = dir ? A.flip_out : 0ull;
    // A segment of one key value already in place in the output (every
    // second level reads the output buffer) needs no copy at all.
    if (dir && A.kin == A.kfinal && flip_out == 0ull && (!PAY || A.pin == A.pfinal)) return;
    uint64_t* kout = (dir ? A.kfinal : A.kout) + seg_base;
    uint32_t* pout = PAY ? (dir ? A.pfinal : A.pout) + seg_base : nullptr;
    const uint64_t* g = A.kin + seg_base + tile_lo;
    const uint32_t* gp = PAY ? A.pin + seg_base + tile_lo : nullptr;
    // One key value: every key keeps its place, so a payload needs no ranking
    // (2^26 equal keys in 1024 segments: local sort 864 -> 640 us).  Keys alone
    // gain nothing by it.
    if (PAY && dir) {
#pragma unroll 4
        for (uint32_t e = tid; e < count; e += kThreads) {
            kout[tile_lo + e] = g[e] ^ A.flip_in ^ flip_out;
            pout[tile_lo + e] = gp[e];
        }
        return;
    }
    // The tile: 16-byte aligned middle by a bulk copy, the ends by small ones.
    const uint32_t hd = (uint32_t)(((uintptr_t)g >> 3) & 1u), m = ((count - hd) >> 1) << 1;
    const uint32_t po = PAY ? (uint32_t)(((uintptr_t)gp >> 2) & 3u) : 0u;
    const uint32_t ph = PAY ? min(count, (4u - po) & 3u) : 0u, pm = PAY ? ((count - ph) >> 2) << 2 : 0u;
    if (tid == 0) {
        mbar_init(&s_bar, 1u);
        mbar_arrive_expect_tx(&s_bar, m * 8u + pm * 4u);
        if (m) bulk_load(s_keys + 2 * hd, g + hd, m * 8u, &s_bar);
        if (PAY && pm) bulk_load(s_pay + po + ph, gp + ph, pm * 4u, &s_bar);
    }
    if (hd && tid == 32) cp_async8(&s_keys[1], g);
    if (hd + m < count && tid == 33) cp_async8(&s_keys[count - 1 + hd], g + count - 1);
    if (PAY) {
        if (tid >= 40 && (uint32_t)(tid - 40) < ph) cp_async4(&s_pay[po + tid - 40], gp + tid - 40);
        if (tid >= 44 && tid < 48 && ph + pm + (uint32_t)(tid - 44) < count)
            cp_async4(&s_pay[po + ph + pm + tid - 44], gp + ph + pm + tid - 44);
    }
    cp_async_commit();
    const bool gather = A.any_large[id] != 0u;  // some sub-bucket is split again: note its key range
    if (gather) {
        if (tid < kRadix) { s_mn[tid] = ~0ull; s_mx[tid] = 0ull; }
        if (tid < 8) s_mask[tid] = A.large_mask[(uint64_t)id * 8 + tid];
    }
    const bool kept = SPL && bysplit && !dir && A.digits != nullptr;  // (a segment of one value writes where they lie)
    uint32_t dk[kItems / 4] = {};
    if (kept) {
        const uint2* q = (const uint2*)((const uint8_t*)(A.digits + seg_base) + tile_lo) + tid * (kItems / 8);
#pragma unroll
        for (int i = 0; i < kItems / 8; ++i) { dk[2 * i] = q[i].x; dk[2 * i + 1] = q[i].y; }
    }
    if (SPL && bysplit && !kept && tid < kRadix) s_spl[tid] = A.spl_tab[(uint64_t)id * kRadix + tid];
    if (!PAY && tid < kRadix) s_total[tid] = 0;
    cp_async_wait_all();
    __syncthreads();  // the barrier is initialised, the small copies have landed
    if (__syncthreads_or(!mbar_wait(&s_bar, 0u))) {  // uniform; not expected: a bulk copy that never landed
        if (tid == 0) {
            atomicOr(A.err, kDevErrTimeout);
            mbar_wait(&s_bar, 0u);  // the CTA's memory stays until the copy is done, or once more the limit
        }
        return;
    }
    const uint64_t* keys = s_keys + hd;
    const uint32_t* pays = s_pay + po;
    auto digit = [&](uint64_t k) -> uint32_t {  // of a key as read
        k ^= A.flip_in;
        if (SPL && bysplit) return splitter_digit(s_spl, k);
        return split_digit(k, shift, dbase, dmult);
    };
    const bool direct = A.scatter && !gather;  // uniform per CTA: each key straight to its run
    const uint64_t flip = A.flip_in ^ flip_out;
    const uint32_t off_d = tid < kRadix ? A.tile_off[(uint64_t)t * kRadix + tid] : 0u;
    auto put = [&](uint32_t dst, uint32_t e) {
        if (dst >= seg_n) {  // never taken when the digit offsets are consistent
            atomicOr(A.err, kDevErrBounds);
            return;
        }
        kout[dst] = keys[e] ^ flip;
        if (PAY) pout[dst] = pays[e];
    };
    // SPL, keys alone: the digit of place j in digit order, the last of [lo, hi]
    // that starts at or before j.  Two neighbouring cells bound it: a cell per
    // 16 keys and a step or two of search take 256 bytes, where a digit per key
    // takes 4 KB and with it one of five CTAs of an SM (2^28 uniform keys, a
    // level that may split on splitters: 1090 us with those, 975 with cells).
    // With a payload three CTAs fit either way and the digits are cheaper (by
    // 5% of the pass).
    auto last_start = [&](uint32_t lo, uint32_t hi, uint32_t j) -> uint32_t {
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) >> 1;
            if (s_start[mid] <= j) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    if constexpr (PAY) {
        // Each key's digit once, byte-packed (past the segment the last one).
        const uint32_t wbase = w * 32 * kItems + lane;
        if (!kept)
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const uint32_t e = wbase + i * 32;
                dk[i >> 2] |= (e < count ? digit(keys[e]) : (uint32_t)kRadix - 1u) << (8 * (i & 3));
            }
        auto digit_of = [&](int i) -> uint32_t { return (dk[i >> 2] >> (8 * (i & 3))) & 255u; };
        block_rank<kWarps, kItems>(
            digit_of, s_hist, s_total, s_start, s_warp,
            [&]() {
                if (tid < kRadix) s_gbase[tid] = off_d - s_start[tid];
            },
            [&](int i, uint32_t rank) {
                const uint32_t e = wbase + i * 32;
                if (direct) {
                    if (e < count) put(s_gbase[digit_of(i)] + rank, e);
                } else {
                    s_idx[rank] = (uint16_t)e;
                    if (SPL && bysplit) s_dg[rank] = (uint8_t)digit_of(i);
                }
            });
        if (direct) return;
    } else {
        // Keys alone: equal keys are indistinguishable, so the order of a
        // digit's keys inside the tile is free and one shared counter per
        // digit hands out the slots (one atomic per key instead of the
        // ballot ranking the payload path needs for stability).  rank[i]
        // holds the digit and, from bit 8, the key's slot.  (Aggregating the
        // lanes of a warp that share a digit with a match instruction costs
        // more than it saves, even on heavily duplicated keys.)
        if (direct && tid < kRadix) s_gbase[tid] = off_d;  // digit d's keys of this tile start here
        uint32_t rank[kItems];
        if (kept) {
#pragma unroll
            for (int i = 0; i < kItems; ++i)
                rank[i] = tid + i * kThreads < count ? (dk[i >> 2] >> (8 * (i & 3))) & 255u : (uint32_t)kRadix;
        } else if (SPL && bysplit) {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const uint32_t e = tid + i * kThreads;
                rank[i] = e < count ? splitter_digit(s_spl, keys[e] ^ A.flip_in) : (uint32_t)kRadix;
            }
        } else {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const uint32_t e = tid + i * kThreads;
                rank[i] = e < count ? split_digit(keys[e] ^ A.flip_in, shift, dbase, dmult) : (uint32_t)kRadix;
            }
        }
        if (A.tile_skew[t]) {  // uniform per CTA: see tile_skew_flag
            const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const uint32_t d = rank[i];
                const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
                const uint32_t eq = __ballot_sync(0xffffffffu, d == d0);
                uint32_t b0 = 0;
                if (lane == 0 && d0 < (uint32_t)kRadix) b0 = atomicAdd(&s_total[d0], (uint32_t)__popc(eq));
                b0 = __shfl_sync(0xffffffffu, b0, 0);
                if (d < (uint32_t)kRadix)
                    rank[i] = d | ((d == d0 ? b0 + (uint32_t)__popc(eq & lt_mask) : atomicAdd(&s_total[d], 1u)) << 8);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kItems; ++i)
                if (rank[i] < (uint32_t)kRadix) rank[i] |= atomicAdd(&s_total[rank[i]], 1u) << 8;
        }
        __syncthreads();
        if (direct) {
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
                const uint32_t e = tid + i * kThreads;
                if (e < count) put(s_gbase[rank[i] & 255u] + (rank[i] >> 8), e);
            }
            return;
        }
        scan256_smem<kThreads>(s_total, s_start, s_warp);
        if (tid < kRadix) s_gbase[tid] = off_d - s_start[tid];
        if (SPL && bysplit && tid < kRadix)
            s_cell[tid] = (uint8_t)last_start(0u, kRadix - 1u, (uint32_t)tid << kCellShift);
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const uint32_t e = tid + i * kThreads;
            if (e < count) s_idx[s_start[rank[i] & 255u] + (rank[i] >> 8)] = (uint16_t)e;
        }
    }
    // The tile's digit-d keys go to the offsets the statistics scan assigned
    // to this tile (digit offset plus the earlier tiles' digit-d keys).
    __syncthreads();
    auto digit_at = [&](uint32_t j, uint64_t k) -> uint32_t {
        if (SPL && PAY && bysplit) return s_dg[j];
        if (SPL && bysplit) {
            const uint32_t c = j >> kCellShift;
            return last_start(s_cell[c], c + 1 < (uint32_t)kRadix ? s_cell[c + 1] : (uint32_t)kRadix - 1u, j);
        }
        return split_digit(k ^ A.flip_in, shift, dbase, dmult);
    };
#pragma unroll 4
    for (uint32_t j = tid; j < count; j += kThreads) {
        const uint32_t e = s_idx[j];
        put(s_gbase[digit_at(j, keys[e])] + j, e);
    }
    if (gather) {  // uniform per CTA
        // Smallest and largest key of every sub-bucket the next level splits
        // again (its digit range there).  The keys come in digit runs, so a
        // warp usually reduces one run and issues one atomic pair.
        for (uint32_t j0 = (uint32_t)w * 32; j0 < count; j0 += kThreads) {
            const uint32_t j = j0 + lane;
            const bool v = j < count;
            const uint64_t raw = v ? keys[s_idx[j]] : 0ull, k = raw ^ A.flip_in;
            const uint32_t d = v ? digit_at(j, raw) : 0x1ffu;
            const bool flagged = v && ((s_mask[d >> 5] >> (d & 31)) & 1u);
            const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
            if (__all_sync(0xffffffffu, d == d0)) {
                if (flagged) {  // the whole warp: one digit
                    uint64_t mn = k, mx = k;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        mn = min(mn, (uint64_t)__shfl_xor_sync(0xffffffffu, mn, o));
                        mx = max(mx, (uint64_t)__shfl_xor_sync(0xffffffffu, mx, o));
                    }
                    if (lane == 0) {
                        if (mn < s_mn[d]) atomicMin((unsigned long long*)&s_mn[d], (unsigned long long)mn);
                        if (mx > s_mx[d]) atomicMax((unsigned long long*)&s_mx[d], (unsigned long long)mx);
                    }
                }
            } else if (flagged) {
                if (k < s_mn[d]) atomicMin((unsigned long long*)&s_mn[d], (unsigned long long)k);
                if (k > s_mx[d]) atomicMax((unsigned long long*)&s_mx[d], (unsigned long long)k);
            }
        }
        __syncthreads();
        if (tid < kRadix && ((s_mask[tid >> 5] >> (tid & 31)) & 1u) && s_mx[tid] >= s_mn[tid]) {
            atomicMin((unsigned long long*)&A.cmin[(uint64_t)id * kRadix + tid], (unsigned long long)s_mn[tid]);
            atomicMax((unsigned long long*)&A.cmax[(uint64_t)id * kRadix + tid], (unsigned long long)s_mx[tid]);
        }
    }
}

// The digit of the next split of every sub-bucket that will be split again:
// its own key range [min, max] interpolated onto 2^b sub-buckets, b chosen so
// that they hold about `target` keys on average; a sub-bucket of one key
// value keeps multiplier 0.  An interpolated split into 2^b sub-buckets
// narrows the key range by a factor of about 2^b - 1, and (rounding of short
// ranges included) of at least 2^(b-1) for b >= 2, whatever the keys, so
// b is at least ceil(B / levels) + 1 for a range of B bits and `levels`
// levels left before the depth limit (one kept for the copy of single-valued
// sub-buckets): clustered keys with a few outliers then still end within the
// limit (each level keeps B / levels from growing).
__global__ void k_child_hints(uint32_t n_children, const uint64_t* __restrict__ sub_lo, const uint64_t* __restrict__ sub_hi,
                              const uint64_t* __restrict__ cmin, const uint64_t* __restrict__ cmax,
                              uint64_t* __restrict__ cmult, uint32_t chip_max, uint32_t target, uint32_t child_depth) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_children) return;
    const uint64_t n = sub_hi[c] - sub_lo[c];
    if (n <= chip_max) return;
    const uint64_t lo = cmin[c], hi = cmax[c];
    if (hi < lo) return;  // no key seen (cannot happen for a non-empty sub-bucket)
    const uint32_t want = (uint32_t)min((n + target - 1) / target, (uint64_t)kRadix);  // sub-buckets wanted
    uint32_t b = 1;
    while (b < 8 && (1u << b) < want) ++b;
    const int levels = kMaxDepth - (int)child_depth - 1;
    const uint32_t B = hi > lo ? 64u - (uint32_t)__clzll((long long)(hi - lo)) : 0u;
    const uint32_t b_min = levels >= 1 ? min(8u, (B + (uint32_t)levels - 1u) / (uint32_t)levels + 1u) : 8u;
    b = max(b, b_min);
    cmult[c] = interp_hint(hi - lo, 1u << b);
}

__global__ void k_even_offsets(uint64_t* __restrict__ seg_off, uint64_t N, uint64_t p) {
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s <= p) seg_off[s] = (uint64_t)(((unsigned __int128)s * N) / p);
}

cudaError_t fill_even_offsets(uint64_t* d_seg_off, uint64_t N, uint64_t p, cudaStream_t st) {
    const uint64_t n = p + 1;
    HSS_LAUNCH(k_even_offsets, (unsigned)ceil_div(n, 256), 256, 0, st, d_seg_off, N, p);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Host driver.
// ---------------------------------------------------------------------------
static int num_sms() { return device_sm_count(); }

template <bool PAY, int THREADS, int CAP, int R, bool FEW>
static cudaError_t launch_chip(const uint64_t* in, uint64_t* out, const uint32_t* pin, uint32_t* pout,
                               const uint64_t* seg_lo, const uint64_t* seg_hi, const uint32_t* list,
                               const uint32_t* nlist, uint64_t count, uint64_t nseg, uint32_t min_n, uint32_t max_n,
                               uint64_t fin, uint64_t fout, uint32_t* err, cudaStream_t st) {
    constexpr size_t smem = chip_smem<PAY, THREADS, CAP, R>();
    const void* fn = (const void*)k_chip<PAY, THREADS, CAP, R, FEW>;
    {
        // all of L1 as shared memory: the CTAs per SM are limited by their buffers
        const cudaError_t e = ensure_func_attrs(fn, (int)smem, 100);
        if (e != cudaSuccess) return e;
    }
    const int per_sm = resident_ctas(fn, THREADS, smem);
    const uint64_t grid = std::min<uint64_t>(count, (uint64_t)num_sms() * per_sm);
    if (grid == 0) return cudaSuccess;
    HSS_LAUNCH((k_chip<PAY, THREADS, CAP, R, FEW>), (unsigned)grid, THREADS, smem, st, in, out, pin, pout, seg_lo, seg_hi, list,
               nlist, nseg, min_n, max_n, fin, fout, err);
    return cudaGetLastError();
}

struct Level {
    const uint64_t* in;
    const uint32_t* pin;
    const uint64_t* seg_lo;
    const uint64_t* seg_hi;
    uint64_t nseg;
    uint64_t flip_in;
    const uint64_t* hint_lo;
    const uint64_t* hint_mult;
    int depth;
    const uint64_t* hint_hi = nullptr;  // largest key of each segment, when known
};

// The on-chip sort of the segments of one size class.  Segments of a few values
// are looked for with keys alone (a payload's positions are counted anyway), but
// not among the packs of a split in the smallest class: they seldom hold a few
// values, and uniform and clustered keys took 0.4% longer for the code and the
// barrier.
template <bool PAY>
static cudaError_t chip_class(int c, const Level& L, uint64_t* dst, uint32_t* pdst, const uint32_t* list,
                              const uint32_t* nlist, uint64_t count, uint32_t lo_n, uint32_t hi_n, uint64_t fout,
                              const SegSortWs& ws, cudaStream_t st) {
    if (c == 0 && !PAY && L.depth == 0)
        return launch_chip<PAY, kC0Threads, kC0Cap, 1024, !PAY>(L.in, dst, L.pin, pdst, L.seg_lo, L.seg_hi, list, nlist,
                                                                count, L.nseg, lo_n, hi_n, L.flip_in, fout, ws.err, st);
    if (c == 0)
        return launch_chip<PAY, kC0Threads, kC0Cap, 1024, false>(L.in, dst, L.pin, pdst, L.seg_lo, L.seg_hi, list, nlist,
                                                                 count, L.nseg, lo_n, hi_n, L.flip_in, fout, ws.err, st);
    if (c == 1)
        return launch_chip<PAY, kC1Threads, kC1Cap, 4096, !PAY>(L.in, dst, L.pin, pdst, L.seg_lo, L.seg_hi, list, nlist,
                                                                count, L.nseg, lo_n, hi_n, L.flip_in, fout, ws.err, st);
    return launch_chip<PAY, kC2Threads, kSmallCap, 8192, !PAY>(L.in, dst, L.pin, pdst, L.seg_lo, L.seg_hi, list, nlist,
                                                               count, L.nseg, lo_n, hi_n, L.flip_in, fout, ws.err, st);
}

// This thread's mapped pinned buffer for the planning counts (allocated once
// per thread; null if the allocation fails, and then the counts are copied).
struct MappedCounts {
    volatile uint32_t* host = nullptr;
    uint32_t* dev = nullptr;
    bool tried = false;
};
static thread_local MappedCounts t_counts;

static void mapped_counts(volatile uint32_t** host, uint32_t** dev) {
    if (!t_counts.tried) {
        t_counts.tried = true;
        void* p = nullptr;
        if (cudaHostAlloc(&p, 64, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) {
            void* dp = nullptr;
            if (cudaHostGetDevicePointer(&dp, p, 0) == cudaSuccess) {
                t_counts.host = (volatile uint32_t*)p;
                t_counts.dev = (uint32_t*)dp;
            } else {
                (void)cudaGetLastError();
                cudaFreeHost(p);
            }
        } else {
            (void)cudaGetLastError();
        }
    }
    *host = t_counts.host;
    *dev = t_counts.dev;
}

template <bool PAY>
static cudaError_t segsort_t(const uint64_t* src, uint64_t* dst, uint64_t* tmp, const uint32_t* psrc, uint32_t* pdst,
                             uint32_t* ptmp, uint64_t N, uint64_t nseg, const uint64_t* d_seg_off, bool flip_in,
                             bool flip_out, const SegSortWs& ws, cudaStream_t st, SegSortTiming* timing,
                             const uint64_t* hint_lo, const uint64_t* hint_mult) {
    if (N == 0 || nseg == 0) return cudaSuccess;
    const uint64_t fout = flip_out ? kSignBit : 0ull;
    const uint32_t tune_chip_max = g_chip_max.load();
    const bool child_interp = g_child_interp.load() != 0u;
    const uint32_t child_keys = g_child_keys.load();
    const uint32_t pack_keys = g_pack_keys.load();
    const uint32_t first_split = g_splitters.load();
    const uint32_t scatter = g_scatter.load();
    volatile uint32_t* mapped = nullptr;  // host view of the planning counts
    uint32_t* mapped_dev = nullptr;        // the kernel's view
    if (ws.mapped_counts) mapped_counts(&mapped, &mapped_dev);
    cudaError_t e;
    Level L{src, psrc, d_seg_off, d_seg_off + 1, nseg, flip_in ? kSignBit : 0ull, hint_lo, hint_mult, 0};
    if (N <= (uint64_t)kSmallCap) {
        // No segment can exceed the on-chip capacity: sort every segment in
        // its class without planning (and without a host round trip).
        for (int c = 0; c < 3; ++c) {
            const uint32_t lo_n = c == 0 || nseg == 1 ? 0u : (c == 1 ? (uint32_t)kC0Cap : (uint32_t)kC1Cap);
            const uint32_t hi_n = c == 0 ? (uint32_t)kC0Cap : (c == 1 ? (uint32_t)kC1Cap : (uint32_t)kSmallCap);
            // one segment: the class of the largest it can be takes it whatever its size
            if (N <= lo_n || (nseg == 1 && c < 2 && N > hi_n)) continue;
            if ((e = chip_class<PAY>(c, L, dst, pdst, nullptr, nullptr, nseg, lo_n, hi_n, fout, ws, st)) != cudaSuccess)
                return e;
            if (nseg == 1) break;
        }
        return cudaSuccess;
    }
    for (;;) {
        if (L.nseg > ws.max_list) return cudaErrorInvalidValue;
        const uint32_t nblk = (uint32_t)ceil_div(L.nseg + 1, 1024);
        // By default a segment above the middle on-chip class is split again
        // (into buckets of about a thousand keys that the small classes sort)
        // rather than sorted by the largest class (tuning.chip_max_keys).
        const uint32_t chip_max = tune_chip_max;
        const PlanOut P{ws.tile_start, ws.large_id, ws.large_seg, ws.list[0], ws.list[1], ws.list[2], ws.err, ws.tile_seg};
        if (nblk <= kPlanOneChunks) {
            HSS_LAUNCH(k_plan_one, 1, 1024, 0, st, L.seg_lo, L.seg_hi, L.nseg, ws.counters, mapped_dev, P, chip_max);
        } else {
            HSS_LAUNCH(k_plan_count, nblk, 1024, 0, st, L.seg_lo, L.seg_hi, L.nseg, ws.blk, chip_max);
            HSS_LAUNCH(k_plan_scan, 1, 1024, 0, st, nblk, ws.blk, ws.counters, mapped_dev);
            HSS_LAUNCH(k_plan_write, nblk, 1024, 0, st, L.seg_lo, L.seg_hi, L.nseg, ws.blk, ws.counters, P, chip_max);
        }
        uint32_t hc[8];
        if (!mapped && (e = cudaMemcpyAsync(hc, ws.counters + 16, sizeof(hc), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
            return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        if (mapped)
            for (int k = 0; k < 8; ++k) hc[k] = mapped[k];
        const uint32_t n_large = hc[3], tiles = hc[4];
        const uint64_t keys_large = (uint64_t)hc[6] | ((uint64_t)hc[7] << 32);
        // Segments of this level that fit on chip: straight to the output.
        for (int c = 0; c < 3; ++c) {
            if (!hc[c]) continue;
            const uint32_t lo_n = c == 0 ? 0u : (c == 1 ? (uint32_t)kC0Cap : (uint32_t)kC1Cap);
            const uint32_t hi_n = c == 0 ? (uint32_t)kC0Cap : (c == 1 ? (uint32_t)kC1Cap : (uint32_t)kSmallCap);
            if ((e = chip_class<PAY>(c, L, dst, pdst, ws.list[c], ws.counters + 16 + c, hc[c], lo_n, hi_n, fout, ws, st)) !=
                cudaSuccess)
                return e;
        }
        if (n_large == 0) return cudaSuccess;
        if (n_large > ws.max_large || tiles > ws.max_tiles || L.depth >= kMaxDepth) return cudaErrorInvalidValue;
        // Statistics per tile, the split window and every tile's offsets.
        if ((e = cudaMemsetAsync(ws.vor, 0, (size_t)n_large * 8, st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(ws.vand, 0xff, (size_t)n_large * 8, st)) != cudaSuccess) return e;
        const int buf = L.depth & 1;
        const uint32_t* prev_shift = L.depth > 0 ? ws.msd_shift[buf ^ 1] : nullptr;
        // The first split of a level-0 segment may take sampled splitters
        // (skewed keys); later levels and hinted splits keep their digits.
        const bool bysplit_level = L.depth == 0 && !L.hint_lo && n_large <= ws.max_spl &&
                                   (first_split == kFirstSampled || (first_split == kFirstAuto && keys_large >= kSplMinKeys &&
                                                                      keys_large / n_large >= kSplMinSeg));
        if (bysplit_level)
            HSS_LAUNCH(k_seg_sample, n_large, 256, 0, st, L.in, L.seg_lo, L.seg_hi, ws.large_seg, ws.counters, L.flip_in,
                       chip_max, ws.spl_tab, ws.spl_mode);
        // The output holds nothing of a large segment yet: the splitter digits
        // found by the statistics pass wait there for the split (8 bytes of a
        // key have room for one), unless the keys are read from there.
        uint64_t* digits = dst + N <= L.in || L.in + N <= dst ? dst : nullptr;
        if (bysplit_level)
            HSS_LAUNCH(k_tile_stats<true>, tiles, 256, 0, st, L.in, L.seg_lo, L.seg_hi, L.nseg, ws.tile_start, ws.tile_seg,
                       ws.large_id, ws.tile_hist, ws.tile_skew, ws.vor, ws.vand, L.hint_lo, L.hint_mult, L.hint_hi,
                       prev_shift, ws.spec, L.flip_in, ws.spl_tab, ws.spl_mode, digits, PAY ? 1u : 0u);
        else
            HSS_LAUNCH(k_tile_stats<false>, tiles, 256, 0, st, L.in, L.seg_lo, L.seg_hi, L.nseg, ws.tile_start, ws.tile_seg,
                       ws.large_id, ws.tile_hist, ws.tile_skew, ws.vor, ws.vand, L.hint_lo, L.hint_mult, L.hint_hi,
                       prev_shift, ws.spec, L.flip_in, nullptr, nullptr, nullptr, 0u);
        if (!L.hint_lo)
            HSS_LAUNCH(k_tile_recount, (unsigned)std::min<uint64_t>(tiles, (uint64_t)num_sms() * 8), 256, 0, st, L.in, L.seg_lo,
                       L.seg_hi, tiles, ws.tile_start, ws.tile_seg, ws.large_id, ws.tile_hist, ws.tile_skew,
                       bysplit_level ? ws.spl_mode : nullptr, ws.vor, ws.vand, ws.spec, L.flip_in);
        HSS_LAUNCH(k_msd_prep, n_large, 256, 0, st, L.seg_lo, ws.large_seg, ws.counters, ws.tile_start, ws.tile_hist,
                   ws.vor, ws.vand, L.hint_lo, L.hint_mult, ws.msd_base, ws.msd_mult, ws.msd_shift[buf], ws.spec,
                   ws.direct, ws.sub_lo[buf], ws.sub_hi[buf], ws.tile_off, child_interp ? chip_max : 0xffffffffu,
                   ws.large_mask, ws.any_large, ws.cmin[buf], ws.cmax[buf], chip_max,
                   std::min(pack_limit(pack_keys, keys_large), chip_max),
                   bysplit_level ? ws.spl_mode : nullptr);
        // The split pass: level buffers alternate tmp, dst, tmp, ... after src.
        uint64_t* next = (L.depth & 1) ? dst : tmp;
        uint32_t* pnext = PAY ? ((L.depth & 1) ? pdst : ptmp) : nullptr;
        SplitArgs A;
        A.kin = L.in; A.kout = next; A.kfinal = dst;
        A.pin = L.pin; A.pout = pnext; A.pfinal = pdst;
        A.seg_lo = L.seg_lo; A.seg_hi = L.seg_hi; A.nseg = L.nseg;
        A.tile_start = ws.tile_start; A.tile_seg = ws.tile_seg; A.large_id = ws.large_id;
        A.tile_off = ws.tile_off; A.tile_skew = ws.tile_skew; A.digits = digits; A.spl_tab = ws.spl_tab; A.msd_shift = ws.msd_shift[buf]; A.msd_base = ws.msd_base; A.msd_mult = ws.msd_mult;
        A.direct = ws.direct;
        A.large_mask = ws.large_mask; A.any_large = ws.any_large; A.cmin = ws.cmin[buf]; A.cmax = ws.cmax[buf];
        A.err = ws.err;
        A.scatter = scatter;
        A.flip_in = L.flip_in; A.flip_out = fout;
        const size_t smem = bysplit_level ? split_smem<PAY, true>(child_interp) : split_smem<PAY, false>(child_interp);
        const size_t smem_max = bysplit_level ? split_smem<PAY, true>(true) : split_smem<PAY, false>(true);
        // all of L1 as shared memory: the CTAs per SM are limited by their tiles
        const void* split_fn = bysplit_level ? (const void*)k_split<PAY, true> : (const void*)k_split<PAY, false>;
        if ((e = ensure_func_attrs(split_fn, (int)smem_max, 100)) != cudaSuccess) return e;
        const bool timed = timing && timing->enabled && timing->n < 16;
        if (timed) {
            cudaEventCreate(&timing->ev[timing->n][0]);
            cudaEventCreate(&timing->ev[timing->n][1]);
            cudaEventRecord(timing->ev[timing->n][0], st);
        }
        if (bysplit_level)
            HSS_LAUNCH((k_split<PAY, true>), tiles, split_threads<PAY>(), smem, st, A);
        else
            HSS_LAUNCH((k_split<PAY, false>), tiles, split_threads<PAY>(), smem, st, A);
        if (timed) {
            cudaEventRecord(timing->ev[timing->n][1], st);
            timing->keys[timing->n] = keys_large;
            timing->n += 1;
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // Next level: the 256 sub-buckets of every large segment; those split
        // again interpolate their own key range (gathered by the split).
        const uint32_t nch = n_large * kRadix;
        if (child_interp) {
            HSS_LAUNCH(k_child_hints, (nch + 255) / 256, 256, 0, st, nch, ws.sub_lo[buf], ws.sub_hi[buf], ws.cmin[buf],
                       ws.cmax[buf], ws.cmult[buf], chip_max, child_keys, (uint32_t)L.depth + 1u);
            L = Level{next, pnext, ws.sub_lo[buf], ws.sub_hi[buf], (uint64_t)n_large * kRadix, 0ull, ws.cmin[buf],
                      ws.cmult[buf], L.depth + 1, ws.cmax[buf]};
        } else {
            L = Level{next, pnext, ws.sub_lo[buf], ws.sub_hi[buf], (uint64_t)n_large * kRadix, 0ull, nullptr, nullptr,
                      L.depth + 1};
        }
    }
}

cudaError_t segsort(const uint64_t* src, uint64_t* dst, uint64_t* tmp, const uint32_t* psrc, uint32_t* pdst,
                    uint32_t* ptmp, uint64_t N, uint64_t nseg, const uint64_t* d_seg_off, bool flip_in, bool flip_out,
                    const SegSortWs& ws, cudaStream_t st, SegSortTiming* timing, const uint64_t* hint_lo,
                    const uint64_t* hint_mult) {
    if (psrc)
        return segsort_t<true>(src, dst, tmp, psrc, pdst, ptmp, N, nseg, d_seg_off, flip_in, flip_out, ws, st, timing,
                               hint_lo, hint_mult);
    return segsort_t<false>(src, dst, tmp, nullptr, nullptr, nullptr, N, nseg, d_seg_off, flip_in, flip_out, ws, st,
                            timing, hint_lo, hint_mult);
}

}  // namespace hss
