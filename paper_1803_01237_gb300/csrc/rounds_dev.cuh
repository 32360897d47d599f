// rounds_dev.cuh -- device helpers of the splitter rounds shared by the
// single-job kernels (rounds.cu) and the batched ones (batch.cu).
#pragma once

#include "hss_internal.cuh"

namespace hss {

// ---------------------------------------------------------------------------
// Block scans (blockDim a multiple of 32, at most 1024).
// ---------------------------------------------------------------------------
template <typename T, typename Op>
__device__ __forceinline__ T warp_incl_scan(T x, Op op) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = op(x, y);
    }
    return x;
}

// Inclusive block scan with identity `id`; returns the inclusive value and
// sets `total`.  Uses s_warp[32] of T.
template <typename T, typename Op>
__device__ __forceinline__ T block_incl_scan(T v, T id, Op op, T* s_warp, T& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T x = warp_incl_scan(v, op);
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    if (w == 0) {
        T y = lane < nw ? s_warp[lane] : id;
        y = warp_incl_scan(y, op);
        s_warp[lane] = y;
    }
    __syncthreads();
    T r = w > 0 ? op(s_warp[w - 1], x) : x;
    total = s_warp[nw - 1];
    __syncthreads();
    return r;
}

struct AddU32 { __device__ uint32_t operator()(uint32_t a, uint32_t b) const { return a + b; } };
struct AddU64 { __device__ uint64_t operator()(uint64_t a, uint64_t b) const { return a + b; } };
struct MaxI32 { __device__ int32_t operator()(int32_t a, int32_t b) const { return a > b ? a : b; } };

__device__ __forceinline__ uint64_t ideal_rank(uint64_t i1, uint64_t N, uint64_t p) {
    // t_i for splitter number i1 (1-based); a 128-bit division is a call of
    // several hundred instructions, needed from i1 N = 2^64 on
    if (__umul64hi(i1, N) == 0) return i1 * N / p;
    return (uint64_t)(((unsigned __int128)i1 * N) / p);
}

// Count of keys in a[0..n) below key: strict (<) or not (<=), branch-free.
__device__ __forceinline__ uint32_t count_below(const uint64_t* __restrict__ a, uint32_t n, uint64_t key, bool strict) {
    uint32_t base = 0;
    while (n > 0) {
        const uint32_t half = n >> 1;
        const uint64_t v = a[base + half];
        const bool go = strict ? (v < key) : (v <= key);
        base = go ? base + half + 1 : base;
        n = go ? n - half - 1 : half;
    }
    return base;
}

// Improve L/U of one splitter with a ranked cut c (Sec. 4.2.2 step 3): L is
// the cut of largest rank <= t, U the cut of smallest rank >= t, equal ranks
// keeping the smaller cut; cl/cu record the probe index that changed them.
__device__ __forceinline__ void offer(DCut& L, DCut& U, int32_t& cl, int32_t& cu, uint64_t t, const DCut& c, int32_t k) {
    if (c.rank <= t && (c.rank > L.rank || (c.rank == L.rank && cut_less(c, L)))) { L = c; cl = k; }
    if (c.rank >= t && (c.rank < U.rank || (c.rank == U.rank && cut_less(c, U)))) { U = c; cu = k; }
}

struct IntervalsOut {
    uint64_t gamma, T;
    uint32_t nint, unresolved, take_all;
};

// Resolved flags, distinct unresolved intervals (their representative
// splitters into int_rep), |gamma| and the next threshold of one job, by one
// CTA of up to 1024 threads walking the splitters in chunks.  The outputs are
// valid in thread 0.
// With int_T non-null, every distinct interval u also gets the threshold of
// the equal-per-interval schedule: probability (s p / nint) / its length.
// With int_seg non-null, also the segment of its lower cut (~0: not a member).
__device__ __forceinline__ void intervals_body(uint32_t S, uint64_t N, uint32_t p, uint64_t tol, float oversample,
                                               const DCut* Lcut, const DCut* Ucut, uint32_t* __restrict__ res,
                                               uint32_t* int_rep, IntervalsOut& out, uint64_t* __restrict__ int_T = nullptr,
                                               uint32_t* __restrict__ int_all = nullptr,
                                               uint32_t* __restrict__ int_seg = nullptr) {
    __shared__ uint32_t s_u32[32];
    __shared__ int32_t s_i32[32];
    __shared__ uint64_t s_u64[32];
    uint32_t carry_heads = 0, carry_f = 0, carry_unres = 0;
    int32_t carry_max = -1;
    uint64_t gamma = 0;
    for (uint32_t base = 0; base < S; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        const bool valid = i < S;
        uint32_t head = 0, unres = 0, member = ~0u;
        uint64_t glen = 0;
        if (valid) {
            const DCut L = Lcut[i], U = Ucut[i];
            const uint64_t t = ideal_rank(i + 1, N, p);
            const bool r = (t - L.rank) <= tol || (U.rank - t) <= tol;
            res[i] = r ? 1u : 0u;
            unres = r ? 0u : 1u;
            head = (i == 0) || !(cut_equal(L, Lcut[i - 1]) && cut_equal(U, Ucut[i - 1]));
            glen = U.rank - L.rank - (L.kind == kMember ? 1u : 0u);
            if (L.kind == kMember) member = (uint32_t)L.seg;
        }
        uint32_t tot;
        const uint32_t heads_incl = block_incl_scan<uint32_t>(head, 0u, AddU32(), s_u32, tot) + carry_heads;
        carry_heads += tot;
        const int32_t rid = (int32_t)heads_incl - 1;
        int32_t mtot;
        const int32_t mv = unres ? rid : -1;
        int32_t mincl = block_incl_scan<int32_t>(mv, -1, MaxI32(), s_i32, mtot);
        mincl = mincl > carry_max ? mincl : carry_max;
        int32_t mexcl = __shfl_up_sync(0xffffffffu, mincl, 1);
        // lane 0 needs the previous warp's last value
        __shared__ int32_t s_last[32];
        if ((threadIdx.x & 31) == 31) s_last[threadIdx.x >> 5] = mincl;
        __syncthreads();
        if ((threadIdx.x & 31) == 0) mexcl = (threadIdx.x == 0) ? carry_max : s_last[(threadIdx.x >> 5) - 1];
        __syncthreads();
        carry_max = carry_max > mtot ? carry_max : mtot;
        const uint32_t f = (valid && unres && mexcl != rid) ? 1u : 0u;
        uint32_t ftot;
        const uint32_t fincl = block_incl_scan<uint32_t>(f, 0u, AddU32(), s_u32, ftot);
        if (f) {
            int_rep[carry_f + fincl - 1] = i;
            if (int_seg) int_seg[carry_f + fincl - 1] = member;
        }
        carry_f += ftot;
        uint32_t utot;
        block_incl_scan<uint32_t>(unres, 0u, AddU32(), s_u32, utot);
        carry_unres += utot;
        uint64_t gtot;
        block_incl_scan<uint64_t>(f ? glen : 0ull, 0ull, AddU64(), s_u64, gtot);
        gamma += gtot;
    }
    if (int_T) {
        __syncthreads();  // int_rep is complete
        const double per_int = carry_f ? ((double)oversample * (double)p) / (double)carry_f : 0.0;
        for (uint32_t u = threadIdx.x; u < carry_f; u += blockDim.x) {
            const uint32_t rep = int_rep[u];
            const DCut L = Lcut[rep], U = Ucut[rep];
            const uint64_t len = U.rank - L.rank - (L.kind == kMember ? 1u : 0u);
            const double q = len ? per_int / (double)len : 1.0;
            if (q >= 1.0) { int_all[u] = 1u; int_T[u] = 0ull; }
            else { int_all[u] = 0u; int_T[u] = (uint64_t)floor(ldexp(q, 64)); }
        }
    }
    if (threadIdx.x == 0) {
        out.gamma = gamma;
        out.nint = carry_f;
        out.unresolved = carry_unres;
        double q = gamma == 0 ? 1.0 : ((double)oversample * (double)p) / (double)gamma;
        if (q >= 1.0) {
            out.take_all = 1u;
            out.T = 0ull;
        } else {
            out.take_all = 0u;
            out.T = (uint64_t)floor(ldexp(q, 64));
        }
    }
}

// ---------------------------------------------------------------------------
// Sampling helpers.
// ---------------------------------------------------------------------------
constexpr int kIntChunk = 2048;
constexpr int kSampThreads = 256;

// Fill the interval ranges of segment s for intervals [u0, u0+nu) and the
// exclusive prefix of their position-pair counts (s_pre, 16-byte aligned).
// Returns the pair total.  Neighbouring threads read neighbouring intervals,
// and (int_seg) the segments of the lower cuts from an array of their own: with
// eight intervals in a row per thread and the cuts' records, 4095 intervals in
// 4096 segments cost a round 30 to 50 us more.
__device__ __forceinline__ uint32_t load_seg_intervals(uint32_t s, uint32_t n_s, uint32_t S, uint32_t u0, uint32_t nu,
                                       const uint32_t* Lpos, const uint32_t* Upos,
                                       const DCut* __restrict__ Lcut, const uint32_t* __restrict__ int_rep,
                                       const uint32_t* __restrict__ int_seg,
                                       uint32_t* s_a, uint32_t* s_b, uint32_t* s_pre, uint32_t* s_warp) {
    constexpr int kPer = kIntChunk / kSampThreads;
    static_assert(kPer == 8, "two vectors of counts per thread");
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if ((uint32_t)(k * kSampThreads) >= nu) break;
        const uint32_t u = threadIdx.x + k * kSampThreads;
        uint32_t np = 0;
        if (u < nu) {
            const uint32_t rep = int_rep[u0 + u];
            uint32_t member;
            if (int_seg) member = int_seg[u0 + u];
            else member = Lcut[rep].kind == kMember ? (uint32_t)Lcut[rep].seg : ~0u;
            uint32_t a = Lpos[(uint64_t)s * S + rep];
            if (member == s) a += 1;
            uint32_t b = Upos[(uint64_t)s * S + rep];
            if (b > n_s) b = n_s;  // defensive: a range never leaves its segment
            s_a[u] = a;
            s_b[u] = b;
            np = b > a ? ((b - 1) >> 1) - (a >> 1) + 1 : 0u;
        }
        s_pre[u] = np;
    }
    __syncthreads();
    uint32_t c[kPer] = {};
    uint4* own = (uint4*)s_pre + 2 * threadIdx.x;
    const bool mine = threadIdx.x * kPer < nu;
    if (mine) {
        const uint4 x = own[0], y = own[1];
        c[0] = x.x; c[1] = x.y; c[2] = x.z; c[3] = x.w; c[4] = y.x; c[5] = y.y; c[6] = y.z; c[7] = y.w;
    }
    uint32_t sum = 0, tot;
#pragma unroll
    for (int k = 0; k < kPer; ++k) sum += c[k];
    uint32_t run = block_incl_scan<uint32_t>(sum, 0u, AddU32(), s_warp, tot) - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const uint32_t x = c[k];
        c[k] = run;
        run += x;
    }
    if (mine) {
        own[0] = make_uint4(c[0], c[1], c[2], c[3]);
        own[1] = make_uint4(c[4], c[5], c[6], c[7]);
    }
    if (threadIdx.x == 0) s_pre[nu] = tot;  // what a thread whose row holds this place writes there too
    __syncthreads();
    return tot;
}

__device__ __forceinline__ uint32_t find_interval(const uint32_t* s_pre, uint32_t nu, uint32_t f) {
    uint32_t lo = 0, hi = nu;  // last u with s_pre[u] <= f
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s_pre[mid] <= f) lo = mid; else hi = mid;
    }
    return lo;
}

// Philox4x32-10 of the counters (m, seg, round, 0) for one (seed, seg,
// round): the round keys and the parts of the first two rounds that do not
// depend on m are computed once, so a word pair costs 18 of the 20
// multiplies and none of the key additions.  Same words as sample_words.
struct PairDraw {
    uint32_t k0[10], k1[10];  // round keys
    uint32_t c0_1, c1_1;      // words 0 and 1 after round 1 (independent of m)
    uint32_t lo0_2, hi0_2;    // M0 x (word 0 after round 1), used in round 2
    __device__ __forceinline__ void init(uint64_t seed, uint32_t seg, uint32_t round) {
        const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u, M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
        uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
#pragma unroll
        for (int r = 0; r < 10; ++r) { k0[r] = a; k1[r] = b; a += W0; b += W1; }
        // round 1 on (m, seg, round, 0): the M1 product and the new word 0
        // involve only seg and round
        const uint32_t lo1 = M1 * round, hi1 = __umulhi(M1, round);
        c0_1 = hi1 ^ seg ^ k0[0];
        c1_1 = lo1;
        lo0_2 = M0 * c0_1;
        hi0_2 = __umulhi(M0, c0_1);
    }
    // The upper halves of the two words alone: they are the low products of
    // the last round, so that round needs no high product and no xor.
    __device__ __forceinline__ void tops(uint32_t m, uint32_t& even, uint32_t& odd) const {
        const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
        uint32_t c0, c1, c2, c3;
        rounds_1_to_9(m, c0, c1, c2, c3);
        even = M1 * c2;
        odd = M0 * c0;
    }
    __device__ __forceinline__ void words(uint32_t m, uint64_t& even, uint64_t& odd) const {
        const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
        uint32_t c0, c1, c2, c3;
        rounds_1_to_9(m, c0, c1, c2, c3);
        const uint32_t l0 = M0 * c0, h0 = __umulhi(M0, c0);
        const uint32_t l1 = M1 * c2, h1 = __umulhi(M1, c2);
        even = ((uint64_t)l1 << 32) | (h1 ^ c1 ^ k0[9]);
        odd = ((uint64_t)l0 << 32) | (h0 ^ c3 ^ k1[9]);
    }

private:
    __device__ __forceinline__ void rounds_1_to_9(uint32_t m, uint32_t& c0, uint32_t& c1, uint32_t& c2,
                                                  uint32_t& c3) const {
        const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
        // round 1: only the M0 x m product varies
        const uint32_t lo0 = M0 * m, hi0 = __umulhi(M0, m);
        c2 = hi0 ^ k1[0];  // ^ word 3 (0)
        c3 = lo0;
        c0 = c0_1;
        c1 = c1_1;
        // round 2: the M0 product is known
        {
            const uint32_t l1 = M1 * c2, h1 = __umulhi(M1, c2);
            const uint32_t n0 = h1 ^ c1 ^ k0[1];
            const uint32_t n2 = hi0_2 ^ c3 ^ k1[1];
            c0 = n0; c1 = l1; c2 = n2; c3 = lo0_2;
        }
#pragma unroll
        for (int r = 2; r < 9; ++r) {
            const uint32_t l0 = M0 * c0, h0 = __umulhi(M0, c0);
            const uint32_t l1 = M1 * c2, h1 = __umulhi(M1, c2);
            const uint32_t n0 = h1 ^ c1 ^ k0[r];
            const uint32_t n2 = h0 ^ c3 ^ k1[r];
            c0 = n0; c1 = l1; c2 = n2; c3 = l0;
        }
    }
};

// Keep the keys at positions 2m and 2m + 1 that lie in [a, b) and whose word is
// below the threshold.  e, o: the upper halves of the two words (PairDraw::tops);
// the whole words are drawn only where one of those does not exceed the
// threshold's, once in 1/q keys.
__device__ __forceinline__ void mark_pair(const PairDraw& pd, uint32_t a, uint32_t b, uint32_t m, uint32_t e, uint32_t o,
                                          uint64_t Tu, bool all_u, uint64_t base, uint32_t* __restrict__ bitmap,
                                          uint32_t& cnt) {
    const uint32_t top = (uint32_t)(Tu >> 32);
    if (!all_u && e > top && o > top) return;
    uint64_t w0, w1;
    pd.words(m, w0, w1);
    const uint32_t p0 = 2 * m, p1 = 2 * m + 1;
    if (p0 >= a && p0 < b && (all_u || w0 < Tu)) {
        const uint64_t g = base + p0;
        atomicOr(&bitmap[g >> 5], 1u << (g & 31));
        ++cnt;
    }
    if (p1 >= a && p1 < b && (all_u || w1 < Tu)) {
        const uint64_t g = base + p1;
        atomicOr(&bitmap[g >> 5], 1u << (g & 31));
        ++cnt;
    }
}

// The draws of pairs [f0, f1) of nu intervals by the CTA (kSampThreads): each
// thread walks a contiguous run of pairs two at a time (two independent Philox
// chains in flight), thr(u, T, all) giving the threshold of interval u.  One
// interval (round 1) needs no walk.
template <class Thr>
__device__ __forceinline__ void mark_pairs(const PairDraw& pd, const uint32_t* s_a, const uint32_t* s_b,
                                           const uint32_t* s_pre, uint32_t nu, uint32_t F0, uint32_t F1, Thr thr,
                                           uint64_t base, uint32_t* __restrict__ bitmap, uint32_t& cnt) {
    if (nu == 1) {
        const uint32_t a = s_a[0], b = s_b[0], m0 = a >> 1;
        uint64_t T;
        bool all;
        thr(0u, T, all);
        uint32_t f = F0 + threadIdx.x;
        for (; f + kSampThreads < F1; f += 2 * kSampThreads) {
            uint32_t e0, o0, e1, o1;
            pd.tops(m0 + f, e0, o0);
            pd.tops(m0 + f + kSampThreads, e1, o1);
            mark_pair(pd, a, b, m0 + f, e0, o0, T, all, base, bitmap, cnt);
            mark_pair(pd, a, b, m0 + f + kSampThreads, e1, o1, T, all, base, bitmap, cnt);
        }
        if (f < F1) {
            uint32_t e0, o0;
            pd.tops(m0 + f, e0, o0);
            mark_pair(pd, a, b, m0 + f, e0, o0, T, all, base, bitmap, cnt);
        }
        return;
    }
    const uint32_t per = (F1 - F0 + kSampThreads - 1) / kSampThreads;
    const uint32_t f0 = min(F1, F0 + threadIdx.x * per), f1 = min(F1, f0 + per);
    if (f0 >= f1) return;
    uint32_t u = find_interval(s_pre, nu, f0);
    uint32_t f = f0;
    for (; f + 1 < f1; f += 2) {
        while (u + 1 < nu && s_pre[u + 1] <= f) ++u;
        uint32_t v = u;
        while (v + 1 < nu && s_pre[v + 1] <= f + 1) ++v;
        const uint32_t m0 = (s_a[u] >> 1) + (f - s_pre[u]);
        const uint32_t m1 = (s_a[v] >> 1) + (f + 1 - s_pre[v]);
        uint32_t e0, o0, e1, o1;
        pd.tops(m0, e0, o0);
        pd.tops(m1, e1, o1);
        uint64_t Tu, Tv;
        bool au, av;
        thr(u, Tu, au);
        thr(v, Tv, av);
        mark_pair(pd, s_a[u], s_b[u], m0, e0, o0, Tu, au, base, bitmap, cnt);
        mark_pair(pd, s_a[v], s_b[v], m1, e1, o1, Tv, av, base, bitmap, cnt);
        u = v;
    }
    if (f < f1) {
        while (u + 1 < nu && s_pre[u + 1] <= f) ++u;
        const uint32_t m0 = (s_a[u] >> 1) + (f - s_pre[u]);
        uint32_t e0, o0;
        uint64_t Tu;
        bool au;
        pd.tops(m0, e0, o0);
        thr(u, Tu, au);
        mark_pair(pd, s_a[u], s_b[u], m0, e0, o0, Tu, au, base, bitmap, cnt);
    }
}

// Segments short enough for a warp each: a CTA per segment of 2^14 keys spent
// its time in the chain of loads and barriers before the first mark (16384
// segments: 101 us a round, by warps 26).
constexpr uint64_t kSampWarpKeys = 1ull << 15;  // keys per segment on average, at most

// The marked positions g in [base, end) of the bitmap, in order, by the CTA
// (kSampThreads) or by one warp: body(g, number of marks before it).  want: how many there
// are.  The marks are cleared on the way, for the next round (a word on the
// border keeps the neighbour's bits).  Marks are rare, so the pass is bound by
// its steps over empty words: a thread reads four words a step (2^28 positions
// in 4096 segments: 35 us a round by single words, 22 by four).
template <bool WARP, class Body>
__device__ __forceinline__ void take_marks(uint32_t* bitmap, uint64_t base, uint64_t end, uint32_t want, uint32_t* s_warp,
                                           Body body) {
    const uint64_t v0 = base >> 7, v1 = (end + 127) >> 7;  // vectors of 128 positions
    const uint32_t lane = threadIdx.x & 31;
    uint32_t found = 0;
    for (uint64_t vb = v0; vb < v1 && found < want; vb += WARP ? 32 : kSampThreads) {
        const uint64_t vi = vb + (WARP ? lane : threadIdx.x);
        uint32_t bits[4] = {0u, 0u, 0u, 0u};
        if (vi < v1) {
            uint4 x;
            if (((uintptr_t)bitmap & 15u) == 0) x = ((const uint4*)bitmap)[vi];
            else x = make_uint4(bitmap[4 * vi], bitmap[4 * vi + 1], bitmap[4 * vi + 2], bitmap[4 * vi + 3]);  // a workspace off 16 bytes
            bits[0] = x.x; bits[1] = x.y; bits[2] = x.z; bits[3] = x.w;
            if (x.x | x.y | x.z | x.w) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint64_t g0 = (vi << 7) + 32 * k;
                    if (g0 + 32 <= base || g0 >= end) { bits[k] = 0u; continue; }
                    const bool whole = g0 >= base && g0 + 32 <= end;
                    if (g0 < base) bits[k] &= ~0u << (uint32_t)(base - g0);                               // the previous segment's
                    if (g0 + 32 > end) bits[k] &= (uint32_t)((1ull << (uint32_t)(end - g0)) - 1ull);      // the next one's
                    if (bits[k]) {
                        if (whole) bitmap[4 * vi + k] = 0u;
                        else atomicAnd(&bitmap[4 * vi + k], ~bits[k]);
                    }
                }
            }
        }
        const uint32_t c = __popc(bits[0]) + __popc(bits[1]) + __popc(bits[2]) + __popc(bits[3]);
        if ((WARP ? __any_sync(0xffffffffu, c != 0u) : __syncthreads_or(c)) == 0) continue;
        uint32_t tot, at;
        if (WARP) {
            uint32_t x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= (uint32_t)o) x += y;
            }
            tot = __shfl_sync(0xffffffffu, x, 31);
            at = found + x - c;
        } else {
            at = found + block_incl_scan<uint32_t>(c, 0u, AddU32(), s_warp, tot) - c;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            while (bits[k]) {
                const uint32_t b = __ffs(bits[k]) - 1;
                bits[k] &= bits[k] - 1;
                body((vi << 7) + 32 * k + b, at++);
            }
        found += tot;
    }
}

// Positions in segment s of the cuts that the last histogram moved.
__device__ __forceinline__ void update_pos_row(uint64_t s, uint32_t S, const int32_t* __restrict__ chgL,
                                               const int32_t* __restrict__ chgU, const uint32_t* __restrict__ probe_pos,
                                               uint64_t cap, uint32_t* Lpos, uint32_t* Upos) {
    for (uint32_t i = threadIdx.x; i < S; i += blockDim.x) {
        const int32_t cl = chgL[i], cu = chgU[i];
        if (cl >= 0) Lpos[s * S + i] = probe_pos[s * cap + (uint32_t)cl];
        if (cu >= 0) Upos[s * S + i] = probe_pos[s * cap + (uint32_t)cu];
    }
}

}  // namespace hss
