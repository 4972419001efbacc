// Per-vertex butterfly counting, Algorithm 1 (pvBcnt).
//
// For every start point sp (both sides), every middle point mp in N_sp and
// every end point ep in N_mp with label(ep) < label(mp) and label(ep) <
// label(sp), wdg[ep] counts the wedges sp-mp-ep. Then C(wdg[ep], 2) goes to
// ep and to sp, and wdg[ep] - 1 goes to mp once per wedge (Algorithm 1,
// "same side" and "opposite side" contributions).
//
// Because neighbour lists are sorted by label, the admissible end points of
// (sp, mp) are a PREFIX of N_mp: those with local id < min(sp, below[mp]).
// Prefixes hold the end points of highest degree, so most wedges end in a few
// of them: on skewed Chung-Lu graphs 94% below id 1,024, on a 10M-edge graph
// of exponents 2.5 / 2.1 84%. Both contributions are sums over end points, so
// the count splits by end point:
//
//  * The first BITS end points (k_count_bits; where masks_pay): every vertex's list has a mask
//    of its first 1,024 possible entries, one word per lane of a warp. A start
//    point adds up its middle points' masks, cut at the prefix, in bit-sliced
//    counters (plane p holds bit p of 32 counts per lane): ~12 instructions
//    add 1,024 end points of one middle point, and a population count of mask
//    and planes gives the middle point's sum of (count - 1).
//  * The others, end point by end point: a plan finds every prefix's length
//    past the masks by binary search, sums each start point's wedges there
//    and lists it in a tier (warp or CTA, by its wedges); the start points of
//    both sides share every launch.
//
// Measured (both sides, ms; before: prefixes of all end points by one warp or
// one 1,024-thread CTA per start point): 20M edges, 4.4e9 wedges, 77.1 -> 17.4
// (bit-sliced 7.6, the rest 8.1, plan 1.0); 10M edges 14.3 -> 6.3; 1M edges
// 1.45 -> 0.8. What bounds it now: instruction issue in the bit-sliced kernels
// (~40 instructions per edge and pass; SMs 68% busy), the chain of dependent loads
// per start point, barriers and instruction fetch in the others.
#include "engine.cuh"
#include "internal.cuh"

#include <algorithm>
#include <mutex>
#include <string>
#include <type_traits>

namespace receipt {

namespace {

// Tiers of start points. W: wedges; T: wedges whose key is past the head.
enum {
    CT_WARP = 0,   // W <= 256: one warp, hash table
    CT_DENSE64,    // W <= 4,096, T <= 256: 64 threads, head + tail table
    CT_DENSE256,   // W <= 65,536, T <= 1,024: 256 threads
    CT_DENSE512,   // W < 2^32, T <= 2,048: 512 threads
    CT_HASH,       // otherwise, W <= 2,048: 256 threads, hash table
    CT_HYBRID,     // otherwise, degree below 65,535 and keys that fit: hybrid engine
    CT_GLOBAL,     // otherwise: global counters
    CT_OVER,       // hybrid start points whose repeat table overflowed: global counters
    CT_WIDE,       // start points of high degree, split by k_count_plan_wide
    CT_BITS,       // bit-sliced part: start points of high degree, a CTA each
    CT_HUGE,       // ... of very high degree, several CTAs each
    CT_LISTS
};
constexpr int COUNT_HEAD = 4096;  // keys with dense 16-bit counters
constexpr int PLAN_DEG = 256;     // larger neighbourhoods are planned by a CTA
constexpr int BITS = 1024;        // end points of the bit-sliced part
// Start points of at least BITS_DEG take a CTA there, of at least HUGE_DEG one per
// HUGE_DEG middle points. Counts with 256 / this / 1,024, ms: 300k edges 0.34 / 0.43
// / 0.60, 1M 0.71 / 0.79 / 0.97, 10M 6.34 / 6.38 / 6.68, 20M 17.40 / 17.12 / 17.11; with
// 2,048 / 4,096 / this: 300k 0.50 / 0.43 / 0.43, 3M 1.93 / 2.03 / 2.26, 10M 6.24 / 6.22
// / 6.38, 20M 17.16 / 17.00 / 17.12: flat near these.
constexpr int BITS_DEG = 512;
constexpr int HUGE_DEG = 8192;

// Start points with at most HASH_W wedges (and more than WARP_MAX_W) and too
// many keys past the head: small CTAs, any key space, any degree.
constexpr int HASH_SLOTS = 4096;
constexpr int HASH_W = HASH_SLOTS / 2;
constexpr int HASH_THREADS = 256;
using CountHash = CtaHashT<HASH_SLOTS>;

// A tier walks as many middle points a step as it has threads, ~0.9 us a step and
// walk however few their wedges are. Hubs with few wedges (the first start points:
// hardly an end point comes before them) of more steps than this take the next
// larger CTA, up to the hybrid's 1,024 threads. Counts of 2M edges on 2.6M vertices
// (degrees up to 69,633) / 1.5M on 2.7M (29,521) / 450k on 98,000 (23,327), ms: any
// degree 2.28 / 1.92 / 0.92, 64 steps 1.72 / 1.06 / 0.68, 16 1.20 / 0.81 / 0.63, 8
// 1.13 / 0.74 / 0.55.
constexpr int TIER_STEPS = 8;

// One side as start side A (B: the other side).
struct CountSide {
    const int64_t *offA;
    const int32_t *adjA;
    const int64_t *offB;
    const int32_t *adjB;
    const int32_t *belowB;
    unsigned long long *cntA, *cntB;
    unsigned long long *hotA, *hotB;  // HOT_REPS x HOT_KEYS (null: none)
    int32_t *plen;         // prefix length of every A-side CSR position
    int32_t *base;         // first key of every start point's packed graph (null: 0)
    const int32_t *first;  // first vertex of every packed graph (null: one graph)
    // masks of the B side's lists over the first BITS keys (null: none) and
    // how many of a list's entries they hold
    const uint32_t *mask;
    const int32_t *held;
    int32_t nA, ng;
};

// The counts of the vertices of highest degree are added to by nearly every
// start point: HOT_REPS copies of the first HOT_KEYS counts per side, a CTA
// adding to its own copy, merged at the end. (With one copy the warp tier of
// the 10M-edge graph took 4.6 ms whatever its walk: all its atomics went to a
// few cache lines.)
constexpr int HOT_KEYS = 4096, HOT_REPS = 32;
// edges from which the copies pay (with them / without, ms: 20k edges 0.100 / 0.090,
// 130k 0.372 / 0.367, 1M 0.79 / 0.89)
constexpr int64_t HOT_MIN_M = 1 << 17;

struct CountPlan {
    CountSide s[2];
    int32_t *list[CT_LISTS];  // start points, side << 31 | id
    int32_t *n;               // entries per list, then work counters per tier
    unsigned long long *wedges;
    int64_t cta_keys;         // key space of the hybrid tier (0: none)
    int32_t *hoff;            // huge start points: first chunk of each
    uint32_t *hplanes;        // planes of every chunk, then of every start point
    int32_t few;              // few launches instead of a tier for every size
};
constexpr int COUNT_CTRS = 2 * CT_LISTS;

__device__ __forceinline__ int32_t tier_of(const CountPlan &p, int64_t W, int64_t T, int64_t deg,
                                           int32_t sp) {
    if (W <= WARP_MAX_W && deg <= 32 * TIER_STEPS) return CT_WARP;
    if (deg < 65535) {
        if (!p.few && W <= 4096 && T <= 256 && deg <= 64 * TIER_STEPS) return CT_DENSE64;
        if (W <= 65536 && T <= 1024 && deg <= 256 * TIER_STEPS) return CT_DENSE256;
    }
    if (!p.few && W <= HASH_W && (deg <= HASH_THREADS * TIER_STEPS || deg >= 65535)) return CT_HASH;
    if (deg < 65535) {
        if (!p.few && T <= 2048 && W < (1ll << 32) && (deg <= 512 * TIER_STEPS || sp > p.cta_keys))
            return CT_DENSE512;
        if (sp <= p.cta_keys) return CT_HYBRID;
    }
    return CT_GLOBAL;
}

// Length of the prefix of edge q = (sp, mp) past the masks, and how much of it
// lies past the head. first: the first key past the masks.
__device__ __forceinline__ int32_t plan_edge(const CountSide &S, int32_t sp, int32_t first, int64_t q,
                                             int32_t &tail) {
    const int32_t mp = S.adjA[q];
    const int32_t lim = min(sp, S.belowB[mp]);
    int32_t P = 0;
    tail = 0;
    if (lim > first) {
        const int64_t b = S.offB[mp] + (S.held ? S.held[mp] : 0), e = S.offB[mp + 1];
        P = (int32_t)lower_bound_i32(S.adjB + b, e - b, lim);
        if (lim > first + COUNT_HEAD && P > 0)
            tail = P - (int32_t)lower_bound_i32(S.adjB + b, P, first + COUNT_HEAD);
    }
    S.plen[q] = P;
    return P;
}

__device__ __forceinline__ int32_t plan_base(const CountSide &S, int32_t sp) {
    if (!S.first) return 0;
    int lo = 0, hi = S.ng - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (S.first[mid] <= sp)
            lo = mid;
        else
            hi = mid - 1;
    }
    return S.first[lo];
}

// Prefix lengths, wedge counts and tiers of both sides' start points, L lanes
// per start point; those of high degree go to k_count_plan_wide.
template <int L>
__global__ void __launch_bounds__(256) k_count_plan(CountPlan p) {
    const int lane = threadIdx.x & 31, l8 = lane & (L - 1);
    const int64_t n0 = p.s[0].nA, n = n0 + p.s[1].nA;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long wsum = 0;
    for (int64_t b = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 / L); b < n;
         b += nw * (32 / L)) {
        const int64_t i = b + lane / L;
        const int side = i >= n0 ? 1 : 0;
        const CountSide &S = p.s[side];
        const int32_t sp = (int32_t)(side ? i - n0 : i);
        int64_t q0 = 0, deg = 0;
        int32_t base = 0;
        if (i < n) {
            q0 = S.offA[sp];
            deg = S.offA[sp + 1] - q0;
            if (S.first && deg > 0) {
                base = plan_base(S, sp);
                if (l8 == 0) S.base[sp] = base;
            }
            if (S.mask) base += BITS;
        }
        // one middle point makes no butterfly (its wedges past the masks are
        // counted all the same)
        const bool wide = deg > PLAN_DEG;
        int64_t W = 0, T = 0;
        if (!wide)
            for (int64_t q = q0 + l8; q < q0 + deg; q += L) {
                int32_t t;
                W += plan_edge(S, sp, base, q, t);
                T += t;
            }
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            W += __shfl_xor_sync(0xffffffffu, W, o);
            T += __shfl_xor_sync(0xffffffffu, T, o);
        }
        const int tier = wide ? CT_WIDE : W > 0 && deg > 1 ? tier_of(p, W, T, deg, sp) : -1;
        const int32_t item = (int32_t)((uint32_t)sp | (uint32_t)side << 31);
        if (l8 == 0 && i < n) wsum += (unsigned long long)W;
        const unsigned any = __reduce_or_sync(0xffffffffu, l8 == 0 && i < n && tier >= 0 ? 1u << tier : 0u);
        for (unsigned m = any; m; m &= m - 1) {
            const int t = __ffs(m) - 1;
            warp_append(l8 == 0 && i < n && tier == t, item, p.n + t, p.list[t]);
        }
    }
    wsum = warp_sum(wsum);
    if (lane == 0 && wsum) atomicAdd(p.wedges, wsum);
}

// A CTA per start point. (256 threads / 512 / 1,024: a hub of degree 69,633 196 / 99
// / 50 us of its plan; counts of 20M edges with degrees up to 100,000 on both sides
// 17.25 / 17.15 / 17.40 ms.)
__global__ void __launch_bounds__(512) k_count_plan_wide(CountPlan p) {
    __shared__ unsigned long long s_w, s_t;
    const int32_t n = p.n[CT_WIDE];
    for (int32_t i = blockIdx.x; i < n; i += gridDim.x) {
        const int32_t item = p.list[CT_WIDE][i];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        if (threadIdx.x == 0) s_w = s_t = 0;
        __syncthreads();
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        const int32_t base = (S.first ? S.base[sp] : 0) + (S.mask ? BITS : 0);
        unsigned long long W = 0, T = 0;
        for (int64_t q = q0 + threadIdx.x; q < q1; q += 512) {
            int32_t t;
            W += (unsigned long long)plan_edge(S, sp, base, q, t);
            T += (unsigned long long)t;
        }
        W = warp_sum(W);
        T = warp_sum(T);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&s_w, W);
            atomicAdd(&s_t, T);
        }
        __syncthreads();
        if (threadIdx.x == 0 && s_w > 0) {
            const int t = tier_of(p, (int64_t)s_w, (int64_t)s_t, q1 - q0, sp);
            p.list[t][atomicAdd(p.n + t, 1)] = item;
            atomicAdd(p.wedges, s_w);
        }
        __syncthreads();
    }
}

struct CountMids {
    const int32_t *adjA;
    const int64_t *offB;
    const int32_t *plen;
    const int32_t *held;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        const int32_t mp = adjA[q];
        beg = offB[mp] + (held ? held[mp] : 0);
        len = plen[q];
    }
};

// Where counts are added: this CTA's copy of the first keys, or the counts.
struct CountSink {
    unsigned long long *cnt, *hot;
    __device__ __forceinline__ CountSink(unsigned long long *c, unsigned long long *h)
        : cnt(c), hot(h ? h + (size_t)(blockIdx.x % HOT_REPS) * HOT_KEYS : nullptr) {}
    __device__ __forceinline__ void add(int32_t k, unsigned long long v) const {
        atomicAdd((hot && k < HOT_KEYS ? hot : cnt) + k, v);
    }
};

__global__ void k_count_merge(CountPlan p) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const CountSide &S = p.s[blockIdx.y];
    if (k >= HOT_KEYS || k >= S.nA) return;
    unsigned long long v = 0;
#pragma unroll 8
    for (int r = 0; r < HOT_REPS; r++) v += S.hotA[(size_t)r * HOT_KEYS + k];
    S.cntA[k] += v;
}

// ---------------- bit-sliced part ----------------
// Word l of a mask holds the keys 32 b + l (bit b), relative to the first key:
// consecutive keys lie in consecutive lanes.

// Masks of all lists of one side over the other side's first BITS keys (of
// each packed graph), one warp per list.
__global__ void __launch_bounds__(256) k_count_masks(const int64_t *__restrict__ off,
                                                     const int32_t *__restrict__ adj, int32_t n,
                                                     const int32_t *__restrict__ first_own,
                                                     const int32_t *__restrict__ first_keys, int ng,
                                                     uint32_t *__restrict__ mask,
                                                     int32_t *__restrict__ held) {
    __shared__ uint32_t s_w[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t y = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; y < n; y += nw) {
        const int64_t q0 = off[y], q1 = off[y + 1];
        int32_t base = 0;
        if (first_own) {
            int lo = 0, hi = ng - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (first_own[mid] <= y)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            base = first_keys[lo];
        }
        s_w[w][lane] = 0;
        __syncwarp();
        int32_t in = 0;
        for (int64_t qb = q0; qb < q1; qb += 32) {
            const int32_t k = qb + lane < q1 ? adj[qb + lane] - base : BITS;
            if (k < BITS) atomicOr(&s_w[w][k & 31], 1u << (k >> 5));
            const unsigned bal = __ballot_sync(0xffffffffu, k < BITS);
            in += __popc(bal);
            if (bal != 0xffffffffu) break;
        }
        __syncwarp();
        mask[y * 32 + lane] = s_w[w][lane];
        if (lane == 0) held[y] = in;
        __syncwarp();
    }
}

// Keys below `lim` (0..BITS) in this lane's word.
__device__ __forceinline__ uint32_t keys_below(int32_t lim, int lane) {
    const uint32_t d = (uint32_t)max(lim - lane + 31, 0) >> 5;  // 0..32
    uint32_t m;
    asm("shl.b32 %0, 1, %1;" : "=r"(m) : "r"(d));  // 0 when d = 32
    return m - 1u;
}

// (carry, sum) of three words
__device__ __forceinline__ uint32_t csa(uint32_t &sum, uint32_t a, uint32_t b) {
    const uint32_t c = (sum & a) | (sum & b) | (a & b);
    sum ^= a ^ b;
    return c;
}

// Adds eight words to the planes: a tree of carry-save adders, then the
// weight-8 carry through the upper planes.
template <int NP>
__device__ __forceinline__ void add8(uint32_t (&pl)[NP], const uint32_t (&w)[8]) {
    const uint32_t a2 = csa(pl[0], w[0], w[1]), b2 = csa(pl[0], w[2], w[3]);
    const uint32_t a4 = csa(pl[1], a2, b2);
    const uint32_t c2 = csa(pl[0], w[4], w[5]), d2 = csa(pl[0], w[6], w[7]);
    const uint32_t b4 = csa(pl[1], c2, d2);
    uint32_t c = csa(pl[2], a4, b4);
#pragma unroll
    for (int p = 3; p < NP; p++) {
        const uint32_t t = pl[p] & c;
        pl[p] ^= c;
        c = t;
    }
}

// One start point's middle points [q0, q1), warp `part` of `parts`: their
// masks added to the planes; the wedges of this lane's keys.
template <int NP>
__device__ __forceinline__ uint32_t bits_add(const CountSide &S, int32_t sp, int32_t base, int64_t q0,
                                             int64_t q1, int part, int parts, int lane,
                                             uint32_t (&pl)[NP]) {
    uint32_t wedges = 0;
    for (int64_t qb = q0 + 32 * part; qb < q1; qb += 32 * parts) {
        int32_t mp = 0, lim = 0;
        if (qb + lane < q1) {
            mp = S.adjA[qb + lane];
            lim = min(min(sp, S.belowB[mp]) - base, BITS);
        }
        const int cnt = (int)imin64(32, q1 - qb);
        for (int j0 = 0; j0 < cnt; j0 += 8) {
            uint32_t w[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int32_t l = __shfl_sync(0xffffffffu, lim, j0 + u);
                const int32_t m = __shfl_sync(0xffffffffu, mp, j0 + u);
                w[u] = l > 0 ? __ldg(S.mask + (size_t)m * 32 + lane) & keys_below(l, lane) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 8; u++) wedges += __popc(w[u]);
            add8<NP>(pl, w);
        }
    }
    return wedges;
}

// The opposite side: sum over a middle point's keys of (count - 1); it is at
// most 1,024 times the start point's degree.
template <int NP>
__device__ __forceinline__ void bits_opposite(const CountSide &S, const CountSink &opp, int32_t sp,
                                              int32_t base, int64_t q0, int64_t q1, int part, int parts,
                                              int lane, const uint32_t (&pl)[NP], int top) {
    using Acc = typename std::conditional<(NP > 20), unsigned long long, uint32_t>::type;
    for (int64_t qb = q0 + 32 * part; qb < q1; qb += 32 * parts) {
        int32_t mp = 0, lim = 0;
        if (qb + lane < q1) {
            mp = S.adjA[qb + lane];
            lim = min(min(sp, S.belowB[mp]) - base, BITS);
        }
        const int cnt = (int)imin64(32, q1 - qb);
        Acc mine = 0;
        for (int j0 = 0; j0 < cnt; j0 += 4) {
            uint32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int32_t l = __shfl_sync(0xffffffffu, lim, j0 + u);
                const int32_t m = __shfl_sync(0xffffffffu, mp, j0 + u);
                w[u] = l > 0 ? __ldg(S.mask + (size_t)m * 32 + lane) & keys_below(l, lane) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                Acc v = (Acc)__popc(w[u] & pl[0]) - (Acc)__popc(w[u]);
#pragma unroll
                for (int p = 1; p < NP; p++) {
                    if (p > top) break;
                    v += (Acc)__popc(w[u] & pl[p]) << p;
                }
                if constexpr (NP > 20)
                    v = warp_sum(v);
                else
                    v = __reduce_add_sync(0xffffffffu, v);
                if (lane == j0 + u) mine = v;
            }
        }
        if (mine) opp.add(mp, mine);
    }
}

// The same side: C(c, 2) of the keys of this warp's bits (b = part, part +
// parts, ...) to the end points; returns this lane's sum.
template <int NP>
__device__ __forceinline__ unsigned long long bits_same(const CountSink &same, int32_t base, int part,
                                                        int parts, int lane,
                                                        const uint32_t (&pl)[NP], uint32_t twos) {
    unsigned long long acc = 0;
    uint32_t any = __reduce_or_sync(0xffffffffu, twos);
    while (any) {
        const int b = __ffs(any) - 1;
        any &= any - 1;
        if (b % parts != part) continue;
        uint32_t c = 0;
#pragma unroll
        for (int p = 0; p < NP; p++) c |= ((pl[p] >> b) & 1u) << p;
        if (c >= 2) {
            const unsigned long long v = choose2(c);
            same.add(base + 32 * b + lane, v);
            acc += v;
        }
    }
    return acc;
}

// Highest plane with a bit (-1: none), the same in every lane.
template <int NP>
__device__ __forceinline__ int top_plane(const uint32_t (&pl)[NP]) {
    uint32_t used = 0;
#pragma unroll
    for (int p = 0; p < NP; p++) used |= pl[p] ? 1u << p : 0u;
    return 31 - __clz(__reduce_or_sync(0xffffffffu, used));
}

// One warp per start point of degree below BITS_DEG, both sides.
__global__ void __launch_bounds__(256) k_count_bits(CountPlan p) {
    constexpr int NP = 10;
    static_assert(BITS_DEG <= 1 << NP, "counts fit the planes");
    const int lane = threadIdx.x & 31;
    const int64_t n0 = p.s[0].nA, n = n0 + p.s[1].nA;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long wedges = 0;
    // consecutive start points (of similar degree) on different CTAs
    for (int64_t i = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; i < n; i += nw) {
        const int side = i >= n0 ? 1 : 0;
        const CountSide &S = p.s[side];
        const int32_t sp = (int32_t)(side ? i - n0 : i);
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        if (q1 == q0) continue;
        if (q1 - q0 >= BITS_DEG) {
            const int t = q1 - q0 >= HUGE_DEG ? CT_HUGE : CT_BITS;
            if (lane == 0)
                p.list[t][atomicAdd(p.n + t, 1)] = (int32_t)((uint32_t)sp | (uint32_t)side << 31);
            continue;
        }
        const int32_t base = S.first ? S.base[sp] : 0;
        uint32_t pl[NP] = {};
        wedges += bits_add<NP>(S, sp, base, q0, q1, 0, 1, lane, pl);
        const int top = top_plane<NP>(pl);
        if (top < 1) continue;  // no end point twice
        uint32_t twos = 0;
#pragma unroll
        for (int k = 1; k < NP; k++) twos |= pl[k];
        const CountSink same(S.cntA, S.hotA), opp(S.cntB, S.hotB);
        const unsigned long long acc = warp_sum(bits_same<NP>(same, base, 0, 1, lane, pl, twos));
        if (lane == 0) same.add(sp, acc);
        bits_opposite<NP>(S, opp, sp, base, q0, q1, 0, 1, lane, pl, top);
    }
    wedges = warp_sum(wedges);
    if (lane == 0 && wedges) atomicAdd(p.wedges, wedges);
}

// Sums the 16 warps' planes of a CTA (bit-sliced adders in a tree); the total
// ends in s_pl[0] and in every warp's planes.
template <int NP>
__device__ __forceinline__ void cta_sum_planes(uint32_t (&pl)[NP], uint32_t (*s_pl)[NP][32], int warp,
                                               int lane) {
    for (int h = 8; h > 0; h >>= 1) {
        __syncthreads();
        if (warp >= h && warp < 2 * h)
#pragma unroll
            for (int k = 0; k < NP; k++) s_pl[warp - h][k][lane] = pl[k];
        __syncthreads();
        if (warp < h) {
            uint32_t c = 0;
#pragma unroll
            for (int k = 0; k < NP; k++) {
                const uint32_t b = s_pl[warp][k][lane], a = pl[k];
                pl[k] = a ^ b ^ c;
                c = (a & b) | (a & c) | (b & c);
            }
        }
    }
    if (warp == 0)
#pragma unroll
        for (int k = 0; k < NP; k++) s_pl[0][k][lane] = pl[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NP; k++) pl[k] = s_pl[0][k][lane];
}

template <int NP>
__device__ __forceinline__ uint32_t upper_planes(const uint32_t (&pl)[NP]) {
    uint32_t t = 0;
#pragma unroll
    for (int k = 1; k < NP; k++) t |= pl[k];
    return t;
}

// One CTA per start point of degree below HUGE_DEG: every warp adds up its
// share of the middle points.
__global__ void __launch_bounds__(512) k_count_bits_wide(CountPlan p) {
    constexpr int NP = 13, NW = 16;
    static_assert(HUGE_DEG <= 1 << NP, "counts fit the planes");
    __shared__ uint32_t s_pl[NW / 2][NP][32];
    __shared__ unsigned long long s_acc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t n = p.n[CT_BITS];
    unsigned long long wedges = 0;
    for (int32_t i = blockIdx.x; i < n; i += gridDim.x) {
        const int32_t item = p.list[CT_BITS][i];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        const int32_t base = S.first ? S.base[sp] : 0;
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        uint32_t pl[NP] = {};
        wedges += bits_add<NP>(S, sp, base, q0, q1, warp, NW, lane, pl);
        if (threadIdx.x == 0) s_acc = 0;
        cta_sum_planes<NP>(pl, s_pl, warp, lane);
        const int top = top_plane<NP>(pl);
        if (top >= 1) {
            const CountSink same(S.cntA, S.hotA), opp(S.cntB, S.hotB);
            const unsigned long long acc =
                warp_sum(bits_same<NP>(same, base, warp, NW, lane, pl, upper_planes<NP>(pl)));
            if (lane == 0 && acc) atomicAdd(&s_acc, acc);
            bits_opposite<NP>(S, opp, sp, base, q0, q1, warp, NW, lane, pl, top);
            __syncthreads();
            if (threadIdx.x == 0 && s_acc) same.add(sp, s_acc);
        }
        __syncthreads();
    }
    wedges = warp_sum(wedges);
    if (lane == 0 && wedges) atomicAdd(p.wedges, wedges);
}

// Start points of very high degree, a CTA per HUGE_DEG middle points: the
// chunks' planes go to global memory (k_huge_add), are summed per start point
// (k_huge_sum, which makes the same-side updates), and every chunk makes its
// opposite-side updates (k_huge_opposite). (One CTA per start point took 1.9
// ms for the 10M-edge graph's hub of degree 50,000 alone.)
constexpr int HUGE_NP = 31;  // counts are below 2^31 (degrees)

__global__ void k_huge_plan(CountPlan p) {
    if (threadIdx.x != 0) return;
    int32_t at = 0;
    const int32_t n = p.n[CT_HUGE];
    for (int32_t i = 0; i < n; i++) {
        const int32_t item = p.list[CT_HUGE][i];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        p.hoff[i] = at;
        at += (int32_t)((S.offA[sp + 1] - S.offA[sp] + HUGE_DEG - 1) / HUGE_DEG);
    }
    p.hoff[n] = at;
}

struct HugeChunk {
    int32_t sp, base;
    int64_t q0, q1;
    int side, item;
    __device__ __forceinline__ HugeChunk(const CountPlan &p, int32_t c) {
        int32_t lo = 0, hi = p.n[CT_HUGE] - 1;
        while (lo < hi) {
            const int32_t mid = (lo + hi + 1) >> 1;
            if (p.hoff[mid] <= c)
                lo = mid;
            else
                hi = mid - 1;
        }
        item = lo;
        const int32_t it = p.list[CT_HUGE][lo];
        side = it < 0 ? 1 : 0;
        sp = it & 0x7fffffff;
        const CountSide &S = p.s[side];
        base = S.first ? S.base[sp] : 0;
        q0 = S.offA[sp] + (int64_t)(c - p.hoff[lo]) * HUGE_DEG;
        q1 = imin64(q0 + HUGE_DEG, S.offA[sp + 1]);
    }
};

__global__ void __launch_bounds__(512) k_huge_add(CountPlan p) {
    constexpr int NP = 14, NW = 16;  // one chunk's counts reach 2^13
    __shared__ uint32_t s_pl[NW / 2][NP][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t nc = p.hoff[p.n[CT_HUGE]];
    unsigned long long wedges = 0;
    for (int32_t c = blockIdx.x; c < nc; c += gridDim.x) {
        const HugeChunk h(p, c);
        uint32_t pl[NP] = {};
        wedges += bits_add<NP>(p.s[h.side], h.sp, h.base, h.q0, h.q1, warp, NW, lane, pl);
        cta_sum_planes<NP>(pl, s_pl, warp, lane);
        if (warp == 0)
#pragma unroll
            for (int k = 0; k < HUGE_NP; k++)
                p.hplanes[((size_t)c * HUGE_NP + k) * 32 + lane] = k < NP ? pl[k < NP ? k : 0] : 0u;
        __syncthreads();
    }
    wedges = warp_sum(wedges);
    if (lane == 0 && wedges) atomicAdd(p.wedges, wedges);
}

// One warp per start point: its total over the chunks, left in its first
// chunk's planes, and the same-side updates.
__global__ void __launch_bounds__(32) k_huge_sum(CountPlan p) {
    constexpr int NP = HUGE_NP;
    const int lane = threadIdx.x;
    const int32_t n = p.n[CT_HUGE];
    for (int32_t i = blockIdx.x; i < n; i += gridDim.x) {
        const int32_t item = p.list[CT_HUGE][i];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        uint32_t pl[NP] = {};
        for (int32_t c = p.hoff[i]; c < p.hoff[i + 1]; c++) {
            uint32_t carry = 0;
#pragma unroll
            for (int k = 0; k < NP; k++) {
                const uint32_t b = p.hplanes[((size_t)c * NP + k) * 32 + lane], a = pl[k];
                pl[k] = a ^ b ^ carry;
                carry = (a & b) | (a & carry) | (b & carry);
            }
        }
#pragma unroll
        for (int k = 0; k < NP; k++) p.hplanes[((size_t)p.hoff[i] * NP + k) * 32 + lane] = pl[k];
        const CountSink same(S.cntA, S.hotA);
        const unsigned long long acc = warp_sum(
            bits_same<NP>(same, S.first ? S.base[sp] : 0, 0, 1, lane, pl, upper_planes<NP>(pl)));
        if (lane == 0 && acc) same.add(sp, acc);
    }
}

__global__ void __launch_bounds__(512) k_huge_opposite(CountPlan p) {
    constexpr int NP = HUGE_NP;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t nc = p.hoff[p.n[CT_HUGE]];
    for (int32_t c = blockIdx.x; c < nc; c += gridDim.x) {
        const HugeChunk h(p, c);
        const CountSide &S = p.s[h.side];
        uint32_t pl[NP];
#pragma unroll
        for (int k = 0; k < NP; k++)
            pl[k] = p.hplanes[((size_t)p.hoff[h.item] * NP + k) * 32 + lane];
        const int top = top_plane<NP>(pl);
        if (top < 1) continue;
        const CountSink opp(S.cntB, S.hotB);
        bits_opposite<NP>(S, opp, h.sp, h.base, h.q0, h.q1, warp, 16, lane, pl, top);
    }
}

// ---------------- warp tier ----------------
// A start point's hash table, slots a power of two with load <= 1/2 (an item
// of few wedges clears and reads few slots).
struct CountTable {
    int32_t *key;
    uint32_t *val;
    __device__ __forceinline__ int add(int32_t k, uint32_t mask) {
        uint32_t h = (hash_key(k) >> 16) & mask;
        for (uint32_t p = 0; p <= mask; p++) {
            int32_t cur = ((volatile int32_t *)key)[h];
            if (cur == EMPTY_KEY) {
                cur = atomicCAS(&key[h], EMPTY_KEY, k);
                if (cur == EMPTY_KEY) cur = k;
            }
            if (cur == k) {
                atomicAdd(&val[h], 1u);
                return (int)h;
            }
            h = (h + 1) & mask;
        }
        return 0;
    }
};

// One warp per start point. The wedges of 32 middle vertices are numbered by a
// warp scan and dealt to the lanes, so all their key loads are independent
// (middle vertex by middle vertex, each step waited for the last: 2.4 ms
// against 0.7 for the 10M-edge graph's two sides). A list of at most 32 middle
// vertices, the usual case, is walked once: every lane keeps the slots of its
// (at most 8) wedges for the opposite side's sums.
__global__ void __launch_bounds__(256) k_count_warp(CountPlan p) {
    __shared__ int32_t skey[8][WARP_SLOTS];
    __shared__ uint32_t sval[8][WARP_SLOTS];
    __shared__ uint32_t sacc[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    CountTable H{skey[w], sval[w]};
    for (int i = lane; i < WARP_SLOTS; i += 32) {
        H.key[i] = EMPTY_KEY;
        H.val[i] = 0;
    }
    sacc[w][lane] = 0;
    __syncwarp();
    const int32_t n = p.n[CT_WARP];
    const int32_t nw = (gridDim.x * blockDim.x) >> 5;
    constexpr int U = WARP_MAX_W / 32;
    for (int32_t idx = w * gridDim.x + blockIdx.x; idx < n; idx += nw) {
        const int32_t item = p.list[CT_WARP][idx];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        const bool one = q1 - q0 <= 32;
        const CountSink same(S.cntA, S.hotA), opp(S.cntB, S.hotB);
        uint32_t mask = WARP_SLOTS - 1;
        int slot[U], seg[U];
        int32_t mp = 0;
        // pass 0 fills the table; pass 1 (more than 32 middle vertices) walks
        // again for the opposite side
        auto walk = [&](int pass, int64_t qb) {
            int32_t len = 0;
            int64_t beg = 0;
            mp = 0;
            if (qb + lane < q1) {
                mp = S.adjA[qb + lane];
                len = S.plen[qb + lane];
                beg = S.offB[mp] + (S.held ? S.held[mp] : 0);
            }
            int32_t inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            const int32_t tot = __shfl_sync(0xffffffffu, inc, 31), ex = inc - len;
            if (one) mask = tot <= 32 ? 63u : tot <= 64 ? 127u : tot <= 128 ? 255u : WARP_SLOTS - 1;
            int32_t key[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                seg[u] = -1;
                if (u * 32 >= tot) continue;
                const int32_t j = u * 32 + lane;
                int lo = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int32_t e = __shfl_sync(0xffffffffu, ex, lo + step);
                    if (e <= j) lo += step;
                }
                const int64_t b = __shfl_sync(0xffffffffu, beg, lo);
                const int32_t e0 = __shfl_sync(0xffffffffu, ex, lo);
                if (j < tot) {
                    seg[u] = lo;
                    key[u] = __ldg(S.adjB + b + (j - e0));
                }
            }
#pragma unroll
            for (int u = 0; u < U; u++)
                if (seg[u] >= 0) {
                    if (pass == 0) {
                        slot[u] = H.add(key[u], mask);
                    } else {
                        uint32_t h = (hash_key(key[u]) >> 16) & mask;
                        while (H.key[h] != key[u]) h = (h + 1) & mask;
                        slot[u] = (int)h;
                    }
                }
            __syncwarp();
        };
        // per middle vertex: sum over its wedges of (count - 1)
        auto opposite = [&]() {
#pragma unroll
            for (int u = 0; u < U; u++)
                if (seg[u] >= 0) {
                    const uint32_t c = H.val[slot[u]];
                    if (c > 1) atomicAdd(&sacc[w][seg[u]], c - 1);
                }
            __syncwarp();
            const uint32_t a = sacc[w][lane];
            if (a) {
                opp.add(mp, a);
                sacc[w][lane] = 0;
            }
            __syncwarp();
        };
        for (int64_t qb = q0; qb < q1; qb += 32) walk(0, qb);
        if (one) {
            opposite();
        } else {
            for (int64_t qb = q0; qb < q1; qb += 32) {
                walk(1, qb);
                opposite();
            }
        }
        // same side: C(c, 2) to ep and (summed) to sp; the table empty again
        unsigned long long acc = 0;
        for (uint32_t i = lane; i <= mask; i += 32) {
            const int32_t k = H.key[i];
            if (k == EMPTY_KEY) continue;
            const uint32_t c = H.val[i];
            if (c >= 2) {
                const unsigned long long b = choose2(c);
                same.add(k, b);
                acc += b;
            }
            H.key[i] = EMPTY_KEY;
            H.val[i] = 0;
        }
        acc = warp_sum(acc);
        if (lane == 0 && acc) same.add(sp, acc);
        __syncwarp();
    }
}

// ---------------- CTA tiers ----------------
struct CountSameEmit {
    CountSink sink;
    int32_t base;  // first key
    unsigned long long acc;
    __device__ __forceinline__ void operator()(int32_t k, uint32_t c) {
        const unsigned long long b = choose2(c);
        sink.add(k + base, b);
        acc += b;
    }
};

// Acc: what a middle vertex's sum over one start point fits. The end points
// of a prefix are distinct, so the sum is at most the start point's wedges:
// 32 bits unless those reach 2^32 (64-bit atomics in shared memory are a
// compare-and-swap loop: the lanes of a group that spans several short
// segments took turns for thousands of cycles).
template <class Eng, class Acc>
struct CountOppVisit {
    Eng *eng;
    Acc *sacc;  // per-mid accumulator (shared)
    int32_t base;              // first key
    // One walk step: where all the warp's wedges of a group share one middle
    // vertex (long lists), the warp sums its contributions first and makes
    // one shared-memory atomic instead of 32 to the same word.
    template <int N>
    __device__ __forceinline__ void many(const int (&kk)[N], const int32_t (&key)[N]) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int u = 0; u < N; u++) {
            uint32_t v = 0;
            if (key[u] >= 0) {
                const uint32_t c = eng->count(key[u] - base);
                v = c > 1 ? c - 1 : 0;
            }
            const int k = key[u] >= 0 ? kk[u] : -1;
            const unsigned valid = __ballot_sync(0xffffffffu, k >= 0);
            if (!valid) continue;
            const int kl = __shfl_sync(0xffffffffu, k, __ffs(valid) - 1);
            if (__all_sync(0xffffffffu, k < 0 || k == kl)) {
                const uint32_t sum = __reduce_add_sync(0xffffffffu, v);
                if (lane == 0 && sum) atomicAdd(&sacc[kl], (Acc)sum);
            } else if (v) {
                atomicAdd(&sacc[k], (Acc)v);
            }
        }
    }
};

template <class Acc>
struct CountOppHook {
    const int32_t *adjA;
    CountSink sink;
    Acc *sacc;
    __device__ void operator()(int64_t c0, int nm) {
        if ((int)threadIdx.x < nm) {
            const Acc s = sacc[threadIdx.x];
            if (s) sink.add(adjA[c0 + threadIdx.x], s);
            sacc[threadIdx.x] = 0;
        }
    }
};

template <class Eng>
struct AddVisit {
    Eng *eng;
    int32_t base;
    __device__ __forceinline__ void operator()(int, int32_t key) { eng->add(key - base); }
};

__device__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long *tmp) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) tmp[w] = v;
    __syncthreads();
    unsigned long long r = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) r += tmp[i];
    __syncthreads();
    return r;
}

// Counters for the first keys (two 16-bit ones per word: key k < hw in the low
// half of word k, the others in the high half of word k - hw) and a hash table
// for the rest, which the plan has made sure can hold them.
template <int TAIL>
struct HeadTail {
    uint32_t *head;  // COUNT_HEAD / 2
    CtaHashT<TAIL> tail;
    int32_t headn, hw;

    static constexpr size_t bytes() { return (size_t)COUNT_HEAD * 2 + CtaHashT<TAIL>::bytes(); }
    __device__ unsigned char *bind(unsigned char *base, int *nt) {
        head = (uint32_t *)base;
        return tail.bind(base + COUNT_HEAD * 2, nt);
    }
    __device__ void clear_all() {
        for (int i = threadIdx.x; i < COUNT_HEAD / 8; i += blockDim.x)
            ((uint4 *)head)[i] = make_uint4(0, 0, 0, 0);
        tail.clear_all();
    }
    __device__ void set_keys(int32_t keys) {
        headn = keys < COUNT_HEAD ? keys : COUNT_HEAD;
        hw = (headn + 1) >> 1;
    }
    // (calls: the few keys past the head do not pay for their code in every
    // copy of a visit)
    __device__ __noinline__ void add_tail(int32_t k) { tail.add(k); }
    __device__ __noinline__ uint32_t count_tail(int32_t k) const { return tail.count(k); }
    __device__ __forceinline__ void add(int32_t k) {
        if (k < headn) {
            const bool hi = k >= hw;
            atomicAdd(&head[hi ? k - hw : k], hi ? 0x10000u : 1u);
        } else {
            add_tail(k);
        }
    }
    __device__ __forceinline__ uint32_t count(int32_t k) const {
        if (k < headn) {
            const bool hi = k >= hw;
            return (head[hi ? k - hw : k] >> (hi ? 16 : 0)) & 0xffffu;
        }
        return count_tail(k);
    }
    template <class Emit>
    __device__ __forceinline__ void emit_all(Emit &emit) {
        // consecutive lanes, consecutive keys: a warp's atomics fall into few
        // cache lines
#pragma unroll 4
        for (int i = threadIdx.x; i < hw; i += blockDim.x) {
            const uint32_t v = head[i];
            const uint32_t c0 = v & 0xffffu, c1 = v >> 16;
            if (c0 >= 2) emit(i, c0);
            if (c1 >= 2) emit(i + hw, c1);
        }
        tail.template sweep<true, false>(emit);
    }
    __device__ __forceinline__ void clear() {
        for (int i = threadIdx.x; i < (hw + 3) / 4; i += blockDim.x)
            ((uint4 *)head)[i] = make_uint4(0, 0, 0, 0);
        NoEmit ne;
        tail.template sweep<false, true>(ne);
    }
};

// One THREADS-thread CTA per start point: walk (counts), C(c, 2) to the end
// points and the start point, second walk (count - 1 to the middle points).
template <int THREADS, int TAIL>
__global__ void __launch_bounds__(THREADS) k_count_dense(CountPlan p, int tier) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_idx, s_nt;
    __shared__ unsigned long long s_acc;
    const int32_t n = p.n[tier];
    if ((int32_t)blockIdx.x >= n) return;
    HeadTail<TAIL> H;
    unsigned char *q = H.bind(smem, &s_nt);
    Chunk ch;
    ch.beg = (int64_t *)q;
    uint32_t *sacc = (uint32_t *)(ch.beg + THREADS);
    ch.pre = (int32_t *)(sacc + THREADS);
    ch.tmp = ch.pre + THREADS + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    H.clear_all();
    sacc[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_acc = 0;
    __syncthreads();
    for (int idx = blockIdx.x; idx < n;) {
        const int32_t item = p.list[tier][idx];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        const int32_t base = (S.first ? S.base[sp] : 0) + (S.mask ? BITS : 0);
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        H.set_keys(sp - base);
        CountMids M{S.adjA, S.offB, S.plen, S.held};
        AddVisit<HeadTail<TAIL>> add{&H, base};
        cta_walk<true, KeysNc, THREADS < 512 ? 4 : 8>(M, q0, q1, S.adjB, ch, add);
        CountSameEmit em{CountSink(S.cntA, S.hotA), base, 0};
        H.emit_all(em);
        const unsigned long long tot = warp_sum(em.acc);
        if ((threadIdx.x & 31) == 0 && tot) atomicAdd(&s_acc, tot);
        CountOppVisit<HeadTail<TAIL>, uint32_t> ov{&H, sacc, base};
        CountOppHook<uint32_t> hook{S.adjA, CountSink(S.cntB, S.hotB), sacc};
        cta_walk<true, KeysNc, THREADS < 512 ? 4 : 8>(M, q0, q1, S.adjB, ch, ov, &hook);  // (its barriers cover s_acc too)
        H.clear();
        if (threadIdx.x == 0) {
            if (s_acc) em.sink.add(sp, s_acc);
            s_acc = 0;
            s_idx = (int)gridDim.x + atomicAdd(p.n + CT_LISTS + tier, 1);
        }
        __syncthreads();
        idx = s_idx;
        H.tail.reset_scalars();
        __syncthreads();
    }
}
template <int THREADS, int TAIL>
constexpr size_t count_dense_smem() {
    return HeadTail<TAIL>::bytes() + THREADS * 4 + chunk_bytes(THREADS);
}

__global__ void __maxnreg__(64) k_count_cta(CountPlan p, int32_t head_cap, int32_t bm_cap) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_idx, s_used, s_over;
    __shared__ unsigned long long s_red[32];
    const int32_t n = p.n[CT_HYBRID];
    if ((int32_t)blockIdx.x >= n) return;
    CtaHybrid H;
    unsigned char *q = H.bind(smem, head_cap, bm_cap, &s_used, &s_over);
    Chunk ch;
    ch.beg = (int64_t *)q;
    unsigned long long *sacc = (unsigned long long *)(ch.beg + MID_CHUNK);
    ch.pre = (int32_t *)(sacc + MID_CHUNK);
    ch.tmp = ch.pre + MID_CHUNK + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    H.clear_all();
    for (int i = threadIdx.x; i < MID_CHUNK; i += blockDim.x) sacc[i] = 0;
    __syncthreads();
    NoEmit ne;
    for (;;) {
        if (threadIdx.x == 0) s_idx = atomicAdd(p.n + CT_LISTS + CT_HYBRID, 1);
        __syncthreads();
        int idx = s_idx;
        if (idx >= n) break;
        const int32_t item = p.list[CT_HYBRID][idx];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        CountMids M{S.adjA, S.offB, S.plen, S.held};
        H.set_range((int32_t)imin64(head_cap, sp), sp);
        AddVisit<CtaHybrid> add{&H, 0};
        cta_walk(M, q0, q1, S.adjB, ch, add);
        const bool over = s_over;
        if (!over) {
            CountSameEmit em{CountSink(S.cntA, S.hotA), 0, 0};
            H.sweep<true, false>(em);
            unsigned long long tot = block_sum_u64(em.acc, s_red);
            if (threadIdx.x == 0 && tot) atomicAdd(&S.cntA[sp], tot);
            CountOppVisit<CtaHybrid, unsigned long long> ov{&H, sacc, 0};
            CountOppHook<unsigned long long> hook{S.adjA, CountSink(S.cntB, S.hotB), sacc};
            cta_walk(M, q0, q1, S.adjB, ch, ov, &hook);
        } else if (threadIdx.x == 0) {
            p.list[CT_OVER][atomicAdd(p.n + CT_OVER, 1)] = item;
        }
        __syncthreads();
        H.sweep<false, true>(ne);
        __syncthreads();
        H.reset_scalars();
    }
}

// gcnt, gtouch: `keyspace` words per CTA; gcnt is cleared here.
__global__ void __maxnreg__(64) k_count_global(CountPlan p, uint32_t *gcnt, int32_t *gtouch,
                                               int64_t keyspace) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_idx, s_nt;
    __shared__ unsigned long long s_red[32];
    const int32_t n1 = p.n[CT_GLOBAL], n2 = p.n[CT_OVER];
    if (n1 + n2 == 0) return;
    Chunk ch;
    ch.beg = (int64_t *)smem;
    unsigned long long *sacc = (unsigned long long *)(ch.beg + MID_CHUNK);
    ch.pre = (int32_t *)(sacc + MID_CHUNK);
    ch.tmp = ch.pre + MID_CHUNK + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    GlobalDense G{gcnt + (size_t)blockIdx.x * keyspace, gtouch + (size_t)blockIdx.x * keyspace, &s_nt};
    for (int i = threadIdx.x; i < MID_CHUNK; i += blockDim.x) sacc[i] = 0;
    for (int64_t i = threadIdx.x; i < keyspace; i += blockDim.x) G.cnt[i] = 0;
    for (;;) {
        if (threadIdx.x == 0) {
            s_idx = atomicAdd(p.n + CT_LISTS + CT_GLOBAL, 1);
            s_nt = 0;
        }
        __syncthreads();
        int idx = s_idx;
        if (idx >= n1 + n2) break;
        const int32_t item = idx < n1 ? p.list[CT_GLOBAL][idx] : p.list[CT_OVER][idx - n1];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        CountMids M{S.adjA, S.offB, S.plen, S.held};
        AddVisit<GlobalDense> add{&G, 0};
        cta_walk(M, q0, q1, S.adjB, ch, add);
        CountSameEmit em{CountSink(S.cntA, S.hotA), 0, 0};
        G.flush(em);
        unsigned long long tot = block_sum_u64(em.acc, s_red);
        if (threadIdx.x == 0 && tot) atomicAdd(&S.cntA[sp], tot);
        CountOppVisit<GlobalDense, unsigned long long> ov{&G, sacc, 0};
        CountOppHook<unsigned long long> hook{S.adjA, CountSink(S.cntB, S.hotB), sacc};
        cta_walk(M, q0, q1, S.adjB, ch, ov, &hook);
        G.clear();
        __syncthreads();
    }
}

// Start points with at most HASH_W wedges: one 256-thread CTA each (several
// per SM) with a shared hash table; the same two walks as the other tiers.
__global__ void __launch_bounds__(HASH_THREADS, 4) k_count_hash(CountPlan p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_idx, s_nt;
    __shared__ unsigned long long s_red[32];
    const int32_t n = p.n[CT_HASH];
    if ((int32_t)blockIdx.x >= n) return;
    CountHash H;
    unsigned char *q = H.bind(smem, &s_nt);
    Chunk ch;
    ch.beg = (int64_t *)q;
    uint32_t *sacc = (uint32_t *)(ch.beg + HASH_THREADS);
    ch.pre = (int32_t *)(sacc + HASH_THREADS);
    ch.tmp = ch.pre + HASH_THREADS + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    H.clear_all();
    for (int i = threadIdx.x; i < HASH_THREADS; i += blockDim.x) sacc[i] = 0;
    __syncthreads();
    NoEmit ne;
    for (;;) {
        if (threadIdx.x == 0) s_idx = atomicAdd(p.n + CT_LISTS + CT_HASH, 1);
        __syncthreads();
        const int idx = s_idx;
        if (idx >= n) break;
        const int32_t item = p.list[CT_HASH][idx];
        const CountSide &S = p.s[item < 0 ? 1 : 0];
        const int32_t sp = item & 0x7fffffff;
        const int64_t q0 = S.offA[sp], q1 = S.offA[sp + 1];
        CountMids M{S.adjA, S.offB, S.plen, S.held};
        AddVisit<CountHash> add{&H, 0};
        cta_walk(M, q0, q1, S.adjB, ch, add);
        CountSameEmit em{CountSink(S.cntA, S.hotA), 0, 0};
        H.sweep<true, false>(em);
        const unsigned long long tot = block_sum_u64(em.acc, s_red);
        if (threadIdx.x == 0 && tot) atomicAdd(&S.cntA[sp], tot);
        CountOppVisit<CountHash, uint32_t> ov{&H, sacc, 0};
        CountOppHook<uint32_t> hook{S.adjA, CountSink(S.cntB, S.hotB), sacc};
        cta_walk(M, q0, q1, S.adjB, ch, ov, &hook);
        H.sweep<false, true>(ne);
        __syncthreads();
        H.reset_scalars();
    }
}

size_t count_cta_smem(int64_t keyspace, int32_t *head_cap, int32_t *bm_cap) {
    return hybrid_bytes(keyspace, head_cap, bm_cap) + MID_CHUNK * 8 /*sacc*/ + CHUNK_BYTES;
}

size_t count_hash_smem() { return CountHash::bytes() + HASH_THREADS * 4 + chunk_bytes(HASH_THREADS); }

void launch_plan(const CountPlan &p, int64_t n, cudaStream_t s) {
    const int64_t sms = num_sms();
    // a warp each while the start points do not fill the SMs eight lanes at a time
    if (n <= sms * 64)
        k_count_plan<32><<<(unsigned)((n + 7) / 8), 256, 0, s>>>(p);
    else
        k_count_plan<8><<<(unsigned)std::min<int64_t>((n + 31) / 32, sms * 32), 256, 0, s>>>(p);
    RC_LAUNCH();
}

template <int THREADS, int TAIL>
void launch_dense(const CountPlan &p, int tier, int64_t items, cudaStream_t s) {
    constexpr size_t smem = count_dense_smem<THREADS, TAIL>();
    const void *fn = (const void *)k_count_dense<THREADS, TAIL>;
    allow_max_smem(fn);
    int occ = 1;
    RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, THREADS, smem));
    const int64_t grid = std::min<int64_t>(items, (int64_t)num_sms() * std::max(1, occ));
    k_count_dense<THREADS, TAIL><<<(unsigned)grid, THREADS, smem, s>>>(p, tier);
    RC_LAUNCH();
}

// The tiers with work (hn: entries per list; null: unknown, launch those that a
// plan for few launches uses).
void launch_tiers(const CountPlan &p, const int32_t *hn, int64_t items, cudaStream_t s) {
    const int sms = num_sms();
    auto has = [&](int t) {
        return hn ? hn[t] > 0 : t == CT_WARP || t == CT_DENSE256 || t == CT_HYBRID;
    };
    auto cap = [&](int t) { return hn ? (int64_t)hn[t] : items; };
    if (has(CT_DENSE512)) launch_dense<512, 4096>(p, CT_DENSE512, cap(CT_DENSE512), s);
    if (p.cta_keys > 0 && has(CT_HYBRID)) {
        int32_t headn = 0, bmw = 0;
        const size_t smem = count_cta_smem(p.cta_keys, &headn, &bmw);
        allow_max_smem((const void *)k_count_cta);
        k_count_cta<<<(unsigned)std::min<int64_t>(sms, cap(CT_HYBRID)), CTA_THREADS, smem, s>>>(p, headn, bmw);
        RC_LAUNCH();
    }
    if (has(CT_DENSE256)) launch_dense<256, 2048>(p, CT_DENSE256, cap(CT_DENSE256), s);
    if (has(CT_DENSE64)) launch_dense<64, 512>(p, CT_DENSE64, cap(CT_DENSE64), s);
    if (has(CT_HASH)) {
        const size_t hsm = count_hash_smem();
        allow_max_smem((const void *)k_count_hash);
        int occ = 1;
        RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_count_hash, HASH_THREADS, hsm));
        k_count_hash<<<(unsigned)std::min<int64_t>(sms * std::max(1, occ), cap(CT_HASH)), HASH_THREADS,
                       hsm, s>>>(p);
        RC_LAUNCH();
    }
    if (has(CT_WARP)) {
        k_count_warp<<<(unsigned)std::min<int64_t>(sms * 6, (cap(CT_WARP) + 7) / 8), 256, 0, s>>>(p);
        RC_LAUNCH();
    }
}

__global__ void k_scatter_counts(const unsigned long long *__restrict__ cnt,
                                 const int32_t *__restrict__ new2old, int32_t n,
                                 unsigned long long *__restrict__ out) {
    int32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < n) out[new2old[x]] = cnt[x];
}

// Both sides' counts to their original ids (out null: not wanted).
__global__ void k_scatter_both(const unsigned long long *__restrict__ cu,
                               const unsigned long long *__restrict__ cv,
                               const int32_t *__restrict__ nou, const int32_t *__restrict__ nov,
                               int32_t nu, int32_t nv, unsigned long long *__restrict__ ou,
                               unsigned long long *__restrict__ ov) {
    const int32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < nu) {
        if (ou) ou[nou[x]] = cu[x];
    } else if (x - nu < nv) {
        if (ov) ov[nov[x - nu]] = cv[x - nu];
    }
}

}  // namespace

// The masks pay from about 20 wedges an edge on (the passes over them cost 128
// bytes and some 80 instructions an edge, whatever the wedges), where their memory
// is not many times the graph's. Counts with / without them, ms: 10M edges on 6M
// vertices, uniform, 1.7 wedges an edge: 7.8 / 4.7; 1M on 1M, power law, 6.9: 1.24 /
// 0.81; 10M on 6.5M, 13.6: 8.1 / 7.5; 30M on 2M, 27: 21.0 / 22.2; 10M on 670,000,
// 32: 6.8 / 9.1; 10M on 2M, 51: 7.1 / 10.8.
static bool masks_pay(int64_t m, int64_t n, uint64_t walks) {
    return walks / 20 >= (uint64_t)m && (double)n * BITS / 8 <= 64.0 * (double)m + (256 << 20);
}

CountMemory count_memory(int64_t m, int64_t nu, int64_t nv, int sms) {
    const size_t n = (size_t)(nu + nv), n_max = (size_t)std::max(nu, nv);
    CountMemory b;
    // prefix lengths, tier lists (and first keys), hot counts, planes of the
    // huge start points (at most 4 m / HUGE_DEG chunks), the global tier
    b.needed = 8 * (size_t)m + 4 * (size_t)(CT_LISTS + 1) * n + 16 * (size_t)HOT_REPS * HOT_KEYS +
               4 * (size_t)m / HUGE_DEG * HUGE_NP * 128 + 8 * (size_t)sms * n_max;
    b.optional = masks_pay(m, (int64_t)n, ~0ull) ? (BITS / 8 + 4) * n : 0;
    return b;
}

// Counts butterflies of both sides into cnt_u / cnt_v (local ids, zeroed
// here). Returns wedges traversed.
uint64_t count_local(const receipt_graph *g, unsigned long long *cnt_u,
                     unsigned long long *cnt_v, cudaStream_t s, int64_t *points) {
    const int64_t m = g->m;
    RC_CUDA(cudaMemsetAsync(cnt_u, 0, sizeof(unsigned long long) * (g->nu > 0 ? g->nu : 1), s));
    RC_CUDA(cudaMemsetAsync(cnt_v, 0, sizeof(unsigned long long) * (g->nv > 0 ? g->nv : 1), s));
    if (m == 0) return 0;
    const int sms = num_sms();
    const int64_t n = (int64_t)g->nu + g->nv;
    const int32_t n_max = std::max(g->nu, g->nv);
    // counters: wedges (8 bytes), entries per list, work counters
    DevBuf<int32_t> ctr(2 + COUNT_CTRS, s);
    ctr.zero();
    DevBuf<int32_t> plen(2 * m, s), lists((size_t)CT_LISTS * n, s), base, first;
    CountPlan p{};
    p.wedges = (unsigned long long *)ctr.get();
    p.n = ctr.get() + 2;
    for (int t = 0; t < CT_LISTS; t++) p.list[t] = lists.get() + (size_t)t * n;
    // key space of a hybrid-tier start point is [0, sp): start points up to
    // the largest key space that fits in shared memory
    p.cta_keys = max_cta_keyspace(n_max, MID_CHUNK * 8 + CHUNK_BYTES);
    p.few = 0;
    // a union of packed graphs: a start point's keys begin at its graph
    const int ng = g->parts.empty() ? 0 : (int)g->parts.size() - 1;
    std::vector<int32_t> hf;
    if (ng > 1 && g->parts_o.size() == g->parts.size()) {
        for (int64_t v : g->parts) hf.push_back((int32_t)v);
        for (int64_t v : g->parts_o) hf.push_back((int32_t)v);
        first.alloc(hf.size(), s);
        base.alloc(n, s);
        RC_CUDA(cudaMemcpyAsync(first.get(), hf.data(), 4 * hf.size(), cudaMemcpyHostToDevice, s));
    }
    // masks of both sides' lists (128 bytes a vertex), unless the wedges are few
    // or there is no memory for them: then every end point is past the masks
    DevBuf<uint32_t> mask;
    DevBuf<int32_t> held;
    const bool bits =
        masks_pay(m, n, g->count_walks) && mask.try_alloc((size_t)n * 32, s) && held.try_alloc(n, s);
    if (!bits) mask.release();
    DevBuf<unsigned long long> hot;
    if (m >= HOT_MIN_M && !first.get()) {
        hot.alloc((size_t)2 * HOT_REPS * HOT_KEYS, s);
        hot.zero();
    }
    for (int A = 0; A < 2; A++) {
        const Side &SA = g->side[A];
        const Side &SB = g->side[1 - A];
        const bool rel = first.get() != nullptr;
        const bool hots = hot.get() != nullptr;
        p.s[A] = CountSide{SA.off, SA.adj, SB.off, SB.adj, SB.below, A ? cnt_v : cnt_u,
                           A ? cnt_u : cnt_v,
                           hots ? hot.get() + (size_t)A * HOT_REPS * HOT_KEYS : nullptr,
                           hots ? hot.get() + (size_t)(1 - A) * HOT_REPS * HOT_KEYS : nullptr, plen.get() + (A ? m : 0),
                           rel ? base.get() + (A ? g->nu : 0) : nullptr,
                           rel ? first.get() + (A ? ng + 1 : 0) : nullptr,
                           // masks of the middle vertices (side 1 - A)
                           bits ? mask.get() + (A ? 0 : (size_t)g->nu * 32) : nullptr,
                           bits ? held.get() + (A ? 0 : g->nu) : nullptr, SA.n, ng};
    }
    if (bits)
        for (int A = 0; A < 2; A++) {
            const Side &SB = g->side[1 - A];
            if (SB.n == 0) continue;
            const CountSide &S = p.s[A];
            k_count_masks<<<(unsigned)std::min<int64_t>(((int64_t)SB.n + 7) / 8, (int64_t)sms * 32), 256, 0,
                            s>>>(SB.off, SB.adj, SB.n, S.first ? p.s[1 - A].first : nullptr, S.first, ng,
                                 const_cast<uint32_t *>(S.mask), const_cast<int32_t *>(S.held));
            RC_LAUNCH();
        }
    launch_plan(p, n, s);
    k_count_plan_wide<<<sms * 4, 512, 0, s>>>(p);
    RC_LAUNCH();
    if (bits) {
        k_count_bits<<<(unsigned)std::min<int64_t>((n + 7) / 8, (int64_t)sms * 32), 256, 0, s>>>(p);
        RC_LAUNCH();
    }
    int32_t hn[2 + CT_LISTS];
    RC_CUDA(cudaMemcpyAsync(hn, ctr.get(), sizeof(hn), cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    const int32_t *ln = hn + 2;
    DevBuf<int32_t> hoff;
    DevBuf<uint32_t> hplanes;
    if (bits && ln[CT_HUGE] > 0) {
        // at most one chunk per start point and per HUGE_DEG edges of a side
        const int64_t chunks = ln[CT_HUGE] + 2 * m / HUGE_DEG;
        hoff.alloc((size_t)ln[CT_HUGE] + 1, s);
        hplanes.alloc((size_t)chunks * HUGE_NP * 32, s);
        p.hoff = hoff.get();
        p.hplanes = hplanes.get();
        const unsigned grid = (unsigned)std::min<int64_t>(sms * 4, chunks);
        k_huge_plan<<<1, 32, 0, s>>>(p);
        RC_LAUNCH();
        k_huge_add<<<grid, 512, 0, s>>>(p);
        RC_LAUNCH();
        k_huge_sum<<<(unsigned)std::min(sms * 32, ln[CT_HUGE]), 32, 0, s>>>(p);
        RC_LAUNCH();
        k_huge_opposite<<<grid, 512, 0, s>>>(p);
        RC_LAUNCH();
    }
    if (bits && ln[CT_BITS] > 0) {
        k_count_bits_wide<<<(unsigned)std::min(sms * 4, ln[CT_BITS]), 512, 0, s>>>(p);
        RC_LAUNCH();
    }
    launch_tiers(p, ln, n, s);
    int32_t over = 0;
    if (ln[CT_HYBRID] > 0) {
        RC_CUDA(cudaMemcpyAsync(&over, p.n + CT_OVER, 4, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
    }
    if (points) {
        points[0] += ln[CT_WARP];
        points[1] += ln[CT_HASH] + ln[CT_DENSE64];
        points[2] += ln[CT_DENSE256] + ln[CT_DENSE512] + ln[CT_HYBRID];
        points[3] += ln[CT_GLOBAL];
        points[4] += over;
    }
    if (ln[CT_GLOBAL] + over > 0) {
        const int gblocks = std::min(sms, ln[CT_GLOBAL] + over);
        DevBuf<uint32_t> gcnt((size_t)gblocks * n_max, s);
        DevBuf<int32_t> gtouch((size_t)gblocks * n_max, s);
        const size_t gsm = MID_CHUNK * 8 + CHUNK_BYTES;
        allow_max_smem((const void *)k_count_global);
        k_count_global<<<gblocks, CTA_THREADS, gsm, s>>>(p, gcnt.get(), gtouch.get(), n_max);
        RC_LAUNCH();
    }
    if (hot.get()) {
        k_count_merge<<<dim3(HOT_KEYS / 128, 2), 128, 0, s>>>(p);
        RC_LAUNCH();
    }
    unsigned long long wedges = 0;
    RC_CUDA(cudaMemcpyAsync(&wedges, p.wedges, 8, cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    return wedges;
}

void scatter_to_original(const unsigned long long *local, const int32_t *new2old, int32_t n,
                         unsigned long long *out, cudaStream_t s) {
    if (n <= 0) return;
    k_scatter_counts<<<ceil_div(n, 256), 256, 0, s>>>(local, new2old, n, out);
    RC_LAUNCH();
}

}  // namespace receipt

// ---------------------------------------------------------------------
// Butterfly counting that allocates no device memory
// ---------------------------------------------------------------------
// Every temporary of the counting pass (local counts, prefix lengths, tier
// lists, work counters and the global-tier counter slots) is carved out of
// one statically sized array in this library's device image, so the call
// makes no cudaMalloc/cudaFree and no allocating library call. The array's
// size fixes the largest graph it accepts.
namespace receipt {

namespace {

constexpr int32_t NOALLOC_MAX_SIDE = 65536;   // vertices per side
constexpr int64_t NOALLOC_MAX_M = 1 << 20;    // edges (after duplicate removal)
constexpr int NOALLOC_GSLOTS = 8;             // CTAs of the global-counter tier

constexpr size_t na_round(size_t b) { return (b + 255) & ~(size_t)255; }
constexpr size_t NA_CNT = na_round(8 * (size_t)NOALLOC_MAX_SIDE);
constexpr size_t NA_PLEN = na_round(2 * 4 * (size_t)NOALLOC_MAX_M);
constexpr size_t NA_LIST = na_round(2 * 4 * (size_t)NOALLOC_MAX_SIDE);
constexpr size_t NA_GLOB = na_round(4 * (size_t)NOALLOC_GSLOTS * NOALLOC_MAX_SIDE);
constexpr size_t NA_MISC = 256;
constexpr size_t NOALLOC_BYTES = 2 * NA_CNT + NA_PLEN + CT_LISTS * NA_LIST + 2 * NA_GLOB + NA_MISC;
static_assert(4 * (2 + COUNT_CTRS) <= NA_MISC, "counters");

// ~19 MB per device, held from module load until the process exits.
static __device__ __align__(256) unsigned char g_count_scratch[NOALLOC_BYTES];

std::mutex g_na_mu;
void *g_na_ptr[64] = {nullptr};

// Device address of the scratch array for the current device; looked up once
// per device (host code may not use the symbol itself as an address).
unsigned char *noalloc_scratch() {
    int d = 0;
    RC_CUDA(cudaGetDevice(&d));
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[d & 63]) {
        void *p = nullptr;
        RC_CUDA(cudaGetSymbolAddress(&p, g_count_scratch));
        g_na_ptr[d & 63] = p;
    }
    return (unsigned char *)g_na_ptr[d & 63];
}

}  // namespace

void count_noalloc(const receipt_graph *g, unsigned long long *d_cnt_u,
                   unsigned long long *d_cnt_v, cudaStream_t s) {
    if (g->nu > NOALLOC_MAX_SIDE || g->nv > NOALLOC_MAX_SIDE || g->m > NOALLOC_MAX_M)
        fail(RECEIPT_ERR_INVALID,
             "graph exceeds the limits of receipt_count_butterflies_noalloc (at most " +
                 std::to_string(NOALLOC_MAX_SIDE) + " vertices per side and " +
                 std::to_string(NOALLOC_MAX_M) + " edges; got " + std::to_string(g->nu) + " x " +
                 std::to_string(g->nv) + " with " + std::to_string(g->m) + " edges)");
    unsigned char *base = noalloc_scratch();
    CountPlan p{};
    p.wedges = (unsigned long long *)base;
    p.n = (int32_t *)base + 2;
    unsigned long long *cnt[2];
    cnt[0] = (unsigned long long *)(base + NA_MISC);
    cnt[1] = cnt[0] + g->nu;
    unsigned char *q = base + NA_MISC + 2 * NA_CNT;
    int32_t *plen = (int32_t *)q;
    q += NA_PLEN;
    for (int t = 0; t < CT_LISTS; t++, q += NA_LIST) p.list[t] = (int32_t *)q;
    uint32_t *gcnt = (uint32_t *)q;
    int32_t *gtouch = (int32_t *)(q + NA_GLOB);
    // the array keeps the previous call's contents: zero what must start at 0,
    // side by side at the front (the global tier clears its own counters)
    RC_CUDA(cudaMemsetAsync(base, 0, NA_MISC + 8 * ((size_t)g->nu + g->nv), s));
    const int64_t m = g->m;
    const int sms = num_sms();
    if (m > 0) {
        const int64_t n = (int64_t)g->nu + g->nv;
        const int32_t n_max = std::max(g->nu, g->nv);
        p.cta_keys = max_cta_keyspace(n_max, MID_CHUNK * 8 + CHUNK_BYTES);
        p.few = 1;
        for (int A = 0; A < 2; A++) {
            const Side &SA = g->side[A];
            const Side &SB = g->side[1 - A];
            p.s[A] = CountSide{SA.off, SA.adj, SB.off, SB.adj, SB.below, cnt[A], cnt[1 - A], nullptr,
                               nullptr, plen + (A ? m : 0), nullptr, nullptr, nullptr, nullptr, SA.n, 0};
        }
        launch_plan(p, n, s);
        k_count_plan_wide<<<sms, 512, 0, s>>>(p);
        RC_LAUNCH();
        launch_tiers(p, nullptr, n, s);
        const size_t gsm = MID_CHUNK * 8 + CHUNK_BYTES;
        allow_max_smem((const void *)k_count_global);
        k_count_global<<<NOALLOC_GSLOTS, CTA_THREADS, gsm, s>>>(p, gcnt, gtouch, n_max);
        RC_LAUNCH();
    }
    const int32_t n_all = g->nu + g->nv;
    if (n_all > 0 && (d_cnt_u || d_cnt_v)) {
        k_scatter_both<<<ceil_div(n_all, 256), 256, 0, s>>>(cnt[0], cnt[1], g->side[0].new2old,
                                                            g->side[1].new2old, g->nu, g->nv, d_cnt_u,
                                                            d_cnt_v);
        RC_LAUNCH();
    }
}

}  // namespace receipt
