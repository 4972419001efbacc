// Fine-grained decomposition, Algorithm 4 (RECEIPT FD), with the
// workload-aware scheduling of Sec. 3.2.1.
//
// Setup (all on the device):
//  * members of every subset U_i, ordered by local id; rank[x] = position of
//    x inside its subset (the key space of G_i's aggregation);
//  * the induced subgraphs G_i = (U_i, V, E_i) all at once: the other side's
//    adjacency (sorted by (y, x)) is stably sorted by sub(x), so the block of
//    subset i lists, for every y, the ranks of y's neighbours inside U_i as
//    one contiguous run; every edge (x, y) of side s records where its run
//    (sub(x), y) starts and how long it is;
//  * a task queue of subset ids in decreasing order of their wedge count
//    (Longest Processing Time first).
//
// The members' updates are aggregated before the peel, all at once, into lists
// (k_fd_pairs).
//
// Peeling: persistent CTAs pop subsets from the queue with one atomic each.
// Inside a subset the CTA runs bottom-up peeling level by level: the level
// mu = max(previous level, min support over the remaining vertices); every
// vertex whose raw support is <= mu is peeled with tip number mu, and the
// updates of Algorithm 2 restricted to G_i are applied. Peeling all
// minimum-support vertices together gives the same tip numbers as peeling
// them one at a time: max(mu, max(mu, a) - b) = max(mu, a - b) for b >= 0,
// and supports are order independent (Lemma 1).
#include <algorithm>

#include "engine.cuh"
#include "internal.cuh"

namespace receipt {

namespace {

constexpr int FD_THREADS = 512;
// dense counters of the fine-grained step: 30,720 words (61,440 16-bit keys)
constexpr int FD_WORDS = 30720;
constexpr int FD_KEYS = 2 * FD_WORDS;
// the touched-word list doubles as the window histogram between passes
using FdEngine = DenseSliceT<FD_WORDS, TOUCH_LIST>;
static_assert(TOUCH_CAP * 2 >= LOG_BUCKETS * 4, "histogram in the touched-word list");
// walk-size flag: the vertex's degree is >= 65535 (counts may need 32 bits)
constexpr unsigned long long WIDE_BIT = 1ull << 63;
// heavy tasks, automatic rule
constexpr unsigned long long HEAVY_MIN_W = 1ull << 23;
constexpr int32_t HEAVY_NI = 1 << 17;
// a level of a heavy task with at most this many members with big walks
// (and at least two CTAs for each) splits each one's walk over the CTAs
// (partial counts summed in global counters) instead of giving each member
// one CTA
constexpr int FDH_SPLIT_NB = 32;
// a task whose walk wedges reach this many times LEVEL_WEDGES per member is
// walk-bound (see the heavy rule)
constexpr unsigned long long HEAVY_WALK_LEVELS = 4;
// parts of one subset are merged into tasks of at least this many members
constexpr int32_t TASK_MIN = 8192;
// LPT weight of one member of a task in wedges. A task's time is its levels',
// 2-3 us each and at most one a member; its walks, done before the peel, tell
// tasks of as many members apart.
constexpr unsigned long long LEVEL_WEDGES = 1ull << 15;

// Sort keys: subset in the high word, vertex (or edge) in the low one.
__global__ void k_sub_keys(const int32_t *__restrict__ sub, int32_t n, uint64_t *__restrict__ key) {
    int32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < n) key[x] = ((uint64_t)(uint32_t)sub[x] << 32) | (uint32_t)x;
}

// First member position of every subset (P + 1 entries) in the sorted keys.
__global__ void k_sub_starts(const uint64_t *__restrict__ key, int32_t n, int32_t P,
                             int32_t *__restrict__ mstart) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > P) return;
    int32_t lo = 0, hi = n;
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo) / 2;
        if ((int64_t)(key[mid] >> 32) < i)
            lo = mid + 1;
        else
            hi = mid;
    }
    mstart[i] = lo;
}

__global__ void k_members(const uint64_t *__restrict__ key, int32_t n,
                          const int32_t *__restrict__ mstart, int32_t *__restrict__ members,
                          int32_t *__restrict__ rank) {
    int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) {
        const uint64_t k = key[p];
        const int32_t x = (int32_t)(uint32_t)k;
        members[p] = x;
        rank[x] = p - mstart[k >> 32];
    }
}

__global__ void k_edge_sub_keys(const int32_t *__restrict__ adj_o, int64_t m,
                                const int32_t *__restrict__ sub, uint64_t *__restrict__ key) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < m) key[k] = ((uint64_t)(uint32_t)sub[adj_o[k]] << 32) | (uint32_t)k;
}

__device__ __forceinline__ int32_t owner_of(const int64_t *off, int32_t n, int64_t q) {
    int32_t lo = 0, hi = n - 1;
    while (lo < hi) {
        int32_t mid = (lo + hi + 1) >> 1;
        if (off[mid] <= q)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// For sorted position p: y, rank, and run head flag (the position before is
// the lane before's, but for a warp's first lane).
__global__ void k_fd_fill(const uint64_t *__restrict__ key, int64_t m, const int32_t *__restrict__ adj_o,
                          const int64_t *__restrict__ off_o, int32_t n_o,
                          const int32_t *__restrict__ rank, int32_t *__restrict__ fd_adj,
                          int32_t *__restrict__ fd_y, uint32_t *__restrict__ head) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t k = p < m ? key[p] : 0;
    const int32_t y = p < m ? owner_of(off_o, n_o, (int64_t)(uint32_t)k) : 0;
    int32_t sub = (int32_t)(k >> 32);
    int32_t y1 = __shfl_up_sync(0xffffffffu, y, 1), sub1 = __shfl_up_sync(0xffffffffu, sub, 1);
    if (p >= m) return;
    if ((threadIdx.x & 31) == 0 && p > 0) {
        const uint64_t k1 = key[p - 1];
        y1 = owner_of(off_o, n_o, (int64_t)(uint32_t)k1);
        sub1 = (int32_t)(k1 >> 32);
    }
    fd_adj[p] = rank[adj_o[(uint32_t)k]];
    fd_y[p] = y;
    head[p] = p == 0 || sub1 != sub || y1 != y ? 1u : 0u;
}

__global__ void k_run_starts(const uint32_t *__restrict__ head, const uint32_t *__restrict__ hpos,
                             int64_t m, int64_t *__restrict__ run_start) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < m && head[p]) run_start[hpos[p]] = p;
}

// Run of every side-s edge (x, y).
__global__ void k_fd_edges(const uint64_t *__restrict__ key, int64_t m,
                           const int32_t *__restrict__ adj_o, const int32_t *__restrict__ fd_y,
                           const uint32_t *__restrict__ head, const uint32_t *__restrict__ hpos,
                           const int64_t *__restrict__ run_start, int64_t nruns,
                           const int64_t *__restrict__ off_s, const int32_t *__restrict__ adj_s,
                           int64_t *__restrict__ fd_beg, int32_t *__restrict__ fd_len) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= m) return;
    int64_t r = (int64_t)hpos[p] + head[p] - 1;  // run id
    int64_t rs = run_start[r];
    int64_t re = r + 1 < nruns ? run_start[r + 1] : m;
    int32_t x = adj_o[(uint32_t)key[p]];
    int32_t y = fd_y[p];
    int64_t b = off_s[x];
    int64_t ps = b + lower_bound_i32(adj_s + b, off_s[x + 1] - b, y);
    fd_beg[ps] = rs;
    fd_len[ps] = (int32_t)(re - rs);
}

__global__ void k_i32_to_i64(const int32_t *__restrict__ v, int64_t m, int64_t *__restrict__ out) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < m) out[q] = v[q];
}

// A member's edges and its walk size inside G_i, by member position.
struct alignas(16) FdMember {
    int64_t q0;
    int32_t deg;
    uint32_t w;  // saturated
};

// Walk size inside G_i of every vertex (sum of its edges' run lengths, from
// the prefix sums `pre`), stored at its member position; WIDE_BIT marks a
// degree >= 65535 (counts may need 32 bits), wide[] its subset.
__global__ void k_fd_walk_sizes(const int64_t *__restrict__ off_s, int32_t n,
                                const int64_t *__restrict__ pre, const int32_t *__restrict__ sub,
                                const int32_t *__restrict__ mstart, const int32_t *__restrict__ rank,
                                unsigned long long *__restrict__ wr, FdMember *__restrict__ info,
                                int32_t *__restrict__ wide) {
    int32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const int64_t q0 = off_s[x], q1 = off_s[x + 1];
    const unsigned long long W = (unsigned long long)(pre[q1] - pre[q0]);
    const int32_t p = mstart[sub[x]] + rank[x];
    wr[p] = W | (q1 - q0 >= 65535 ? WIDE_BIT : 0ull);
    info[p] = FdMember{q0, (int32_t)(q1 - q0), (uint32_t)(W < 0xffffffffull ? W : 0xffffffffull)};
    if (q1 - q0 >= 65535) wide[sub[x]] = 1;
}

// Task boundaries: the first member of every subset and, when the side is a
// union of packed graphs (parts = first vertex of each graph), every member
// whose graph differs from the previous member's.
__global__ void k_task_flags(const int32_t *__restrict__ members, int32_t n,
                             const int32_t *__restrict__ sub, const int32_t *__restrict__ mstart,
                             const int64_t *__restrict__ parts, int ng,
                             uint32_t *__restrict__ flag) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int32_t x = members[p];
    uint32_t f = p == mstart[sub[x]] ? 1u : 0u;
    if (!f && ng > 0) {
        auto graph_of = [&](int64_t v) {
            int lo = 0, hi = ng - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (parts[mid] <= v)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            return lo;
        };
        f = graph_of(x) != graph_of(members[p - 1]) ? 1u : 0u;
    }
    flag[p] = f;
}

__global__ void k_flag_positions(const uint32_t *__restrict__ flag, const uint32_t *__restrict__ pos,
                                 int32_t n, int32_t *__restrict__ out) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n && flag[p]) out[pos[p]] = p;
}

// a member's cost: its wedges and a constant; and each subset's wedge count,
// the sum of L (L - 1) over its runs L (a member's walk counts itself once per
// edge)
__global__ void k_walk_cost(const unsigned long long *__restrict__ wr, int32_t n, int64_t add,
                            const FdMember *__restrict__ info, const int32_t *__restrict__ members,
                            const int32_t *__restrict__ sub, int64_t *__restrict__ out,
                            unsigned long long *__restrict__ wsub) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = p < n;
    const unsigned long long w = in ? wr[p] & ~WIDE_BIT : 0;
    const unsigned long long others = in && w ? w - (unsigned)info[p].deg : 0;
    const int32_t sb = in ? sub[members[p]] : -1;
    if (in) out[p] = (int64_t)w + add;
    // members of one subset are together
    const int32_t s0 = __shfl_sync(0xffffffffu, sb, 0);
    if (__all_sync(0xffffffffu, sb == s0 || sb < 0)) {
        const unsigned long long t = warp_sum(others);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(&wsub[s0], t);
    } else if (others) {
        atomicAdd(&wsub[sb], others);
    }
}

__global__ void k_task_weights(const int32_t *__restrict__ tstart, const int32_t *__restrict__ tlen,
                               const int64_t *__restrict__ cw, int64_t add, int32_t T,
                               unsigned long long *__restrict__ w) {
    const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < T)
        w[t] = (unsigned long long)(cw[tstart[t] + tlen[t]] - cw[tstart[t]] - add * tlen[t]);
}

// ------------------------------------------------------------------------
// Tasks that one CTA hands over to all of them
//
// On graphs whose vertices are much alike (uniform ones, members of the same
// hubs) a task's levels peel a few members each until one sets off the next, and
// three to ten levels peel nearly all: 150 levels of 860 members, then 2,059 and
// 1,743 with lists of 4,650 entries. A CTA applies an entry in 0.85 ns (17 ms); all
// CTAs take ~70 us a level and 3.3 ps a wedge. When a level's lists cost more than
// that, the hand-over (~0.6 ms) and what was handed over before (one after the
// other), the CTA leaves the task as it was before the level, and it is peeled on
// as a heavy task. Levels of power-law graphs stay far below (no level of 150,000
// entries in tasks of 10M and 40M edges; the line is ~800,000).
// Step by one CTA / handed over / heavy from the start, ms: 3.9M uniform edges,
// 4,660 members 19.3 / 7.8 / 11.4; 20M, 30,000 members 327 / 91 / 114; 3M, 10,000
// members 45 / 15 / 27; 1.5M power-law edges with a hub of degree 125,000 in 245
// tasks 185 / 45 / 86; 1.7M uniform, 35,400 members 10.9 / 8.2 / 6.3.
// ------------------------------------------------------------------------
struct FdHandOver {
    const unsigned long long *tw;  // per task: wedges (null: no task is handed over)
    int32_t *count;                // [0]: tasks handed over or, for a moment, refused;
    int32_t *list;                 // [1]: handed over; their ids
    unsigned long long *level;     // per task: its level then
};
constexpr float FD_HAND_OVER_NS = 6e5f;

// ns of one peeled member of a task of n: from its list (entries: all lists'), as
// a heavy task
__device__ __forceinline__ float2 fd_member_ns(unsigned long long entries, unsigned long long w,
                                               int32_t n) {
    return make_float2(0.85f * (float)entries / (float)n, 0.0033f * (float)w / (float)n);
}
// Members of a level from which on it may pay.
__device__ __forceinline__ int fd_hand_over_from(float2 ns) {
    const float gain = ns.x - ns.y;
    return gain > 0.f ? (int)fminf(2e9f, (FD_HAND_OVER_NS + 70000.f) / gain) + 1 : INT32_MAX;
}
// Whether a level of np members is (one thread).
__device__ __forceinline__ bool fd_hand_over(const FdHandOver &h, float2 ns, int np, int32_t task,
                                             unsigned long long level) {
    const int before = atomicAdd(h.count, 1);
    const float cost = FD_HAND_OVER_NS + 70000.f + ns.y * (float)np;
    if (ns.x * (float)np <= (float)(before + 1) * cost) {
        atomicSub(h.count, 1);
        return false;
    }
    h.list[atomicAdd(h.count + 1, 1)] = task;
    h.level[task] = level;
    return true;
}

struct FdArgs {
    const int32_t *queue;      // task ids, LPT order
    int32_t P;                 // tasks
    int32_t *qhead;
    const int32_t *tstart;     // per task: first member position
    const int32_t *tlen;       // per task: members
    const int32_t *tkb;        // per task: rank of its first member inside its subset
    const int32_t *members;
    const int64_t *fd_beg;
    const int32_t *fd_len;
    const int32_t *fd_adj;
    const int32_t *new2old;
    const unsigned long long *init;
    unsigned long long *fsup;  // by member position
    uint8_t *alive;            // by member position
    int32_t *alist;            // by member position: alive members outside the window (two buffers)
    int32_t *alist2;
    int32_t *clist;            // by member position: members inside the window (two buffers)
    int32_t *clist2;
    int32_t *plist;            // by member position
    const FdMember *info;      // by member position
    const uint32_t *pool;      // the members' lists, and where each lies
    const unsigned long long *rec;
    unsigned long long *tip;   // output, original ids
    unsigned long long *stats; // [0] wedges, [1] levels
    unsigned long long *sub_ns;     // per task: nanoseconds spent
    unsigned long long *sub_levels; // per task: peeling levels
    FdHandOver ho;
};

struct FdMids {
    static constexpr bool LARGE_FIRST = false;
    const int64_t *fd_beg;
    const int32_t *fd_len;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        beg = fd_beg[q];
        len = fd_len[q];
    }
};

// Support decrement of an alive member. Values below the window bound T
// also lower *mn, so that after a level's updates *mn holds the minimum
// support of the window's survivors (together with the minimum of the
// untouched ones, taken when the level's peeled vertices are selected); a
// member whose support falls below T here joins the window's list.
struct FdEmit {
    unsigned long long *fsup;  // subset base
    const uint8_t *alive;      // subset base
    unsigned long long *mn;    // next level's minimum (shared or global)
    unsigned long long T;      // window bound (~0: everything is inside)
    int32_t *cand;             // window list (null without a window)
    int *n_cand;
    __device__ __forceinline__ void operator()(int32_t k, uint32_t c) {
        if (alive[k]) {
            const unsigned long long d = choose2(c);
            const unsigned long long old = atomicAdd(&fsup[k], 0ull - d);
            const unsigned long long nv = old - d;
            if (nv < T) {
                atomicMin(mn, nv);
                if (old >= T) cand[atomicAdd(n_cand, 1)] = k;
            }
        }
    }
    // N pairs at once (k < 0: none): all `alive` loads, then all support
    // atomics, then the bookkeeping, so their latencies overlap.
    template <int N>
    __device__ __forceinline__ void many(const int32_t (&k)[N], const uint32_t (&c)[N]) {
        bool al[N];
#pragma unroll
        for (int u = 0; u < N; u++) al[u] = k[u] >= 0 && alive[k[u]];
        unsigned long long old[N], d[N];
#pragma unroll
        for (int u = 0; u < N; u++) {
            d[u] = choose2(c[u]);
            old[u] = al[u] ? atomicAdd(&fsup[k[u]], 0ull - d[u]) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < N; u++) {
            if (!al[u]) continue;
            const unsigned long long nv = old[u] - d[u];
            if (nv < T) {
                atomicMin(mn, nv);
                if (old[u] >= T) cand[atomicAdd(n_cand, 1)] = k[u];
            }
        }
    }
};

// ------------------------------------------------------------------------
// Every member's updates, before the peel
//
// What peeling a member r takes from the others of its subset depends only on
// how many middle vertices they share, not on when r is peeled: C(c, 2) for
// each member sharing c >= 2. So the walks of all members are done first, by
// the whole chip and in any order, and leave each member a list of (rank,
// count) entries; a level of the peel, a chain of dependent steps on one SM,
// then reads a list instead of walking (runs, keys, counters, sweep).
//
// Walks have 100 to 2,000 wedges over about ten middle vertices in the tasks
// that take longest, and up to a million in the last ones: each is counted by
// a group of warps (FpPlan). Members whose counters exceed a CTA's words up to
// 8 times walk once per slice of them.
// The entries lie in one pool, taken by each group in blocks; a member whose
// list does not fit it, or that is too large for all this, has no list and
// walks when it is peeled.
// Two CTAs of 16 warps an SM: bound by instruction issue (60% of the slots, the
// rest mostly fixed-latency waits and group barriers; DRAM under 1%).
// 1.93e9 wedges of a 40M-edge graph in 9.1 ms, 3.9e8 of a 10M-edge graph in 3.0
// ms; walked during the peel they made the whole step 101 and 26 ms (34 and 10
// now).
// ------------------------------------------------------------------------
constexpr int FP_THREADS = FP_WARPS * 32;
constexpr int FP_BLOCK = 1024;           // pool entries taken at a time
constexpr int64_t FP_MEMBER_COST = 128;  // a member's fixed cost in wedges
// An entry holds the rank in its low fp_rank_bits and the count above.
constexpr unsigned long long FP_NONE = ~0ull;  // no list; else offset << 24 | length

// Pool entries that the lists of n members of w wedges will take, about: where
// two members share c = w / n^2 << 1 middle vertices on average, c^2 / 2 for each
// two (uniform graphs; power-law ones have half of that), at least a twelfth of
// the wedges (tasks of very unlike members: 300,000 members of all degrees, c =
// 0.03, a sixteenth), at most a third; more by the ends of blocks that stay unused.
// With lists_at_most as a bound, the tasks of whole graphs of 1M to 40M edges,
// uniform, dense and power law, had 0.5 to 1.0 of this in entries.
inline unsigned long long lists_about(unsigned long long w, int32_t n) {
    const double c = (double)w / ((double)n * (double)n);
    const double e = (double)w * std::min(1.0 / 3, std::max(1.0 / 12, c / 2));
    const double len = e / n;
    return (unsigned long long)(len < FP_BLOCK ? e * (1.0 + len / FP_BLOCK) : e);
}

// Pool entries of the lists of n vertices of w wedges together, at most: one for
// two wedges, one for each other vertex (twice that where a block's end may stay
// unused because the next list is longer).
inline unsigned long long lists_at_most(unsigned long long w, int32_t n) {
    const unsigned long long pairs = (unsigned long long)n * (unsigned long long)n;
    return std::min(w / 2, n < 2 * FP_BLOCK ? 2 * pairs : pairs);
}

struct FdPairArgs {
    const int32_t *tstart, *tlen, *tkb;
    const uint8_t *tskip;     // tasks without lists
    int32_t T;
    const int32_t *item_p;    // per item: first member position (nitems + 1)
    int32_t nitems;
    int32_t *qhead;
    const FdMember *info;     // by member position
    const int32_t *keys;      // the runs' keys
    uint32_t *pool;
    unsigned long long cap;   // entries
    unsigned long long *head;
    unsigned long long *rec;  // by member position
    unsigned long long *wedges;
};

// First member position of every item of Q cost units (cw: prefix costs).
__global__ void k_pair_items(const int64_t *__restrict__ cw, int32_t n, int64_t Q, int32_t nitems,
                             int32_t *__restrict__ item_p) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > nitems) return;
    int32_t lo = 0, hi = n;
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo) / 2;
        if (cw[mid] < (int64_t)i * Q)
            lo = mid + 1;
        else
            hi = mid;
    }
    item_p[i] = i == nitems ? n : lo;
}

__device__ __forceinline__ FdMember fd_load(const FdMember *p) {
    const int4 q = __ldg((const int4 *)p);
    return FdMember{(int64_t)(uint32_t)q.x | ((int64_t)q.y << 32), q.z, (uint32_t)q.w};
}

// A member's plan in a task of ni; g above FP_WARPS: no list.
__device__ __forceinline__ FpPlan fd_plan(const FdMember &m, int32_t ni) {
    FpPlan p = fp_plan(m.deg, m.w, ni);
    if ((int64_t)m.deg >= 1ll << (32 - fp_rank_bits(ni))) p.g = 2 * FP_WARPS;
    return p;
}

// Weight of each task's members that get no list.
__global__ void k_listless(const FdMember *__restrict__ info, int32_t n,
                           const int32_t *__restrict__ tstart, const int32_t *__restrict__ tlen,
                           int32_t T, int32_t ni_max, unsigned long long *__restrict__ lw) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const FdMember m = fd_load(info + p);
    if (ni_max <= FP_MAX_NI && fd_plan(m, ni_max).g <= FP_WARPS) return;
    int32_t t = 0;
    for (int32_t hi = T - 1; t < hi;) {
        const int32_t mid = (t + hi + 1) / 2;
        if (tstart[mid] <= p)
            t = mid;
        else
            hi = mid - 1;
    }
    if (tlen[t] > FP_MAX_NI || fd_plan(m, tlen[t]).g > FP_WARPS)
        atomicAdd(&lw[t], (unsigned long long)m.w);
}

template <class Mids>
__global__ void __launch_bounds__(FP_THREADS, 2) k_fd_pairs(FdPairArgs a, Mids M) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_item;
    __shared__ int s_cnt[FP_WARPS];                  // entries found by each warp
    __shared__ unsigned long long s_off[FP_WARPS];   // by group: where its list lies
    uint32_t *tab = (uint32_t *)smem;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < FP_WARPS * FP_WORDS / 4; j += FP_THREADS)
        ((uint4 *)tab)[j] = make_uint4(0, 0, 0, 0);
    unsigned long long wedges = 0;             // lane 0
    unsigned long long blk = 0, blk_end = 0;   // lane 0: this warp's pool block
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(a.qhead, 1);
        __syncthreads();
        if (s_item >= a.nitems) break;
        // the largest walks first: last in a task's order, first in a side's
        const int it = Mids::LARGE_FIRST ? s_item : a.nitems - 1 - s_item;
        const int32_t p0 = a.item_p[it], p1 = a.item_p[it + 1];
        // last task starting at or before p0
        int32_t t = 0;
        for (int32_t hi = a.T - 1; t < hi;) {
            const int32_t mid = (t + hi + 1) / 2;
            if (a.tstart[mid] <= p0)
                t = mid;
            else
                hi = mid - 1;
        }
        for (; t < a.T && a.tstart[t] < p1; t++) {
            const int32_t ts = a.tstart[t], ni = a.tlen[t], kb = a.tkb[t];
            if (a.tskip[t] || ni > FP_MAX_NI) continue;
            const int32_t pa = max(p0, ts), pb = min(p1, ts + ni);
            const int rb = fp_rank_bits(ni);
            for (int g = 1; g <= FP_WARPS; g *= 2) {
                const int grp = warp / g, part = warp & (g - 1);
                uint32_t *w = tab + grp * g * FP_WORDS;
                bool more = false;
                for (int32_t p = pa + grp; p < pb; p += FP_WARPS / g) {
                    const FdMember m = fd_load(a.info + p);
                    const FpPlan pl = fd_plan(m, ni);
                    if (pl.g != g) {
                        more |= pl.g > g && pl.g <= FP_WARPS;
                        continue;
                    }
                    if (m.w == 0) {
                        if (part == 0 && lane == 0) a.rec[p] = 0;
                        continue;
                    }
                    const int32_t self = p - ts;
                    const int slices = pl.lw > 14 ? 1 << (pl.lw - 14) : 1;
                    const uint32_t wmask = (1u << min(pl.lw, 14)) - 1u;
                    unsigned long long off = 0;  // lane 0 of part 0: where the next slice's entries go
                    unsigned found = 0;          // ... and those before
                    for (int sc = 0; sc < slices; sc++) {
                        if (pl.bits) {
                            auto add = [&](int32_t key) {
                                const int32_t k = key - kb;
                                if (k == self) return;
                                if (slices > 1 && ((k >> 14) & (slices - 1)) != sc) return;
                                atomicAdd(&w[k & wmask], 1u << ((k >> pl.lw) * pl.bits));
                            };
                            warp_walk<4>(M, m.q0, m.q0 + m.deg, a.keys, add, part, g);
                        } else {
                            auto add = [&](int32_t key) {
                                const int32_t k = key - kb;
                                if (k != self) fp_table_add(w, wmask, k);
                            };
                            warp_walk<4>(M, m.q0, m.q0 + m.deg, a.keys, add, part, g);
                        }
                        fp_sync(grp, g);
                        // entries in words 4 sl .. 4 sl + 3 of this lane
                        int cnt = 0;
                        for (uint32_t sl = part * 32 + lane; sl <= wmask / 4; sl += 32 * g) {
                            const uint4 v = ((const uint4 *)w)[sl];
                            if (!(v.x | v.y | v.z | v.w)) continue;
                            const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int x = 0; x < 4; x++)
                                cnt += pl.bits ? __popc(fp_repeats(e[x], pl.bits))
                                               : (e[x] & 1023u) >= 2;
                        }
                        int inc = cnt;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int y = __shfl_up_sync(0xffffffffu, inc, o);
                            if (lane >= o) inc += y;
                        }
                        const int wtot = __shfl_sync(0xffffffffu, inc, 31);
                        int before = 0, total = wtot;
                        if (g > 1) {
                            if (lane == 0) s_cnt[warp] = wtot;
                            fp_sync(grp, g);
                            const int c = lane < g ? s_cnt[grp * g + lane] : 0;
                            total = __reduce_add_sync(0xffffffffu, c);
                            before = __reduce_add_sync(0xffffffffu, lane < part ? c : 0);
                        }
                        unsigned long long dst = 0;
                        if (part == 0 && lane == 0) {
                            if (sc == 0) {
                                // room for the list: its length, or with more
                                // slices to come the most it can be
                                const unsigned long long room =
                                    slices == 1 ? (unsigned)total : min(m.w / 2, (uint32_t)ni);
                                if (blk + room > blk_end) {
                                    const unsigned long long take =
                                        max((unsigned long long)FP_BLOCK, slices == 1 ? room : 16 * room);
                                    blk = atomicAdd(a.head, take);
                                    blk_end = blk + take;
                                }
                                off = blk_end <= a.cap ? blk : FP_NONE;
                            }
                            dst = off == FP_NONE ? FP_NONE : off + found;
                            found += total;
                            if (g > 1) s_off[grp] = dst;
                            if (sc == slices - 1) {
                                a.rec[p] = off == FP_NONE ? FP_NONE : (off << 24) | found;
                                blk += found;
                                wedges += (unsigned long long)m.w * slices;
                            }
                        }
                        if (g > 1) {
                            fp_sync(grp, g);
                            dst = s_off[grp];
                        } else {
                            dst = __shfl_sync(0xffffffffu, dst, 0);
                        }
                        uint32_t *out = a.pool + dst + before + (inc - cnt);
                        for (uint32_t sl = part * 32 + lane; sl <= wmask / 4; sl += 32 * g) {
                            const uint4 v = ((const uint4 *)w)[sl];
                            if (!(v.x | v.y | v.z | v.w)) continue;
                            ((uint4 *)w)[sl] = make_uint4(0, 0, 0, 0);
                            if (dst == FP_NONE) continue;
                            const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int x = 0; x < 4; x++) {
                                if (pl.bits == 0) {
                                    const uint32_t c = e[x] & 1023u;
                                    if (c >= 2) *out++ = ((e[x] >> 10) - 1u) | (c << rb);
                                    continue;
                                }
                                const uint32_t k0 = ((uint32_t)sc << 14) + 4 * sl + x;
                                for (uint32_t f = fp_repeats(e[x], pl.bits); f; f &= f - 1) {
                                    const int b = __ffs(f) - 1;
                                    const uint32_t c = (e[x] >> b) & (0xffffffffu >> (32 - pl.bits));
                                    *out++ = (k0 + ((uint32_t)(b / pl.bits) << pl.lw)) | (c << rb);
                                }
                            }
                        }
                        fp_sync(grp, g);
                    }
                }
                if (!__syncthreads_or(more)) break;
            }
        }
    }
    if (lane == 0 && wedges) atomicAdd(a.wedges, wedges);
}

// The listed updates of one level's np members (list: ranks in the task; rec:
// the task's records). Up to 16 members get a group of warps each, the widest
// groups there are enough of. More members go in blocks of up to 32 to the
// warps, whose lanes take a block's entries as one list: with a warp a member
// the short lists of wide levels cost a chain of loads each (uniform graphs of
// 1M and 5M edges, a few levels: the step took 2.9 and 3.7 ms, 1.3 and 1.8 so).
// Members without a list are returned in list[0, n). All threads, after a
// barrier; ends with one.
constexpr int FD_WARPS = FD_THREADS / 32;
template <class List, class Emit>
__device__ __forceinline__ int fd_lists(const uint32_t *__restrict__ pool,
                                        const unsigned long long *__restrict__ rec, List *list,
                                        int np, int rb, Emit &emit, int *s_nbig) {
    constexpr uint32_t MARK = 1u << (8 * sizeof(List) - 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t rmask = (1u << rb) - 1u;
    bool left = false;
    auto apply = [&](const uint32_t (&v)[4]) {  // entries, 0: none
        int32_t k[4];
        uint32_t c[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            c[u] = v[u] >> rb;
            k[u] = c[u] ? (int32_t)(v[u] & rmask) : -1;
        }
        emit.template many<4>(k, c);
    };
    if (np <= FD_WARPS) {
        const int g = np > 0 ? FD_WARPS >> (32 - __clz(np - 1)) : FD_WARPS;
        const int pi = warp / g, part = warp & (g - 1);
        if (pi < np) {
            const uint32_t r = (uint32_t)list[pi] & ~MARK;
            const unsigned long long q = __ldg(rec + r);
            const uint32_t *e = pool + (q >> 24);
            const int len = q == FP_NONE ? 0 : (int)(q & 0xffffffu);
            if (q == FP_NONE) {
                if (part == 0 && lane == 0) list[pi] = (List)(r | MARK);
                left = true;
            }
            for (int j0 = part * 32 + lane; j0 < len; j0 += 128 * g) {
                uint32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int j = j0 + u * 32 * g;
                    v[u] = j < len ? __ldg(e + j) : 0u;
                }
                apply(v);
            }
        }
    } else {
        const int bs = min(32, (np + FD_WARPS - 1) / FD_WARPS);
        for (int base = warp * bs; base < np; base += FD_WARPS * bs) {
            const bool in = lane < bs && base + lane < np;
            const uint32_t r = in ? (uint32_t)list[base + lane] & ~MARK : 0u;
            const unsigned long long q = in ? __ldg(rec + r) : 0ull;
            if (q == FP_NONE) {
                list[base + lane] = (List)(r | MARK);
                left = true;
            }
            const int len = q == FP_NONE ? 0 : (int)(q & 0xffffffu);
            int inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            const int total = __shfl_sync(0xffffffffu, inc, 31), ex = inc - len;
            for (int j0 = lane; j0 - lane < total; j0 += 128) {
                uint32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int j = j0 + u * 32;
                    int lo = 0;  // last lane whose list starts at or before j
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(0xffffffffu, ex, lo + step) <= j) lo += step;
                    const unsigned long long b = __shfl_sync(0xffffffffu, q >> 24, lo);
                    const int e0 = __shfl_sync(0xffffffffu, ex, lo);
                    v[u] = j < total ? __ldg(pool + b + (j - e0)) : 0u;
                }
                apply(v);
            }
        }
    }
    if (!__syncthreads_or(left)) return 0;
    // gather the marked: entries move to lower places only, each after the
    // barrier behind its own read
    for (int base = 0; base < np; base += FD_THREADS) {
        const int j = base + threadIdx.x;
        const uint32_t r = j < np ? (uint32_t)list[j] : 0u;
        const unsigned bal = __ballot_sync(0xffffffffu, (r & MARK) != 0);
        __syncthreads();
        if (bal) {
            int pos = 0;
            if (lane == 0) pos = atomicAdd(s_nbig, __popc(bal));
            pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(bal & lanemask_lt());
            if (r & MARK) list[pos] = (List)(r ^ MARK);
        }
    }
    __syncthreads();
    np = *s_nbig;
    __syncthreads();
    if (threadIdx.x == 0) *s_nbig = 0;
    __syncthreads();
    return np;
}

// Ranks of one slice [base, end) of the subset's rank space: the run of a
// middle vertex is sorted by rank, so the slice is a sub-run found by two
// binary searches.
struct FdSliceMids {
    const int64_t *fd_beg;
    const int32_t *fd_len;
    const int32_t *fd_adj;
    int32_t base, end;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        const int64_t b = fd_beg[q];
        const int32_t l = fd_len[q];
        const int64_t lo = lower_bound_i32(fd_adj + b, l, base);
        const int64_t hi = lo + lower_bound_i32(fd_adj + b + lo, l - lo, end);
        beg = b + lo;
        len = (int32_t)(hi - lo);
    }
};

// Keys of a run are ranks inside the subset; a task covering the subset's
// ranks [kb, kb + ni) sees them shifted by kb.
struct FdSliceVisit {
    FdEngine *eng;
    int32_t base;  // first rank of the slice (subset ranks)
    int32_t self;  // the anchor's own rank (subset ranks)
    __device__ __forceinline__ void operator()(int, int32_t key) {
        if (key != self) eng->add(key - base);
    }
};

struct FdSliceEmit {
    FdEmit *e;
    int32_t base;
    template <int N>
    __device__ __forceinline__ void many(const int32_t (&k)[N], const uint32_t (&c)[N]) {
        int32_t kk[N];
#pragma unroll
        for (int u = 0; u < N; u++) kk[u] = k[u] >= 0 ? k[u] + base : -1;
        e->template many<N>(kk, c);
    }
};

// window of the level loop: about max(MIN, min(MAX, alive / 32)) members
constexpr int FD_WINDOW_MIN = 512;
constexpr int FD_WINDOW_MAX = 4096;

// Update of one peeled member r (anchor x, edges [q0, q1) of side s) whose
// walk has at most WARP_MAX_W wedges: one warp with its private table.
__device__ __forceinline__ void fd_update_warp(WarpHash &WH, const FdMids &M,
                                               const int32_t *__restrict__ fd_adj, int64_t q0,
                                               int64_t q1, int32_t r, int32_t kb, int lane,
                                               FdEmit &emit) {
    auto add = [&](int32_t key) {
        const int32_t k = key - kb;
        if (k != r) WH.add(k);
    };
    warp_walk<4>(M, q0, q1, fd_adj, add);
    __syncwarp();
    WH.flush_clear(emit, lane);
    __syncwarp();
}

// Update of one peeled member r with a bigger walk: the whole CTA aggregates
// slice by slice of the subset's rank space (ni ranks) with dense counters,
// 32-bit ones when the anchor's degree lets a count reach 2^16. Returns the
// wedges walked (the same value in every thread). All threads must call it.
// What a CTA does with one aggregated slice: apply the member's updates
// (count c of a key -> support decrement C(c, 2)) ...
struct FdSweepOut {
    FdEmit *emit;
    __device__ __forceinline__ void slice(FdEngine &H, int32_t base) {
        FdSliceEmit em{emit, base};
        H.sweep<true, true>(em);
    }
};

// ... or add its partial counts (the walk of part of the member's middle
// vertices) to global counters over the task's ranks, listing each key the
// first time its counter leaves 0; the slice is cleared either way.
struct FdPartialOut {
    uint32_t *gcnt;  // ni counters of this member
    int32_t *gtl;    // keys with a non-zero counter
    int32_t *gnt;    // their number
    __device__ __forceinline__ void add(int32_t z, uint32_t c) {
        if (atomicAdd(&gcnt[z], c) == 0u) gtl[atomicAdd(gnt, 1)] = z;
    }
    __device__ __forceinline__ void slice(FdEngine &H, int32_t base) {
        const int nt = *(volatile int *)H.s_nt;
        const bool listed = nt <= FdEngine::TCAP;
        const int n = listed ? nt : H.hw;  // touched words, or every word of the slice
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int w = listed ? (int)H.tl[i] : i;
            const uint32_t v = H.cnt[w];
            if (v == 0u) continue;
            H.cnt[w] = 0u;
            if (H.wide) {
                add(base + w, v);
            } else {
                if (v & 0xffffu) add(base + w, v & 0xffffu);
                if (v >> 16) add(base + w + H.hw, v >> 16);
            }
        }
    }
};

// Part of a member's walk: the runs of its edges [q0, q1) with the first run
// taken from position `skip` on and the last one up to position `keep`
// (split heavy levels cut a walk into equal wedge shares), optionally only
// the ranks of one slice [base, end) of each.
struct FdClipMids {
    const int64_t *fd_beg;
    const int32_t *fd_len;
    const int32_t *fd_adj;
    int64_t qa, ql;       // first and last edge
    int32_t skip, keep;
    int32_t base, end;
    bool sliced;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        const int64_t b = fd_beg[q];
        const int32_t s0 = q == qa ? skip : 0;
        const int32_t e0 = q == ql ? keep : fd_len[q];
        if (sliced) {
            const int64_t lo = s0 + lower_bound_i32(fd_adj + b + s0, e0 - s0, base);
            const int64_t hi = lo + lower_bound_i32(fd_adj + b + lo, e0 - lo, end);
            beg = b + lo;
            len = (int32_t)(hi - lo);
        } else {
            beg = b + s0;
            len = e0 - s0;
        }
    }
};

// keep < 0: the last run whole (no cut).
template <class Out>
__device__ int64_t fd_update_cta(FdEngine &H, Chunk &ch, const int64_t *__restrict__ fd_beg,
                                 const int32_t *__restrict__ fd_len,
                                 const int32_t *__restrict__ fd_adj, int64_t q0, int64_t q1,
                                 int32_t r, int32_t ni, int32_t kb, Out &out, int32_t skip = 0,
                                 int32_t keep = -1) {
    const bool clip = skip != 0 || keep >= 0;
    if (clip && keep < 0) keep = fd_len[q1 - 1];
    const bool wide = q1 - q0 >= 65535;
    const int32_t SWk = wide ? FD_WORDS : FD_KEYS;
    const int32_t C = (ni + SWk - 1) / SWk;
    // only the slices that meet the anchor's rank window (first and last
    // entries of its runs, which are sorted by rank)
    int32_t j0 = 0, j1 = C - 1;
    if (C > 1) {
        int32_t *win = ch.tmp;  // scan scratch, idle here
        if (threadIdx.x == 0) {
            win[0] = INT32_MAX;
            win[1] = -1;
        }
        __syncthreads();
        int32_t lo = INT32_MAX, hi = -1;
        for (int64_t q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
            const int32_t l = fd_len[q];
            if (l > 0) {
                const int64_t b = fd_beg[q];
                lo = min(lo, fd_adj[b]);
                hi = max(hi, fd_adj[b + l - 1]);
            }
        }
        lo = warp_min(lo);
        hi = -warp_min(-hi);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&win[0], lo);
            atomicMax(&win[1], hi);
        }
        __syncthreads();
        const int32_t wlo = win[0], whi = win[1];
        __syncthreads();  // win is rewritten by the next call
        if (whi < 0) return 0;  // no runs
        j0 = (wlo - kb) / SWk;
        j1 = (whi - kb) / SWk;
    }
    int64_t wedges = 0;
    for (int32_t j = j0; j <= j1; j++) {
        const int32_t base = j * SWk;
        const int32_t w = (int32_t)imin64(SWk, (int64_t)ni - base);
        H.set_width(w, wide);
        FdSliceVisit v{&H, base + kb, r + kb};
        int64_t walked;
        if (clip) {
            FdClipMids MC{fd_beg, fd_len, fd_adj, q0,       q1 - 1,  skip,
                          keep,   base + kb, base + kb + w, j0 != j1};
            walked = cta_walk(MC, q0, q1, fd_adj, ch, v);
        } else if (j0 == j1) {
            FdMids M{fd_beg, fd_len};
            walked = cta_walk(M, q0, q1, fd_adj, ch, v);
        } else {
            FdSliceMids MS{fd_beg, fd_len, fd_adj, base + kb, base + kb + w};
            walked = cta_walk(MS, q0, q1, fd_adj, ch, v);
        }
        wedges += walked;
        if (walked == 0) continue;
        out.slice(H, base);
        __syncthreads();
        H.reset_scalars();
    }
    return wedges;
}

__device__ __forceinline__ int64_t fd_update_cta(FdEngine &H, Chunk &ch,
                                                 const int64_t *__restrict__ fd_beg,
                                                 const int32_t *__restrict__ fd_len,
                                                 const int32_t *__restrict__ fd_adj, int64_t q0,
                                                 int64_t q1, int32_t r, int32_t ni, int32_t kb,
                                                 FdEmit &emit) {
    FdSweepOut o{&emit};
    return fd_update_cta(H, ch, fd_beg, fd_len, fd_adj, q0, q1, r, ni, kb, o);
}

__device__ __forceinline__ unsigned char *fd_bind_smem(unsigned char *smem, int *s_dn, FdEngine &H,
                                                       Chunk &ch) {
    unsigned char *p = H.bind(smem, s_dn);
    ch.beg = (int64_t *)p;
    ch.pre = (int32_t *)(ch.beg + MID_CHUNK);
    ch.tmp = ch.pre + MID_CHUNK + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    return (unsigned char *)(((uintptr_t)(ch.len + MID_CHUNK) + 15) & ~(uintptr_t)15);
}

__global__ void __launch_bounds__(FD_THREADS, 1) k_fd_peel(FdArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_t, s_dn, s_np, s_nbig, s_nf, s_pick, s_peel, s_rk;
    // window list count and next level's minimum, by level parity: level L
    // fills set L & 1 while stragglers of level L - 1 may still read the other
    __shared__ int s_nk[2];
    __shared__ unsigned long long s_mn[2];
    __shared__ unsigned long long s_rmn;  // minimum of a refilled window
    __shared__ unsigned long long s_T;   // window bound
    __shared__ int32_t s_scan[33];
    __shared__ unsigned long long s_entries;
    __shared__ int s_over;
    FdEngine H;
    Chunk ch;
    fd_bind_smem(smem, &s_dn, H, ch);
    const int lane = threadIdx.x & 31;
    H.clear_all();
    if (threadIdx.x == 0) s_nbig = 0;
    // per warp (lane 0): wedges walked; thread 0 also counts levels
    unsigned long long wedges = 0, levels = 0;
    __syncthreads();
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            s_t = atomicAdd(a.qhead, 1);
            s_entries = 0;
        }
        __syncthreads();
        const int t = s_t;
        if (t >= a.P) break;
        const int32_t i = a.queue[t];
        const int32_t mb = a.tstart[i];
        const int32_t ni = a.tlen[i];
        const int32_t kb = a.tkb[i];
        if (ni == 0) continue;
        unsigned long long t_start = 0;
        if (threadIdx.x == 0) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_start));
        const unsigned long long levels0 = levels;
        unsigned long long *fsup = a.fsup + mb;
        uint8_t *alive = a.alive + mb;
        // members outside the window (far) and inside it (cand), each
        // double-buffered for compaction
        int32_t *flist = a.alist + mb;
        int32_t *flist_next = a.alist2 + mb;
        int32_t *clist = a.clist + mb;
        int32_t *clist_next = a.clist2 + mb;
        int32_t *plist = a.plist + mb;
        const int32_t *mem = a.members + mb;
        const FdMember *info = a.info + mb;
        const int rb = fp_rank_bits(ni);
        unsigned long long entries = 0;
        for (int r = threadIdx.x; r < ni; r += blockDim.x) {
            fsup[r] = a.init[mem[r]];
            alive[r] = 1;
            flist[r] = r;
            const unsigned long long q = a.rec[mb + r];
            entries += q == FP_NONE ? 0 : q & 0xffffffu;
        }
        entries = warp_sum(entries);
        if (lane == 0 && entries) atomicAdd(&s_entries, entries);
        int32_t nalive = ni, nfar = ni, ncand = 0;
        unsigned long long level = 0, mn = ~0ull;
        int par = 0;
        __syncthreads();
        const float2 ns = a.ho.tw ? fd_member_ns(s_entries, a.ho.tw[i], ni) : make_float2(0.f, 0.f);
        const int wide_level = fd_hand_over_from(ns);
        while (nalive > 0) {
            if (ncand == 0) {
                // Window refill: the smallest supports among the far members,
                // about `target` of them, become the window [.., T); a level
                // then scans the window only, and members whose support
                // falls below T during updates join it.
                uint32_t *hist = (uint32_t *)H.tl;  // idle between passes
                for (int b = threadIdx.x; b < LOG_BUCKETS; b += blockDim.x) hist[b] = 0;
                if (threadIdx.x == 0) {
                    s_pick = LOG_BUCKETS - 1;
                    s_nf = 0;
                    s_rk = 0;
                    s_rmn = ~0ull;
                }
                __syncthreads();
                for (int j = threadIdx.x; j < nfar; j += blockDim.x) {
                    const int32_t r = flist[j];
                    if (alive[r]) atomicAdd(&hist[log_bucket_of(fsup[r])], 1u);
                }
                __syncthreads();
                {
                    constexpr int PER = (LOG_BUCKETS + FD_THREADS - 1) / FD_THREADS;
                    const int target = max(FD_WINDOW_MIN, min(FD_WINDOW_MAX, nalive / 32));
                    int32_t c[PER], sum = 0;
#pragma unroll
                    for (int e = 0; e < PER; e++) {
                        const int b = threadIdx.x * PER + e;
                        c[e] = b < LOG_BUCKETS ? (int32_t)hist[b] : 0;
                        sum += c[e];
                    }
                    int32_t run = block_exclusive_scan<int32_t>(sum, s_scan, nullptr);
#pragma unroll
                    for (int e = 0; e < PER; e++) {
                        run += c[e];
                        if (run >= target && c[e] > 0) atomicMin(&s_pick, threadIdx.x * PER + e);
                    }
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    const unsigned long long top = log_bucket_top(s_pick);
                    s_T = top == ~0ull ? ~0ull : top + 1ull;
                }
                __syncthreads();
                const unsigned long long T = s_T;
                for (int base = 0; base < nfar; base += blockDim.x) {
                    const int j = base + threadIdx.x;
                    int32_t r = -1;
                    unsigned long long v = ~0ull;
                    if (j < nfar) {
                        r = flist[j];
                        if (alive[r])
                            v = fsup[r];
                        else
                            r = -1;
                    }
                    const bool in = r >= 0 && v < T;
                    warp_append(in, r, &s_rk, clist);
                    warp_append(r >= 0 && !in, r, &s_nf, flist_next);
                    const unsigned long long kv = warp_min(in ? v : ~0ull);
                    if (lane == 0 && kv != ~0ull) atomicMin(&s_rmn, kv);
                }
                __syncthreads();
                ncand = s_rk;
                nfar = s_nf;
                mn = s_rmn;
                {
                    int32_t *tmp = flist;
                    flist = flist_next;
                    flist_next = tmp;
                }
                if (ncand == 0) break;  // cannot happen while members are alive
            }
            // mu from the minimum left by the previous level (or the refill);
            // this level's counters: the per-level ones and set `par`
            const unsigned long long mu = mn > level ? mn : level;
            const unsigned long long T = s_T;
            level = mu;
            levels++;
            if (threadIdx.x == 0) {
                s_np = 0;
                s_nk[par] = 0;
                s_peel = 0;
                s_mn[par] = ~0ull;
            }
            __syncthreads();
            // peel every window member with support <= mu; the rest go to
            // the other window buffer (ballot compaction, order irrelevant)
            int peeled = 0;
            constexpr int SCAN_U = 4;  // window entries per thread with their loads in flight
            for (int base0 = 0; base0 < ncand; base0 += SCAN_U * blockDim.x) {
                int32_t rr[SCAN_U];
                unsigned long long vv[SCAN_U];
#pragma unroll
                for (int u = 0; u < SCAN_U; u++) {
                    const int j = base0 + u * blockDim.x + threadIdx.x;
                    rr[u] = j < ncand ? clist[j] : -1;
                }
#pragma unroll
                for (int u = 0; u < SCAN_U; u++) vv[u] = rr[u] >= 0 ? fsup[rr[u]] : 0ull;
#pragma unroll
                for (int u = 0; u < SCAN_U; u++) {
                    const int32_t r = rr[u];
                    const unsigned long long v = vv[u];
                    const bool keep = r >= 0 && v > mu;
                    const bool peel = r >= 0 && !keep;
                    if (peel) {
                        alive[r] = 0;
                        a.tip[a.new2old[mem[r]]] = mu;
                        peeled++;
                    }
                    warp_append(keep, r, &s_nk[par], clist_next);
                    warp_append(peel && v > 0, r, &s_np, plist);
                    // minimum of the survivors before this level's updates
                    const unsigned long long kv = warp_min(keep ? v : ~0ull);
                    if (lane == 0 && kv != ~0ull) atomicMin(&s_mn[par], kv);
                }
            }
            peeled = warp_sum(peeled);
            if (lane == 0 && peeled) atomicAdd(&s_peel, peeled);
            __syncthreads();
            nalive -= s_peel;
            {
                int32_t *tmp = clist;
                clist = clist_next;
                clist_next = tmp;
            }
            if (s_np >= wide_level) {
                if (threadIdx.x == 0) s_over = fd_hand_over(a.ho, ns, s_np, i, level);
                __syncthreads();
                if (s_over) {
                    // back to where the level began (any support up to mu does)
                    for (int j = threadIdx.x; j < s_np; j += blockDim.x) {
                        fsup[plist[j]] = mu;
                        alive[plist[j]] = 1;
                    }
                    levels--;
                    break;
                }
            }
            // updates of the peeled vertices inside G_i
            FdEmit emit{fsup, alive, &s_mn[par], T, clist, &s_nk[par]};
            const int np = fd_lists(a.pool, a.rec + mb, plist, s_np, rb, emit, &s_nbig);
            for (int pi = 0; pi < np; pi++) {
                const int32_t r = plist[pi];
                const FdMember m = fd_load(info + r);
                const int64_t walked = fd_update_cta(H, ch, a.fd_beg, a.fd_len, a.fd_adj, m.q0,
                                                     m.q0 + m.deg, r, ni, kb, emit);
                if (threadIdx.x == 0) wedges += (unsigned long long)walked;
            }
            if (np > 0) __syncthreads();
            // window survivors plus the members that fell below T
            ncand = s_nk[par];
            mn = s_mn[par];
            par ^= 1;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long t_end;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_end));
            a.sub_ns[i] = t_end - t_start;
            a.sub_levels[i] = levels - levels0;
        }
    }
    if (lane == 0 && wedges) atomicAdd(&a.stats[0], wedges);
    if (threadIdx.x == 0) atomicAdd(&a.stats[1], levels);
}

// ------------------------------------------------------------------------
// Tasks of at most FS_MEMBERS members: their supports live in shared memory.
//
// Such a task is a chain of thousands of levels that each peel a member or
// two, so a level's cost is its dependent steps. With supports, lists and the
// window in global memory, and walking, a level took 7-14 us (1,268 levels of
// a 1,552-member task 9.4 ms; 6,861 levels of 9,817 members 94 ms). Here a
// level is one scan of the supports (peel what is <= mu, minimum of the rest),
// two dependent loads per member (its record, its list) and two barriers: 1.6
// us at 1,552 members, 2.4 at 9,817. Peeled members have support FS_DEAD. Of
// 227 KB, supports and the level's list take 10 bytes a member, the counters
// for members without a list 64 KB.
// ------------------------------------------------------------------------
constexpr int FS_MEMBERS = 15360;
constexpr int FS_WORDS = 12288;  // dense counters: 24,576 keys
using FsEngine = DenseSliceT<FS_WORDS, TOUCH_LIST>;
static_assert(2 * FS_WORDS >= FS_MEMBERS, "one member's keys fit");
static_assert(FS_MEMBERS <= 1 << 14, "ranks and a mark in 16 bits");
constexpr unsigned long long FS_DEAD = ~0ull;
constexpr size_t FS_CHUNK = (chunk_bytes(FD_THREADS) + 15) & ~(size_t)15;
constexpr size_t FS_SMEM = FS_CHUNK + FsEngine::bytes() + (size_t)FS_MEMBERS * 10;

struct FsEmit {
    unsigned long long *sup;  // shared
    unsigned long long mn;    // this thread's least new support
    __device__ __forceinline__ void operator()(int32_t k, uint32_t c) {
        if (sup[k] == FS_DEAD) return;
        const unsigned long long d = choose2(c);
        const unsigned long long nv = atomicAdd(&sup[k], 0ull - d) - d;
        mn = nv < mn ? nv : mn;
    }
    template <int N>
    __device__ __forceinline__ void many(const int32_t (&k)[N], const uint32_t (&c)[N]) {
#pragma unroll
        for (int u = 0; u < N; u++)
            if (k[u] >= 0) (*this)(k[u], c[u]);
    }
};

// A member alone in a pass of the whole CTA.
struct FsVisit {
    FsEngine *eng;
    int32_t kb, self;  // subset ranks
    __device__ __forceinline__ void operator()(int, int32_t key) {
        if (key != self) eng->add(key - kb);
    }
};

struct FsArgs {
    const int32_t *queue;  // task ids, LPT order
    int32_t T;
    int32_t *qhead;
    const int32_t *tstart, *tlen, *tkb;
    const int32_t *members;
    const FdMember *info;  // by member position
    const uint32_t *pool;
    const unsigned long long *rec;
    const int64_t *fd_beg;
    const int32_t *fd_len;
    const int32_t *fd_adj;
    const int32_t *new2old;
    const unsigned long long *init;
    unsigned long long *rtip;  // by member position
    unsigned long long *tip;   // output, original ids
    unsigned long long *fsup;  // supports of a task that is handed over, by member position
    uint8_t *alive;
    unsigned long long *stats; // [0] wedges, [1] levels
    unsigned long long *sub_ns, *sub_levels;
    FdHandOver ho;
};

// minimum over a warp, in every lane
__device__ __forceinline__ unsigned long long warp_min_all(unsigned long long v) {
    const uint32_t hi = (uint32_t)(v >> 32);
    const uint32_t mh = __reduce_min_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_min_sync(0xffffffffu, hi == mh ? (uint32_t)v : ~0u);
    return ((unsigned long long)mh << 32) | ml;
}

__global__ void __launch_bounds__(FD_THREADS, 1) k_fd_small(FsArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_t, s_dn, s_nbig;
    // by level parity: a level's counts, and the warps' minima for the next
    __shared__ int s_np[2], s_peel[2];
    __shared__ unsigned long long s_mn[2][FD_WARPS];
    __shared__ unsigned long long s_entries;
    __shared__ int s_over;
    Chunk ch;
    ch.beg = (int64_t *)smem;
    ch.pre = (int32_t *)(ch.beg + FD_THREADS);
    ch.tmp = ch.pre + FD_THREADS + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    FsEngine H;
    unsigned long long *sup = (unsigned long long *)H.bind(smem + FS_CHUNK, &s_dn);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    H.clear_all();
    if (threadIdx.x == 0) s_nbig = 0;
    FdMids M{a.fd_beg, a.fd_len};
    unsigned long long wedges = 0, levels = 0;  // wedges: per warp (lane 0)
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            s_t = atomicAdd(a.qhead, 1);
            s_entries = 0;
        }
        __syncthreads();
        const int t = s_t;
        if (t >= a.T) break;
        const int32_t i = a.queue[t];
        const int32_t mb = a.tstart[i], ni = a.tlen[i], kb = a.tkb[i];
        const int32_t *mem = a.members + mb;
        const FdMember *info = a.info + mb;
        unsigned long long *rtip = a.rtip + mb;
        unsigned long long t_start = 0;
        if (threadIdx.x == 0) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_start));
        const int rb = fp_rank_bits(ni);
        const int32_t nip = (ni + 1) & ~1;
        uint16_t *plist = (uint16_t *)(sup + nip);
        unsigned long long mn = FS_DEAD;
        uint32_t entries = 0;  // below FS_MEMBERS^2 in all
        for (int r = threadIdx.x; r < nip; r += FD_THREADS) {
            const unsigned long long v = r < ni ? a.init[mem[r]] : FS_DEAD;
            sup[r] = v;
            mn = v < mn ? v : mn;
            const unsigned long long q = r < ni ? a.rec[mb + r] : 0;
            entries += q == FP_NONE ? 0 : (uint32_t)(q & 0xffffffu);
        }
        entries = __reduce_add_sync(0xffffffffu, entries);
        if (lane == 0 && entries) atomicAdd(&s_entries, (unsigned long long)entries);
        mn = warp_min_all(mn);
        if (lane == 0) s_mn[0][warp] = mn;
        if (threadIdx.x == 0) s_np[0] = s_peel[0] = 0;
        const unsigned long long levels0 = levels;
        unsigned long long level = 0;
        int32_t nalive = ni;
        int par = 0;
        __syncthreads();
        const float2 ns = a.ho.tw ? fd_member_ns(s_entries, a.ho.tw[i], ni) : make_float2(0.f, 0.f);
        const int wide_level = fd_hand_over_from(ns);
        bool over = false;
        while (nalive > 0) {
            // ---- peel every member with support <= mu; minimum of the others
            mn = warp_min_all(s_mn[par][lane & (FD_WARPS - 1)]);
            const unsigned long long mu = mn > level ? mn : level;
            level = mu;
            levels++;
            FsEmit emit{sup, FS_DEAD};
            int peeled = 0;
            for (int base = 0; base < nip; base += 4 * FD_THREADS) {
                unsigned long long v[4];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int r = base + 2 * (h * FD_THREADS + threadIdx.x);
                    const ulonglong2 x = r < nip ? *(const ulonglong2 *)(sup + r)
                                                 : make_ulonglong2(FS_DEAD, FS_DEAD);
                    v[2 * h] = x.x;
                    v[2 * h + 1] = x.y;
                }
                bool any = false;
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    any |= v[u] <= mu;
                    emit.mn = v[u] > mu && v[u] < emit.mn ? v[u] : emit.mn;
                }
                if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const int r = base + 2 * ((u >> 1) * FD_THREADS + threadIdx.x) + (u & 1);
                    const bool peel = v[u] <= mu;
                    if (peel) {
                        sup[r] = FS_DEAD;
                        rtip[r] = mu;
                        peeled++;
                    }
                    const bool upd = peel && v[u] > 0;
                    const unsigned bal = __ballot_sync(0xffffffffu, upd);
                    if (bal) {
                        int pos = 0;
                        if (lane == 0) pos = atomicAdd(&s_np[par], __popc(bal));
                        pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(bal & lanemask_lt());
                        if (upd) plist[pos] = (uint16_t)r;
                    }
                }
            }
            peeled = __reduce_add_sync(0xffffffffu, peeled);
            if (lane == 0 && peeled) atomicAdd(&s_peel[par], peeled);
            __syncthreads();
            nalive -= s_peel[par];
            if (threadIdx.x == 0) s_np[par ^ 1] = s_peel[par ^ 1] = 0;
            if (s_np[par] >= wide_level) {
                if (threadIdx.x == 0) s_over = fd_hand_over(a.ho, ns, s_np[par], i, level);
                __syncthreads();
                over = s_over;
                if (over) {
                    // back to where the level began (any support up to mu does)
                    for (int j = threadIdx.x; j < s_np[par]; j += FD_THREADS) sup[plist[j]] = mu;
                    levels--;
                    __syncthreads();
                    break;
                }
            }
            // ---- updates of the peeled members inside G_i
            const int np = fd_lists(a.pool, a.rec + mb, plist, s_np[par], rb, emit, &s_nbig);
            if (np > 0) {
                for (int pi = 0; pi < np; pi++) {
                    const int32_t r = plist[pi];
                    const FdMember m = fd_load(info + r);
                    H.set_width(ni, m.deg >= 65535);
                    FsVisit v{&H, kb, r + kb};
                    const int64_t walked = cta_walk(M, m.q0, m.q0 + m.deg, a.fd_adj, ch, v);
                    if (walked > 0) H.template sweep<true, true>(emit);
                    __syncthreads();
                    H.reset_scalars();
                    if (threadIdx.x == 0) wedges += (unsigned long long)walked;
                }
            }
            mn = warp_min_all(emit.mn);
            if (lane == 0) s_mn[par ^ 1][warp] = mn;
            par ^= 1;
            __syncthreads();
        }
        for (int r = threadIdx.x; r < ni; r += FD_THREADS) {
            if (!over) {
                a.tip[a.new2old[mem[r]]] = rtip[r];
                continue;
            }
            const unsigned long long v = sup[r];
            a.fsup[mb + r] = v;
            a.alive[mb + r] = v != FS_DEAD;
            if (v == FS_DEAD) a.tip[a.new2old[mem[r]]] = rtip[r];
        }
        if (threadIdx.x == 0) {
            unsigned long long t_end;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_end));
            a.sub_ns[i] = t_end - t_start;
            a.sub_levels[i] = levels - levels0;
        }
    }
    if (lane == 0 && wedges) atomicAdd(&a.stats[0], wedges);
    if (threadIdx.x == 0) atomicAdd(&a.stats[1], levels);
}

// ------------------------------------------------------------------------
// Heavy subsets: one subset peeled by all CTAs, level by level. A subset
// whose wedge count dwarfs the others' would otherwise keep one CTA busy
// long after the rest of the queue is done. Per level: mu from the minimum
// support of the alive members; every alive member with support <= mu is
// peeled (tip mu) and listed by the size of its walk; the warp kernel and the
// CTA kernel apply the updates of the listed members, one warp or one CTA per
// member, and the survivors' minimum for the next level is gathered on the
// way. Same levels, same tip numbers as the one-CTA peel.
// ------------------------------------------------------------------------
struct FdhDev {
    unsigned long long mn;       // minimum support of the alive members
    unsigned long long mn_next;  // the same after this level (survivors, updates)
    unsigned long long level;    // mu of the last level
    unsigned long long wedges, levels;
    unsigned long long t0, t1;   // globaltimer at the start and at the end
    unsigned long long cpeel;    // walk sizes of this level's peeled members with updates
    unsigned long long rcnt;     // C_rcnt of the task's induced subgraph
    int32_t nalive, nkeep, nw, nb;
    int32_t gnt[FDH_SPLIT_NB];   // split levels: keys listed per member
    unsigned long long splits;   // split levels so far
};

struct FdhArgs {
    const int32_t *mem;  // task members (local ids), rank order
    int32_t ni;
    int32_t kb;          // rank of the task's first member inside its subset
    const int64_t *off_s;
    const int64_t *fd_beg;
    const int32_t *fd_len;
    const int32_t *fd_adj;
    const int32_t *new2old;
    const unsigned long long *init;
    unsigned long long *fsup;  // by rank
    uint8_t *alive;            // by rank
    unsigned long long *wr;    // by rank: wedges of the member's walk inside G_i
    int32_t *Lw, *Lb;          // peeled members with small / big walks
    unsigned long long *tip;   // output, original ids
    FdhDev *st;
    uint32_t *gcnt;            // split levels: FDH_SPLIT_NB x ni counters, zero between levels
    int32_t *gtl;              // split levels: FDH_SPLIT_NB x ni listed keys
    const int64_t *wpre;       // side-s edges: exclusive prefix of the run lengths
};

// A level splits its big-walk members' middle vertices over the CTAs when it
// has few of them (the same test in the update and the sweep kernel).
__device__ __forceinline__ bool fdh_split(int32_t nb, int32_t grid) {
    return nb > 0 && nb <= FDH_SPLIT_NB && grid >= 2 * nb;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void k_fdh_reset(FdhDev *st, int32_t ni) {
    st->mn = st->mn_next = ~0ull;
    st->cpeel = st->rcnt = 0;
    st->level = 0;
    st->wedges = st->levels = 0;
    st->t0 = globaltimer_ns();
    st->t1 = 0;
    st->nalive = ni;
    st->nkeep = st->nw = st->nb = 0;
    for (int i = 0; i < FDH_SPLIT_NB; i++) st->gnt[i] = 0;
    st->splits = 0;
}

__global__ void k_fdh_init(FdhArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long mn = ~0ull;
    for (int64_t r = w0; r < a.ni; r += nw) {
        if (lane == 0) {
            const unsigned long long v = a.init[a.mem[r]];
            a.fsup[r] = v;
            a.alive[r] = 1;
            mn = v < mn ? v : mn;
        }
    }
    if (lane == 0 && mn != ~0ull) atomicMin(&a.st->mn, mn);
}

// A task that was handed over: its supports and alive members are there.
__global__ void k_fdh_resume(FdhArgs a, const unsigned long long *__restrict__ level) {
    unsigned long long mn = ~0ull;
    int32_t alive = 0;
    for (int32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < a.ni; r += gridDim.x * blockDim.x)
        if (a.alive[r]) {
            const unsigned long long v = a.fsup[r];
            alive++;
            mn = v < mn ? v : mn;
        }
    alive = warp_sum(alive);
    mn = warp_min(mn);
    if ((threadIdx.x & 31) == 0 && alive) {
        atomicAdd(&a.st->nalive, alive);
        atomicMin(&a.st->mn, mn);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->level = *level;
}

__global__ void k_fdh_select(FdhArgs a) {
    const unsigned long long lv = a.st->level, mn = a.st->mn;
    const unsigned long long mu = mn > lv ? mn : lv;
    int32_t keep = 0;
    unsigned long long kmin = ~0ull, cpeel = 0;
    for (int32_t base = blockIdx.x * blockDim.x; base < a.ni; base += gridDim.x * blockDim.x) {
        const int32_t r = base + threadIdx.x;
        const bool al = r < a.ni && a.alive[r];
        const unsigned long long v = al ? a.fsup[r] : 0;
        const bool peel = al && v <= mu;
        if (peel) {
            a.alive[r] = 0;
            a.tip[a.new2old[a.mem[r]]] = mu;
        }
        const bool upd = peel && v > 0;
        const bool small = upd && a.wr[r] <= (unsigned long long)WARP_MAX_W;
        if (upd) cpeel += a.wr[r] & ~WIDE_BIT;
        warp_append(small, r, &a.st->nw, a.Lw);
        warp_append(upd && !small, r, &a.st->nb, a.Lb);
        if (al && !peel) {
            keep++;
            kmin = v < kmin ? v : kmin;
        }
    }
    keep = warp_sum(keep);
    kmin = warp_min(kmin);
    cpeel = warp_sum(cpeel);
    if ((threadIdx.x & 31) == 0) {
        if (keep) atomicAdd(&a.st->nkeep, keep);
        if (kmin != ~0ull) atomicMin(&a.st->mn_next, kmin);
        if (cpeel) atomicAdd(&a.st->cpeel, cpeel);
    }
}

// Hybrid update computation inside the fine-grained step (Sec. 4.1): a
// member's support is the butterflies it shares with the vertices of higher
// subsets (constant while its task is peeled: init minus its count inside
// G_i) plus those it shares with the task's members still alive (its count
// inside the alive part of G_i). A level of a heavy task may therefore
// replace its updates by a recount of the alive part.
//
// C_rcnt of the task's induced subgraph: sum over its members' edges (x, y)
// of min(d_x, d_y inside G_i).
__global__ void k_fdh_rcnt(FdhArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long sum = 0;
    for (int64_t r = w0; r < a.ni; r += nw) {
        const int32_t x = a.mem[r];
        const int64_t q0 = a.off_s[x], q1 = a.off_s[x + 1];
        for (int64_t q = q0 + lane; q < q1; q += 32)
            sum += (unsigned long long)imin64(q1 - q0, a.fd_len[q]);
    }
    sum = warp_sum(sum);
    if (lane == 0 && sum) atomicAdd(&a.st->rcnt, sum);
}

// keep[mem[r]] = -1 for the task's members (alive ones only with alive_only),
// the others of the side stay excluded (0).
__global__ void k_fdh_keep(FdhArgs a, int32_t *__restrict__ keep, int alive_only) {
    const int32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < a.ni && (!alive_only || a.alive[r])) keep[a.mem[r]] = -1;
}

// Supports of the alive members after a recount: init - (count inside G_i)
// + (count inside the alive part of G_i); the next level's minimum follows.
__global__ void k_fdh_apply(FdhArgs a, const unsigned long long *__restrict__ cnt0,
                            const unsigned long long *__restrict__ cntr) {
    const int32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long v = ~0ull;
    if (r < a.ni && a.alive[r]) {
        const int32_t x = a.mem[r];
        v = a.init[x] - cnt0[x] + cntr[x];
        a.fsup[r] = v;
    }
    v = warp_min(v);
    if ((threadIdx.x & 31) == 0 && v != ~0ull) atomicMin(&a.st->mn_next, v);
}

__global__ void __launch_bounds__(256) k_fdh_warp(FdhArgs a) {
    __shared__ int32_t skey[8][WARP_SLOTS];
    __shared__ uint32_t sval[8][WARP_SLOTS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    WarpHash WH{skey[w], sval[w]};
    WH.clear(lane);
    __syncwarp();
    FdEmit emit{a.fsup, a.alive, &a.st->mn_next, ~0ull, nullptr, nullptr};
    FdMids M{a.fd_beg, a.fd_len};
    const int32_t nw = a.st->nw;
    unsigned long long wedges = 0;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t ngw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = gw; i < nw; i += ngw) {
        const int32_t r = a.Lw[i];
        const int32_t x = a.mem[r];
        fd_update_warp(WH, M, a.fd_adj, a.off_s[x], a.off_s[x + 1], r, a.kb, lane, emit);
        wedges += a.wr[r];
    }
    if (lane == 0 && wedges) atomicAdd(&a.st->wedges, wedges);
}

__global__ void __launch_bounds__(FD_THREADS, 1) k_fdh_cta(FdhArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_dn;
    FdEngine H;
    Chunk ch;
    fd_bind_smem(smem, &s_dn, H, ch);
    H.clear_all();
    __syncthreads();
    FdEmit emit{a.fsup, a.alive, &a.st->mn_next, ~0ull, nullptr, nullptr};
    const int32_t nb = a.st->nb;
    unsigned long long wedges = 0;
    if (fdh_split(nb, gridDim.x)) {
        // K CTAs per member, each over an equal share of its walk's wedges
        // (runs cut at the share's ends); k_fdh_sweep applies the summed
        // counts
        const int32_t K = gridDim.x / nb;
        for (int32_t it = blockIdx.x; it < nb * K; it += gridDim.x) {
            const int32_t i = it / K, k = it % K;
            const int32_t r = a.Lb[i];
            const int32_t x = a.mem[r];
            const int64_t q0 = a.off_s[x], q1 = a.off_s[x + 1];
            const int64_t w0 = a.wpre[q0], W = a.wpre[q1] - w0;
            const int64_t lo = w0 + W * k / K, hi = w0 + W * (k + 1) / K;
            if (lo == hi) continue;
            // edge whose run holds wedge position p: the last q in [q0, q1)
            // with wpre[q] <= p (runs of length 0 are passed over)
            auto run_of = [&](int64_t p) {
                int64_t l = q0, h = q1 - 1;
                while (l < h) {
                    const int64_t md = (l + h + 1) >> 1;
                    if (a.wpre[md] <= p)
                        l = md;
                    else
                        h = md - 1;
                }
                return l;
            };
            const int64_t qa = run_of(lo), ql = run_of(hi - 1);
            const int32_t skip = (int32_t)(lo - a.wpre[qa]);
            const int32_t keep = (int32_t)(hi - a.wpre[ql]);
            FdPartialOut o{a.gcnt + (size_t)i * a.ni, a.gtl + (size_t)i * a.ni, &a.st->gnt[i]};
            wedges += (unsigned long long)fd_update_cta(H, ch, a.fd_beg, a.fd_len, a.fd_adj, qa,
                                                        ql + 1, r, a.ni, a.kb, o, skip, keep);
        }
    } else {
        for (int32_t i = blockIdx.x; i < nb; i += gridDim.x) {
            const int32_t r = a.Lb[i];
            const int32_t x = a.mem[r];
            wedges += (unsigned long long)fd_update_cta(H, ch, a.fd_beg, a.fd_len, a.fd_adj,
                                                        a.off_s[x], a.off_s[x + 1], r, a.ni, a.kb,
                                                        emit);
        }
    }
    if (threadIdx.x == 0 && wedges) atomicAdd(&a.st->wedges, wedges);
}

// Split levels: the summed count c of every listed key becomes the support
// decrement C(c, 2) of that member (alive ones only), and the counters return
// to zero. `grid` is the update kernel's grid.
__global__ void k_fdh_sweep(FdhArgs a, int32_t grid) {
    const int32_t nb = a.st->nb;
    if (!fdh_split(nb, grid)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->splits++;
    FdEmit emit{a.fsup, a.alive, &a.st->mn_next, ~0ull, nullptr, nullptr};
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nt = (int64_t)gridDim.x * blockDim.x;
    for (int32_t i = 0; i < nb; i++) {
        uint32_t *gc = a.gcnt + (size_t)i * a.ni;
        const int32_t *gl = a.gtl + (size_t)i * a.ni;
        const int32_t n = a.st->gnt[i];
        for (int64_t t = t0; t < n; t += nt) {
            const int32_t z = gl[t];
            const uint32_t c = gc[z];
            gc[z] = 0u;
            if (c >= 2u) emit(z, c);
        }
    }
}

// Closes a level. Launched again after the subset is empty, it changes
// nothing that is read later (the host enqueues levels ahead of its check).
__device__ void fdh_close_level(FdhDev *st) {
    for (int i = 0; i < FDH_SPLIT_NB; i++) st->gnt[i] = 0;
    if (st->nalive == 0) return;
    const unsigned long long mu = st->mn > st->level ? st->mn : st->level;
    st->level = mu;
    st->mn = st->mn_next;
    st->mn_next = ~0ull;
    st->nalive = st->nkeep;
    st->nkeep = st->nw = st->nb = 0;
    st->cpeel = 0;
    st->levels++;
    if (st->nalive == 0) st->t1 = globaltimer_ns();
}

__global__ void k_fdh_next(FdhDev *st) { fdh_close_level(st); }

// The same inside a graph's while-node: the loop goes on while members are
// alive (at most ni levels: every level peels at least one member).
__global__ void k_fdh_next_loop(FdhDev *st, int32_t ni, cudaGraphConditionalHandle cond) {
    fdh_close_level(st);
    cudaGraphSetConditional(cond, (st->nalive > 0 && st->levels < (unsigned long long)ni) ? 1u : 0u);
}

}  // namespace

// A graph and its executable, destroyed together.
struct GraphOwner {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t e = nullptr;
    ~GraphOwner() {
        if (e) cudaGraphExecDestroy(e);
        if (g) cudaGraphDestroy(g);
    }
};

// Levels of one heavy task one at a time, each deciding on the host between
// its updates and a recount of the task's alive members (hybrid update
// computation, Sec. 4.1): with D.fd_huc == 1 every level with updates
// recounts (test hook), otherwise a level whose peeled members' walks exceed
// D.huc_factor * rcnt does. Exact either way.
static void fdh_levels_with_recount(Decomp &D, const FdhArgs &ha, FdhDev *dst, FdhDev *hst_out,
                             uint64_t rcnt, int grid_h, size_t smem_h, int gm, cudaStream_t s) {
    const Side &S = *D.S;
    const Side &O = *D.O;
    const int32_t n = S.n;
    const int sms = num_sms();
    FdhDev *h = (FdhDev *)pinned_scratch(sizeof(FdhDev));
    DevBuf<int32_t> keep, adjc, lenc;
    DevBuf<unsigned long long> cnt0, cntr;
    bool have0 = false;
    // counts of the task's members (all, or the alive ones) inside G_i
    auto count_members = [&](int alive_only, unsigned long long *out) {
        if (!keep.get()) {
            keep.alloc(n, s);
            adjc.alloc(D.m, s);
            lenc.alloc(O.n, s);
        }
        keep.zero();
        k_fdh_keep<<<ceil_div(ha.ni, 256), 256, 0, s>>>(ha, keep.get(), alive_only);
        RC_LAUNCH();
        RC_CUDA(cudaMemcpyAsync(adjc.get(), O.adj, sizeof(int32_t) * D.m, cudaMemcpyDeviceToDevice, s));
        list_lengths(O.off, O.n, lenc.get(), s);
        compact_lists(O.off, lenc.get(), adjc.get(), O.n, keep.get(), s);
        return recount_masked(D, keep.get(), out, lenc.get(), adjc.get(), s);
    };
    for (;;) {
        k_fdh_select<<<gm, 256, 0, s>>>(ha);
        RC_LAUNCH();
        RC_CUDA(cudaMemcpyAsync(h, dst, sizeof(FdhDev), cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
        const bool updates = h->nw + h->nb > 0;
        const bool recount =
            updates && (D.fd_huc == 1 || (double)h->cpeel > D.huc_factor * (double)rcnt);
        if (recount) {
            if (!have0) {
                cnt0.alloc(n, s);
                cntr.alloc(n, s);
                D.wedges_fd_recount += count_members(0, cnt0.get());
                have0 = true;
            }
            D.wedges_fd_recount += count_members(1, cntr.get());
            k_fdh_apply<<<ceil_div(ha.ni, 256), 256, 0, s>>>(ha, cnt0.get(), cntr.get());
            RC_LAUNCH();
            D.fd_recounts++;
        } else {
            k_fdh_warp<<<sms * 8, 256, 0, s>>>(ha);
            RC_LAUNCH();
            k_fdh_cta<<<grid_h, FD_THREADS, smem_h, s>>>(ha);
            RC_LAUNCH();
            k_fdh_sweep<<<sms * 4, 256, 0, s>>>(ha, grid_h);
            RC_LAUNCH();
        }
        k_fdh_next<<<1, 1, 0, s>>>(dst);
        RC_LAUNCH();
        if (h->nkeep == 0) break;
    }
    RC_CUDA(cudaMemcpyAsync(hst_out, dst, sizeof(FdhDev), cudaMemcpyDeviceToHost, s));
}

// Dense tasks that all CTAs peel sooner than their lists are made and applied by
// one CTA (others are handed over when that shows, FdHandOver, after their lists
// were made: 1.7 ps a wedge, which dense tasks have many of for an entry. 8M edges
// on 20,000 x 1,000, 160 wedges for each two members: the step took 428 ms in one
// CTA, 232 handed over, 152 so; 3M on 10,000 x 50,000, 1.8 wedges: 45, 15, 27; 2M on
// 5,000 x 20,000, 8: 20, 6.8, 8.4).
// One CTA takes 2.5 us a level and 0.85 ns an entry, all CTAs ~70 us a level and 3
// ps a wedge. The levels are not known before the peel: at most a member each, and
// while every peeled member sets off others as many as the range's share of its
// bound (the narrowest ranges, one bucket, hold 1/32), or 16 to each support of a
// range of few supports (measured: 1.2 to 14 times fewer). Entries: one for every
// two members (all share middle vertices).
// One CTA a task peels the tasks left side by side, the heavy ones come one by
// one: the longest go first while the sum falls.
constexpr double DENSE_TASK = 16;  // wedges for each two members, at least
struct DenseTask {
    int32_t id;
    double list, heavy, walks;  // ns by one CTA, by all, to make its lists
};
// n members, w wedges, range [lo, hi)
static DenseTask dense_task(int32_t id, int32_t n, unsigned long long w, uint64_t lo, uint64_t hi) {
    const double span = (double)(hi - lo), nd = (double)n, wd = (double)w;
    const double levels = std::max(1.0, std::min({nd * std::min(1.0, span / (double)hi), nd, 16.0 * span}));
    const double entries = std::min(wd / 4, nd * nd);
    return DenseTask{id, 2500.0 * levels + 0.85 * entries, 7e4 * levels + 0.003 * wd, 0.0017 * wd};
}
static std::vector<int32_t> heavy_by_lists(std::vector<DenseTask> t, int ctas) {
    // (stored costs: computed in the comparison they may be rounded in two ways)
    std::stable_sort(t.begin(), t.end(),
                     [](const DenseTask &a, const DenseTask &b) { return a.list > b.list; });
    double left = 0, walks = 0;  // of the tasks not heavy
    for (const DenseTask &k : t) {
        left += k.list;
        walks += k.walks;
    }
    double first = 0, best = 0, sum = 0;
    size_t n = 0;
    for (size_t k = 0; k <= t.size(); k++) {
        const double now = sum + walks + std::max(k < t.size() ? t[k].list : 0.0, left / ctas);
        if (k == 0) first = best = now;
        if (now < best && now < 0.9 * first) {
            best = now;
            n = k;
        }
        if (k == t.size()) break;
        sum += t[k].heavy;
        left -= t[k].list;
        walks -= t[k].walks;
        if (sum > best) break;
    }
    std::vector<int32_t> out;
    for (size_t k = 0; k < n; k++) out.push_back(t[k].id);
    return out;
}

void fd_run(Decomp &D, uint64_t *d_tip, cudaStream_t s) {
    const int32_t n = D.n;
    const int64_t m = D.m;
    const int32_t P = D.p_eff;
    if (n == 0 || P == 0) return;
    const Side &S = *D.S;
    const Side &O = *D.O;
    // members and ranks
    DevBuf<int32_t> mstart(P + 1, s), members(n, s), rank(n, s);
    {
        DevBuf<uint64_t> key(n, s);
        k_sub_keys<<<ceil_div(n, 256), 256, 0, s>>>(D.sub, n, key.get());
        RC_LAUNCH();
        radix_sort(key, n, 32, 32 + bits_for((uint64_t)P), s);
        k_sub_starts<<<ceil_div(P + 1, 256), 256, 0, s>>>(key.get(), n, P, mstart.get());
        RC_LAUNCH();
        k_members<<<ceil_div(n, 256), 256, 0, s>>>(key.get(), n, mstart.get(), members.get(),
                                                   rank.get());
        RC_LAUNCH();
    }
    // induced subgraphs
    DevBuf<int32_t> fd_adj(m, s), fd_len(m, s);
    DevBuf<int64_t> fd_beg(m, s), wpre;
    DevBuf<unsigned long long> wr(n, s);
    DevBuf<FdMember> info(n, s);
    DevBuf<int32_t> wide(P, s);
    DevBuf<unsigned long long> wsub(P, s);
    wsub.zero();
    wide.zero();
    if (m > 0) {
        DevBuf<uint64_t> key(m, s);
        k_edge_sub_keys<<<ceil_div(m, 256), 256, 0, s>>>(O.adj, m, D.sub, key.get());
        RC_LAUNCH();
        radix_sort(key, m, 32, 32 + bits_for((uint64_t)P), s);
        DevBuf<int32_t> fd_y(m, s);
        DevBuf<uint32_t> head(m + 1, s), hpos(m + 1, s);
        k_fd_fill<<<ceil_div(m, 256), 256, 0, s>>>(key.get(), m, O.adj, O.off, O.n, rank.get(),
                                                   fd_adj.get(), fd_y.get(), head.get());
        RC_LAUNCH();
        RC_CUDA(cudaMemsetAsync(head.get() + m, 0, 4, s));
        scan_exclusive<uint32_t>(head.get(), hpos.get(), m + 1, s);
        uint32_t nruns = 0;
        RC_CUDA(cudaMemcpyAsync(&nruns, hpos.get() + m, 4, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
        DevBuf<int64_t> run_start(nruns + 1, s);
        k_run_starts<<<ceil_div(m, 256), 256, 0, s>>>(head.get(), hpos.get(), m, run_start.get());
        RC_LAUNCH();
        k_fd_edges<<<ceil_div(m, 256), 256, 0, s>>>(key.get(), m, O.adj, fd_y.get(), head.get(),
                                                    hpos.get(), run_start.get(), nruns, S.off, S.adj,
                                                    fd_beg.get(), fd_len.get());
        RC_LAUNCH();
        // walk sizes of all vertices: prefix sums of the run lengths (kept
        // for the split levels of heavy tasks)
        DevBuf<int64_t> l64(m + 1, s);
        wpre.alloc(m + 1, s);
        k_i32_to_i64<<<ceil_div(m, 256), 256, 0, s>>>(fd_len.get(), m, l64.get());
        RC_LAUNCH();
        RC_CUDA(cudaMemsetAsync(l64.get() + m, 0, sizeof(int64_t), s));
        scan_exclusive<int64_t>(l64.get(), wpre.get(), m + 1, s);
        k_fd_walk_sizes<<<ceil_div(n, 256), 256, 0, s>>>(S.off, n, wpre.get(), D.sub, mstart.get(),
                                                         rank.get(), wr.get(), info.get(),
                                                         wide.get());
        RC_LAUNCH();
    } else {
        wr.zero();
        info.zero();
    }
    // subset sizes and wedge counts
    std::vector<int32_t> hms(P + 1);
    std::vector<unsigned long long> hw(P);
    std::vector<int32_t> hwide(P);
    RC_CUDA(cudaMemcpyAsync(hwide.data(), wide.get(), sizeof(int32_t) * P, cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaMemcpyAsync(hms.data(), mstart.get(), sizeof(int32_t) * (P + 1),
                            cudaMemcpyDeviceToHost, s));
    // Tasks: a subset, or, in a batch's disjoint union, each packed graph's
    // part of a subset (parts share no butterfly, so each is peeled on its
    // own; consecutive small parts of one subset are merged up to TASK_MIN
    // members). A task covers consecutive member positions, which are
    // consecutive ranks of its subset.
    std::vector<int32_t> tstart, tlen, tkb, tsub;
    {
        const int ng = D.parts ? (int)D.parts->size() - 1 : 0;
        DevBuf<int64_t> dparts(ng > 0 ? ng + 1 : 1, s);
        if (ng > 0)
            RC_CUDA(cudaMemcpyAsync(dparts.get(), D.parts->data(), 8 * (ng + 1),
                                    cudaMemcpyHostToDevice, s));
        DevBuf<uint32_t> flag(n + 1, s), fpos(n + 1, s);
        k_task_flags<<<ceil_div(n, 256), 256, 0, s>>>(members.get(), n, D.sub, mstart.get(),
                                                      dparts.get(), ng, flag.get());
        RC_LAUNCH();
        RC_CUDA(cudaMemsetAsync(flag.get() + n, 0, 4, s));
        scan_exclusive<uint32_t>(flag.get(), fpos.get(), n + 1, s);
        uint32_t nseg = 0;
        RC_CUDA(cudaMemcpyAsync(&nseg, fpos.get() + n, 4, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
        DevBuf<int32_t> segs(nseg > 0 ? nseg : 1, s);
        k_flag_positions<<<ceil_div(n, 256), 256, 0, s>>>(flag.get(), fpos.get(), n, segs.get());
        RC_LAUNCH();
        std::vector<int32_t> hseg(nseg);
        if (nseg > 0)
            RC_CUDA(cudaMemcpyAsync(hseg.data(), segs.get(), 4 * (size_t)nseg,
                                    cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
        int sub_i = 0;
        for (uint32_t k = 0; k < nseg; k++) {
            const int32_t b = hseg[k];
            while (sub_i + 1 <= P && hms[sub_i + 1] <= b) sub_i++;  // subset holding b
            const bool new_sub = tsub.empty() || tsub.back() != sub_i;
            if (new_sub || tlen.back() >= TASK_MIN) {
                tstart.push_back(b);
                tlen.push_back(0);
                tkb.push_back(b - hms[sub_i]);
                tsub.push_back(sub_i);
            }
            const int32_t e = k + 1 < nseg ? hseg[k + 1] : n;
            tlen.back() += e - b;
        }
    }
    const int T = (int)tstart.size();
    // task weights: walk sizes summed over the task's members (LPT key)
    std::vector<unsigned long long> tw(T), tlw(T);  // tlw: of members without a list
    DevBuf<int64_t> cw;  // prefix of the members' costs, by member position
    DevBuf<unsigned long long> dtw;  // tw on the device
    DevBuf<int32_t> d_tstart(T > 0 ? T : 1, s), d_tlen(T > 0 ? T : 1, s), d_tkb(T > 0 ? T : 1, s);
    if (T > 0) {
        RC_CUDA(cudaMemcpyAsync(d_tstart.get(), tstart.data(), 4 * (size_t)T, cudaMemcpyHostToDevice, s));
        RC_CUDA(cudaMemcpyAsync(d_tlen.get(), tlen.data(), 4 * (size_t)T, cudaMemcpyHostToDevice, s));
        RC_CUDA(cudaMemcpyAsync(d_tkb.get(), tkb.data(), 4 * (size_t)T, cudaMemcpyHostToDevice, s));
        DevBuf<int64_t> w64(n + 1, s);
        cw.alloc(n + 1, s);
        dtw.alloc(T, s);
        k_walk_cost<<<ceil_div(n, 256), 256, 0, s>>>(wr.get(), n, FP_MEMBER_COST, info.get(),
                                                     members.get(), D.sub, w64.get(), wsub.get());
        RC_LAUNCH();
        RC_CUDA(cudaMemsetAsync(w64.get() + n, 0, 8, s));
        scan_exclusive<int64_t>(w64.get(), cw.get(), n + 1, s);
        k_task_weights<<<ceil_div(T, 256), 256, 0, s>>>(d_tstart.get(), d_tlen.get(), cw.get(),
                                                        FP_MEMBER_COST, T, dtw.get());
        RC_LAUNCH();
        DevBuf<unsigned long long> dlw(T, s);
        dlw.zero();
        k_listless<<<ceil_div(n, 256), 256, 0, s>>>(info.get(), n, d_tstart.get(), d_tlen.get(), T,
                                                    *std::max_element(tlen.begin(), tlen.end()),
                                                    dlw.get());
        RC_LAUNCH();
        RC_CUDA(cudaMemcpyAsync(tw.data(), dtw.get(), 8 * (size_t)T, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaMemcpyAsync(hw.data(), wsub.get(), 8 * P, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaMemcpyAsync(tlw.data(), dlw.get(), 8 * (size_t)T, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
    }
    // LPT order (ties by task id), a member counting as LEVEL_WEDGES wedges.
    std::vector<int32_t> hq(T);
    for (int k = 0; k < T; k++) hq[k] = k;
    std::stable_sort(hq.begin(), hq.end(), [&](int32_t x, int32_t y) {
        const unsigned long long kx = tw[x] + LEVEL_WEDGES * (unsigned long long)tlen[x];
        const unsigned long long ky = tw[y] + LEVEL_WEDGES * (unsigned long long)tlen[y];
        return kx > ky;
    });
    const size_t smem = FdEngine::bytes() + CHUNK_BYTES;
    allow_max_smem((const void *)k_fd_peel);
    int occ = 0;
    RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_fd_peel, FD_THREADS, smem));
    const int sms = num_sms();
    const int grid_all = sms * std::max(occ, 1);
    // Heavy tasks (peeled first by all CTAs, ~60-110 us a level): those above
    // the threshold in wedges. Automatic: (a) what the members without a list
    // walk outweighs the task's levels several times (or its walks do, if its
    // lists would not fit the pool); (b) tasks of HEAVY_NI members and more
    // with a range so narrow that few levels peel them: a one-CTA level scans
    // at ~8 ns a member (1.9M members, width 1, one level: 16 ms, 0.8 heavy;
    // 132K members, width 1, 28 levels: 27 ms for the step, 29 unless heavy);
    // (c) dense tasks (heavy_by_lists). Otherwise one CTA is faster (4,751
    // levels of 80K members take 36 ms there and took 590 heavy, 20,000 levels
    // of 42K members 117 ms), or notices that it is not (FdHandOver).
    // The pool has room for the most entries the lists can have as long as that
    // is cheap (FD_LIST_BYTES an edge), else for about as many as they will have,
    // up to an eighth of the memory there is; members past it walk.
    unsigned long long entries_max = 0, entries = 0;
    for (int k = 0; k < T; k++) {
        entries_max += lists_at_most(tw[k], tlen[k]);
        entries += std::min(lists_about(tw[k], tlen[k]), lists_at_most(tw[k], tlen[k]));
    }
    unsigned long long pool_cap = (unsigned long long)(FD_LIST_BYTES / 4 * m);
    if (entries_max > pool_cap && entries > pool_cap && !D.list_bound)
        pool_cap = std::max(pool_cap, std::min<unsigned long long>(entries, available_bytes() / 32));
    pool_cap = std::min(pool_cap, entries_max);
    // Queue: the heavy tasks, then the large ones (k_fd_peel), then those of
    // at most FS_MEMBERS members (FS_WORDS with 32-bit counts; k_fd_small),
    // each in LPT order.
    const std::vector<int32_t> lpt = hq;
    int nheavy = 0, nsmall_at = 0;
    auto order = [&](unsigned long long cap) {
        hq = lpt;
        nheavy = 0;
        if (D.fd_heavy_w >= 0 && T > 0) {
            const bool overflow = entries > cap;
            std::vector<int32_t> front, back;
            for (int32_t t : lpt) {
                const unsigned long long lw = LEVEL_WEDGES * (unsigned long long)tlen[t];
                const unsigned long long walk = overflow ? tw[t] : tlw[t];
                const int sub_i = tsub[t];
                const uint64_t width = (size_t)sub_i + 1 < D.bounds.size()
                                           ? D.bounds[sub_i + 1] - D.bounds[sub_i]
                                           : ~0ull;
                const bool heavy =
                    D.fd_heavy_w > 0
                        ? tw[t] >= (unsigned long long)D.fd_heavy_w
                        : (walk >= HEAVY_MIN_W && walk >= HEAVY_WALK_LEVELS * lw) ||
                              (tlen[t] >= HEAVY_NI && width <= (uint64_t)(tlen[t] / (HEAVY_NI / 2)));
                (heavy && tlen[t] > 0 ? front : back).push_back(t);
            }
            if (D.fd_heavy_w == 0 && cap > 0) {
                std::vector<DenseTask> lt;
                for (int32_t t : back) {
                    const int sub_i = tsub[t];
                    if ((double)tw[t] < DENSE_TASK * (double)tlen[t] * (double)tlen[t]) continue;
                    const bool open = (size_t)sub_i + 1 >= D.bounds.size();
                    lt.push_back(dense_task(t, tlen[t], tw[t], open ? 0 : D.bounds[sub_i],
                                            open ? ~0ull : D.bounds[sub_i + 1]));
                }
                const std::vector<int32_t> more = heavy_by_lists(lt, sms);
                std::vector<bool> is(T, false);
                for (int32_t t : more) is[t] = true;
                front.insert(front.end(), more.begin(), more.end());
                back.erase(std::remove_if(back.begin(), back.end(), [&](int32_t t) { return is[t]; }),
                           back.end());
            }
            nheavy = (int)front.size();
            int pos = 0;
            for (int32_t t : front) hq[pos++] = t;
            for (int32_t t : back) hq[pos++] = t;
        }
        nsmall_at = (int)(std::stable_partition(hq.begin() + nheavy, hq.end(),
                                                [&](int32_t t) {
                                                    return tlen[t] > (hwide[tsub[t]] ? FS_WORDS
                                                                                     : FS_MEMBERS);
                                                }) -
                          hq.begin());
    };
    // The lists' pool: room for the tasks that are not heavy, and each warp's
    // last block. Without memory for it the order is another.
    const int pair_ctas = 2 * sms;
    DevBuf<uint32_t> pool;
    unsigned long long cap = 0;
    auto make_pool = [&]() {
        unsigned long long most = 0;
        for (int k = nheavy; k < T; k++) most += lists_at_most(tw[hq[k]], tlen[hq[k]]);
        cap = std::min(pool_cap, most) + (unsigned long long)pair_ctas * FP_WARPS * FP_BLOCK;
        return nheavy == T || pool.try_alloc((size_t)cap, s);
    };
    order(pool_cap);
    if (!make_pool()) {
        cap = 0;
        order(0);
    } else if (nheavy > 0) {
        pool.release();  // the heavy tasks' recounts may want the memory
    }
    DevBuf<int32_t> queue(T > 0 ? T : 1, s);
    if (T > 0)
        RC_CUDA(cudaMemcpyAsync(queue.get(), hq.data(), 4 * (size_t)T, cudaMemcpyHostToDevice, s));
    DevBuf<unsigned long long> fsup(n, s);
    DevBuf<uint8_t> alive(n, s);
    DevBuf<int32_t> alist(n, s), alist2(n, s), clist(n, s), clist2(n, s), plist(n, s), blist(n, s),
        qhead(2, s);
    // stats: wedges, levels, tasks handed over (FdHandOver::count)
    DevBuf<unsigned long long> stats(3, s), sub_ns(T > 0 ? T : 1, s), sub_lv(T > 0 ? T : 1, s);
    qhead.zero();
    stats.zero();
    sub_ns.zero();
    sub_lv.zero();
    D.fd_heavy = nheavy;
    D.fd_heavy_ms = 0;
    D.fd_heavy_levels = 0;
    D.fd_split_levels = 0;
    std::vector<FdhDev> hh;  // of the heavy tasks, in the order in which they were peeled
    std::vector<int32_t> heavy_tasks;
    // level: null, or per task the level at which it was handed over
    auto peel_heavy = [&](const int32_t *tasks, int count, const unsigned long long *level) {
        heavy_tasks.insert(heavy_tasks.end(), tasks, tasks + count);
        hh.resize(heavy_tasks.size());
        FdhDev *hh0 = hh.data() + (hh.size() - count);
        DevBuf<FdhDev> hst(1, s);
        const size_t smem_h = FdEngine::bytes() + CHUNK_BYTES;
        allow_max_smem((const void *)k_fdh_cta);
        int occ_h = 0;
        RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_h, k_fdh_cta, FD_THREADS, smem_h));
        const int grid_h = sms * std::max(occ_h, 1);
        // global counters of split levels, sized for the largest heavy task
        int32_t ni_max = 1;
        for (int h = 0; h < count; h++) ni_max = std::max(ni_max, tlen[tasks[h]]);
        DevBuf<uint32_t> gcnt((size_t)FDH_SPLIT_NB * ni_max, s);
        DevBuf<int32_t> gtl((size_t)FDH_SPLIT_NB * ni_max, s);
        gcnt.zero();
        for (int h = 0; h < count; h++) {
            const int32_t i = tasks[h];
            const int32_t mb = tstart[i], ni = tlen[i];
            FdhArgs ha{members.get() + mb, ni,           tkb[i],         S.off,
                       fd_beg.get(),       fd_len.get(), fd_adj.get(),   S.new2old,
                       D.init,             fsup.get() + mb, alive.get() + mb, wr.get() + mb,
                       plist.get() + mb,   blist.get() + mb, (unsigned long long *)d_tip,
                       hst.get(),          gcnt.get(),   gtl.get(),      wpre.get()};
            const int gm = std::max(1, std::min(ceil_div(ni, 256), sms * 4));
            const int gi = std::max(1, std::min(ceil_div((int64_t)ni * 32, 256), sms * 16));
            k_fdh_reset<<<1, 1, 0, s>>>(hst.get(), level ? 0 : ni);
            RC_LAUNCH();
            if (level)
                k_fdh_resume<<<gm, 256, 0, s>>>(ha, level + i);
            else
                k_fdh_init<<<gi, 256, 0, s>>>(ha);
            RC_LAUNCH();
            // Recount rule (Sec. 4.1) of this task: a level recounts when its
            // peeled members' walks exceed factor * C_rcnt of the task; no
            // level can when the task's whole walk weight does not.
            bool may_recount = D.fd_huc == 1;
            uint64_t rcnt = 0;
            if (D.fd_huc == 0) {
                k_fdh_rcnt<<<gi, 256, 0, s>>>(ha);
                RC_LAUNCH();
                RC_CUDA(cudaMemcpyAsync(&hh0[h], hst.get(), sizeof(FdhDev), cudaMemcpyDeviceToHost, s));
                RC_CUDA(cudaStreamSynchronize(s));
                rcnt = hh0[h].rcnt;
                may_recount = rcnt > 0 && (double)tw[i] > D.huc_factor * (double)rcnt;
            }
            // the levels in one graph launch: a while-node repeats select,
            // updates, sweep and close while members are alive
            GraphOwner lg;
            if (!may_recount) {
                RC_CUDA(cudaGraphCreate(&lg.g, 0));
                cudaGraphConditionalHandle cond;
                RC_CUDA(cudaGraphConditionalHandleCreate(&cond, lg.g, 1, cudaGraphCondAssignDefault));
                cudaGraphNodeParams np{};
                np.type = cudaGraphNodeTypeConditional;
                np.conditional.handle = cond;
                np.conditional.type = cudaGraphCondTypeWhile;
                np.conditional.size = 1;
                cudaGraphNode_t wnode;
                RC_CUDA(cudaGraphAddNode(&wnode, lg.g, nullptr, nullptr, 0, &np));
                cudaGraph_t body = np.conditional.phGraph_out[0];
                cudaStream_t cs = aux_stream();
                RC_CUDA(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0,
                                                      cudaStreamCaptureModeThreadLocal));
                k_fdh_select<<<gm, 256, 0, cs>>>(ha);
                RC_LAUNCH();
                k_fdh_warp<<<sms * 8, 256, 0, cs>>>(ha);
                RC_LAUNCH();
                k_fdh_cta<<<grid_h, FD_THREADS, smem_h, cs>>>(ha);
                RC_LAUNCH();
                k_fdh_sweep<<<sms * 4, 256, 0, cs>>>(ha, grid_h);
                RC_LAUNCH();
                k_fdh_next_loop<<<1, 1, 0, cs>>>(hst.get(), ni, cond);
                RC_LAUNCH();
                RC_CUDA(cudaStreamEndCapture(cs, &body));
                uncount_launches(5);  // counted per level below
                RC_CUDA(cudaGraphInstantiate(&lg.e, lg.g, 0));
                RC_CUDA(cudaGraphLaunch(lg.e, s));
            } else {
                fdh_levels_with_recount(D, ha, hst.get(), &hh0[h], rcnt, grid_h, smem_h, gm, s);
            }
            RC_CUDA(cudaMemcpyAsync(&hh0[h], hst.get(), sizeof(FdhDev), cudaMemcpyDeviceToHost, s));
            RC_CUDA(cudaStreamSynchronize(s));
            if (!may_recount) count_launches(5 * (uint64_t)hh0[h].levels);
            D.fd_heavy_ms += (float)((hh0[h].t1 - hh0[h].t0) * 1e-6);
            D.fd_heavy_levels += (int64_t)hh0[h].levels;
            D.fd_split_levels += (int64_t)hh0[h].splits;
        }
    };
    if (nheavy > 0) {
        peel_heavy(hq.data(), nheavy, nullptr);
        RC_CUDA(cudaMemcpyAsync(qhead.get(), &nheavy, 4, cudaMemcpyHostToDevice, s));
    }
    DevBuf<unsigned long long> rtip(nsmall_at < T ? n : 1, s);
    // the members' lists: walks in items of equal cost, 8 a CTA
    DevBuf<unsigned long long> rec;
    std::vector<uint8_t> skip;  // (kept until the stream has passed its copy)
    if (nheavy < T) {
        allow_max_smem((const void *)k_fd_pairs<FdMids>);
        rec.alloc(n, s);
        if (!pool.get() && (cap == 0 || !make_pool())) {
            cap = 0;  // no memory: members walk when they are peeled
            pool.alloc(1, s);
        }
        RC_CUDA(cudaMemsetAsync(rec.get(), 0xff, 8 * (size_t)n, s));
        DevBuf<unsigned long long> head(1, s);
        DevBuf<int32_t> pq(1, s);
        head.zero();
        pq.zero();
        skip.assign(T, 0);
        for (int k = 0; k < nheavy; k++) skip[hq[k]] = 1;
        DevBuf<uint8_t> dskip(T, s);
        RC_CUDA(cudaMemcpyAsync(dskip.get(), skip.data(), T, cudaMemcpyHostToDevice, s));
        unsigned long long cost = (unsigned long long)n * FP_MEMBER_COST;
        for (int k = 0; k < T; k++) cost += tw[k];
        const int64_t Q = std::max<int64_t>(8192, (int64_t)(cost / (8ull * pair_ctas)));
        const int32_t nitems = (int32_t)(cost / Q + 1);
        DevBuf<int32_t> items(nitems + 1, s);
        k_pair_items<<<ceil_div(nitems + 1, 256), 256, 0, s>>>(cw.get(), n, Q, nitems, items.get());
        RC_LAUNCH();
        FdPairArgs a{d_tstart.get(), d_tlen.get(), d_tkb.get(), dskip.get(), T, items.get(), nitems,
                     pq.get(), info.get(), fd_adj.get(), pool.get(), cap, head.get(), rec.get(),
                     stats.get()};
        if (cap > 0) {
            k_fd_pairs<<<std::min(pair_ctas, nitems), FP_THREADS, FP_WARPS * FP_WORDS * 4, s>>>(
                a, FdMids{fd_beg.get(), fd_len.get()});
            RC_LAUNCH();
        }
    }
    // tasks that go over to all CTAs after all (automatic rule)
    DevBuf<int32_t> over(T > 0 ? T : 1, s);
    DevBuf<unsigned long long> over_level(T > 0 ? T : 1, s);
    const FdHandOver ho{D.fd_heavy_w == 0 ? dtw.get() : nullptr, (int32_t *)(stats.get() + 2),
                        over.get(), over_level.get()};
    // large and small tasks side by side
    const int nlarge = nsmall_at - nheavy, nsmall = T - nsmall_at;
    cudaEvent_t fork_ev[2] = {};
    cudaStream_t ls = s;  // the large tasks' stream
    struct ForkGuard {
        cudaEvent_t *e;
        cudaStream_t &ls;
        bool joined = true;  // else the buffers wait for the other stream
        ~ForkGuard() {
            if (!joined) cudaStreamSynchronize(ls);
            for (int k = 0; k < 2; k++)
                if (e[k]) cudaEventDestroy(e[k]);
        }
    } fg{fork_ev, ls};
    if (nlarge > 0 && nsmall > 0) {
        for (cudaEvent_t &e : fork_ev) RC_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        ls = tier_stream(0);
        RC_CUDA(cudaEventRecord(fork_ev[0], s));
        RC_CUDA(cudaStreamWaitEvent(ls, fork_ev[0], 0));
        fg.joined = false;
    }
    if (nlarge > 0) {
        const int grid = std::max(1, std::min(grid_all, nlarge));
        FdArgs a{queue.get(),   nsmall_at,   qhead.get(),     d_tstart.get(), d_tlen.get(),
                 d_tkb.get(),   members.get(), fd_beg.get(), fd_len.get(),   fd_adj.get(), S.new2old,
                 D.init,        fsup.get(),  alive.get(),     alist.get(),  alist2.get(),
                 clist.get(),   clist2.get(),
                 plist.get(),   info.get(),   pool.get(),      rec.get(),
                 (unsigned long long *)d_tip, stats.get(),    sub_ns.get(), sub_lv.get(), ho};
        k_fd_peel<<<grid, FD_THREADS, smem, ls>>>(a);
        RC_LAUNCH();
    }
    if (nsmall > 0) {
        allow_max_smem((const void *)k_fd_small);
        FsArgs a{queue.get() + nsmall_at, nsmall, qhead.get() + 1, d_tstart.get(), d_tlen.get(),
                 d_tkb.get(), members.get(), info.get(), pool.get(), rec.get(), fd_beg.get(),
                 fd_len.get(), fd_adj.get(), S.new2old, D.init, rtip.get(), (unsigned long long *)d_tip,
                 fsup.get(), alive.get(), stats.get(), sub_ns.get(), sub_lv.get(), ho};
        k_fd_small<<<std::min(sms, nsmall), FD_THREADS, FS_SMEM, s>>>(a);
        RC_LAUNCH();
    }
    if (ls != s) {
        RC_CUDA(cudaEventRecord(fork_ev[1], ls));
        RC_CUDA(cudaStreamWaitEvent(s, fork_ev[1], 0));
        fg.joined = true;
    }
    unsigned long long hs[3] = {0, 0, 0};
    RC_CUDA(cudaMemcpyAsync(hs, stats.get(), sizeof(hs), cudaMemcpyDeviceToHost, s));
    std::vector<unsigned long long> hns(T), hlv(T);
    if (T > 0) {
        RC_CUDA(cudaMemcpyAsync(hns.data(), sub_ns.get(), 8 * (size_t)T, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaMemcpyAsync(hlv.data(), sub_lv.get(), 8 * (size_t)T, cudaMemcpyDeviceToHost, s));
    }
    RC_CUDA(cudaStreamSynchronize(s));
    const int32_t nover = (int32_t)(hs[2] >> 32);
    if (nover > 0) {
        std::vector<int32_t> ids(nover);
        RC_CUDA(cudaMemcpyAsync(ids.data(), over.get(), 4 * (size_t)nover, cudaMemcpyDeviceToHost, s));
        RC_CUDA(cudaStreamSynchronize(s));
        pool.release();
        peel_heavy(ids.data(), nover, over_level.get());
        D.fd_heavy += nover;
    }
    D.wedges_fd = hs[0];
    D.levels = (int64_t)hs[1];
    std::vector<bool> heavy(T, false);
    for (size_t h = 0; h < hh.size(); h++) {
        const int32_t t = heavy_tasks[h];
        heavy[t] = true;
        D.fd_heavy_levels += (int64_t)hlv[t];  // before it was handed over
        hns[t] += hh[h].t1 - hh[h].t0;
        hlv[t] += hh[h].levels;
        D.wedges_fd += hh[h].wedges;
        D.levels += (int64_t)hh[h].levels;
    }
    // per subset: its tasks' levels and device time summed
    D.subsets.assign(P, receipt_subset{});
    for (int i = 0; i < P; i++) {
        D.subsets[i].n = hms[i + 1] - hms[i];
        D.subsets[i].wedges_est = hw[i];
    }
    int worst = -1;
    for (int t = 0; t < T; t++) {
        receipt_subset &r = D.subsets[tsub[t]];
        r.levels += (int64_t)hlv[t];
        r.ms += (float)(hns[t] * 1e-6);
        if (heavy[t]) r.heavy = 1;
        if (!heavy[t] && (worst < 0 || hns[t] > hns[worst])) worst = t;
    }
    // slowest task peeled by one CTA
    D.fd_max_ms = worst >= 0 ? (float)(hns[worst] * 1e-6) : 0.f;
    D.fd_max_n = worst >= 0 ? tlen[worst] : 0;
    D.fd_max_levels = worst >= 0 ? (int64_t)hlv[worst] : 0;
    D.fd_tasks = T;
}

namespace {

// Middle vertices of a side's vertices, whole lists.
struct SideMids {
    static constexpr bool LARGE_FIRST = true;
    const int32_t *adj_s;
    const int64_t *off_o;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        const int32_t y = adj_s[q];
        beg = off_o[y];
        len = (int32_t)(off_o[y + 1] - beg);
    }
};

__global__ void k_side_members(const int64_t *__restrict__ off_s,
                               const unsigned long long *__restrict__ wfull, int32_t n, int64_t add,
                               FdMember *__restrict__ info, int64_t *__restrict__ cost) {
    const int32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const unsigned long long w = wfull[x];
    info[x] = FdMember{off_s[x], (int32_t)(off_s[x + 1] - off_s[x]),
                       (uint32_t)(w < 0xffffffffull ? w : 0xffffffffull)};
    cost[x] = (int64_t)w + add;
}

}  // namespace

bool side_pair_lists(const Decomp &D, PairLists &L, cudaStream_t s) {
    const int32_t n = D.n;
    const int64_t m = D.m;
    if (n > FP_MAX_NI || m == 0) return false;
    const int T = D.parts ? (int)D.parts->size() - 1 : 1;
    std::vector<int32_t> ts(T), tl(T);
    for (int t = 0; t < T; t++) {
        ts[t] = D.parts ? (int32_t)(*D.parts)[t] : 0;
        tl[t] = (D.parts ? (int32_t)(*D.parts)[t + 1] : n) - ts[t];
    }
    // every vertex must get a list (fd_plan): 16-bit counters of all keys in eight
    // times a CTA's words, counts above the rank bits
    const int32_t keys = *std::max_element(tl.begin(), tl.end());
    if ((int64_t)keys * 16 > (int64_t)32 * 8 * FP_WARPS * FP_WORDS || D.max_deg_s >= 65536 ||
        (int64_t)D.max_deg_s >= 1ll << (32 - bits_for((uint64_t)std::max(1, keys - 1))))
        return false;
    const int ctas = 2 * num_sms();
    const unsigned long long w = D.wedges_bup + (unsigned long long)m;  // sum of wfull
    // room for all lists
    unsigned long long most = 0;
    for (int t = 0; t < T; t++) most += lists_at_most(w, tl[t]);
    most = std::min(most, w / 2);
    const unsigned long long small = (unsigned long long)(FD_LIST_BYTES / 4 * m);
    const unsigned long long cap =
        (most <= small
             ? most
             : std::min(most, std::max(small, (unsigned long long)available_bytes() / 32))) +
        (unsigned long long)ctas * FP_WARPS * FP_BLOCK;
    DevBuf<FdMember> info(n, s);
    DevBuf<int64_t> cost(n + 1, s), cw(n + 1, s);
    DevBuf<int32_t> dts(T, s), dtl(T, s), pq(1, s);
    DevBuf<uint8_t> skip(T, s);
    DevBuf<unsigned long long> scal(2, s);  // pool head, wedges
    RC_CUDA(cudaMemcpyAsync(dts.get(), ts.data(), 4 * (size_t)T, cudaMemcpyHostToDevice, s));
    RC_CUDA(cudaMemcpyAsync(dtl.get(), tl.data(), 4 * (size_t)T, cudaMemcpyHostToDevice, s));
    skip.zero();
    scal.zero();
    pq.zero();
    RC_CUDA(cudaMemsetAsync(cost.get() + n, 0, 8, s));
    k_side_members<<<ceil_div(n, 256), 256, 0, s>>>(D.S->off, D.wfull, n, FP_MEMBER_COST, info.get(),
                                                    cost.get());
    RC_LAUNCH();
    scan_exclusive<int64_t>(cost.get(), cw.get(), n + 1, s);
    const unsigned long long total = w + (unsigned long long)n * FP_MEMBER_COST;
    const int64_t Q = std::max<int64_t>(8192, (int64_t)(total / (8ull * ctas)));
    const int32_t nitems = (int32_t)(total / Q + 1);
    DevBuf<int32_t> items(nitems + 1, s);
    k_pair_items<<<ceil_div(nitems + 1, 256), 256, 0, s>>>(cw.get(), n, Q, nitems, items.get());
    RC_LAUNCH();
    if (!L.pool.try_alloc((size_t)cap, s) || !L.rec.try_alloc(n, s)) {
        L.pool.release();
        return false;
    }
    allow_max_smem((const void *)k_fd_pairs<SideMids>);
    // keys are vertices: a task's first key is its first vertex
    FdPairArgs a{dts.get(), dtl.get(), dts.get(), skip.get(), T, items.get(), nitems, pq.get(),
                 info.get(), D.O->adj, L.pool.get(), cap, scal.get(), L.rec.get(), scal.get() + 1};
    k_fd_pairs<<<std::min(ctas, nitems), FP_THREADS, FP_WARPS * FP_WORDS * 4, s>>>(
        a, SideMids{D.S->adj, D.O->off});
    RC_LAUNCH();
    unsigned long long head = 0;
    RC_CUDA(cudaMemcpyAsync(&head, scal.get(), 8, cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    if (head <= cap) return true;
    L.pool.release();
    L.rec.release();
    return false;
}

}  // namespace receipt
