// The coarse-grained decomposition (Algorithm 3) in one cooperative launch.
//
// A round of a small side is a chain of short steps: the per-round kernels of
// cd.cu spend ~28 us on a round and ~65 us on a range's start whatever their
// size (kernel edges of a graph, a host round trip per range). Here one
// launch runs every range: the CTAs stay resident and meet at a grid barrier
// (~1.5 us) between the steps,
//   range start: supports -> weighted histogram, init <- support, and, when
//                due, the lists' compaction (Sec. 4.2);         barrier
//   bound:       every CTA evaluates findHi on the same histogram;
//   activeSet:   scan of the remaining vertices, which assigns them to the
//                subset and lists their anchors by tier;         barrier
//   peel:        updates of the listed anchors;                  barrier
// with the last two repeated until the activeSet is empty. Sides whose key
// space (or, in a union of packed graphs, every graph's) fits one dense
// window take this form: their anchors need only the warp table and the
// dense-window engine. Same ranges, rounds and counters as cd.cu.
//
// Three forms of the peel: dense windows, a CTA per item; groups of warps for
// sides with short walks (cd_persist_wide); and, on sides small enough to make
// every vertex's list of updates beforehand (cd_persist_by_lists), reading those
// lists, which leaves a round two dependent loads and no walk. Each is a kernel
// of its own: the groups' code and lists alone cost the others (256 packed
// graphs: 44 ms without, 47 with).
//
// What bounds it: the latency of a round's chain of dependent steps. On a
// 20,000 x 5,000 graph of 200k edges (V side, 312 rounds in 149 ranges; us):
// scan 3.4, barrier 1.9, counters and first item 1.6, walk 4.3, sweep 1.2,
// barrier 2.1; bound 3.3 a range. That call took 17.4 ms by the per-round
// kernels, 7.0 by windows and takes 5.4 by lists; 2,000 x 500 with 20k edges 5.3,
// 2.4 (2.2 by groups) and 1.9; 30,000 x 9,000 with 300k edges from host buffers
// 20.1, 9.7 and 7.0; 256 packed graphs 76, 44 and 36.5.
//
// What changes during the launch (supports, subsets, working lists, the
// activeSet) is read from L2 (ld.cg): another CTA may have written it since
// this SM last cached the line.
#include <algorithm>

#include "cd.cuh"

namespace receipt {

namespace {

constexpr int PT = 512;  // threads per CTA (two CTAs per SM)
constexpr int GROUP = 8;  // dense-window anchors side by side in one pass
// With groups (WIDE), walks of more wedges still take the whole CTA. (8,192, this or
// 131,072: the same within 2% on five sides of 500k to 5M edges; the wedge counts
// of the groups' counters end near here. So are the classes' thresholds, half or
// four times as high: 5% on uniform graphs of 5M edges.)
constexpr unsigned long long GROUP_MAX_W = 32768;
// Polls of a barrier wait before it gives up (each takes at least an L2 round
// trip: ~10 s in all). CTAs fetch their items as they go, so they wait for one
// another's last fetch at most: GROUP_W wedges (1.6 s at the 1.6 10^9 wedges a
// second of a CTA on dense graphs), or one anchor's walk, 65,534 lists of 36,864
// keys at most and no longer.
constexpr unsigned BAR_POLLS = 1u << 24;
constexpr uint64_t GROUP_W = 2500000000ull;

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// All CTAs of the (cooperative) launch meet here; `target` counts arrivals.
// False when the wait ran out; every CTA then leaves.
__device__ bool grid_barrier(PersistDev *pd, unsigned &target, int *s_ok) {
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&pd->bar, 1u);
        unsigned polls = 0;
        while ((int)(ld_acquire(&pd->bar) - target) < 0 && polls < BAR_POLLS) polls++;
        if (polls == BAR_POLLS) {
            pd->err = 1;
            *s_ok = 0;
        }
        __threadfence();
    }
    __syncthreads();
    return *s_ok != 0;
}

// Warp-private table of the warp tier in the dense engine's counters, which
// are all zero between passes: key + 1 per slot, 0 = empty.
struct WarpTable {
    uint32_t *key, *val;  // WARP_SLOTS each
    __device__ __forceinline__ void add(int32_t k) {
        const uint32_t kk = (uint32_t)k + 1u;
        uint32_t h = hash_key(k) & (WARP_SLOTS - 1);
        for (int p = 0; p < WARP_SLOTS; p++) {
            uint32_t cur = ((volatile uint32_t *)key)[h];
            if (cur == 0u) {
                cur = atomicCAS(&key[h], 0u, kk);
                if (cur == 0u) cur = kk;
            }
            if (cur == kk) {
                atomicAdd(&val[h], 1u);
                return;
            }
            h = (h + 1) & (WARP_SLOTS - 1);
        }
    }
    template <class Emit>
    __device__ __forceinline__ void flush_clear(Emit &emit, int lane) {
        for (int s0 = 0; s0 < WARP_SLOTS; s0 += 32 * 8) {
            int32_t kk[8];
            uint32_t cc[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int sl = s0 + u * 32 + lane;
                const uint32_t k = key[sl];
                cc[u] = val[sl];
                kk[u] = cc[u] >= 2 ? (int32_t)(k - 1u) : -1;
                if (k) {
                    key[sl] = 0;
                    val[sl] = 0;
                }
            }
            emit_many<8>(emit, kk, cc);
        }
    }
};
static_assert(PT / 32 * WARP_SLOTS * 2 <= DENSE_WORDS, "warp tables fit the dense counters");
static_assert(PT == FP_WARPS * 32 && FP_WARPS * FP_WORDS <= DENSE_WORDS, "group counters");
static_assert(3 * NBUCKET <= DENSE_WORDS, "range histogram fits the dense counters");

// Support decrements of remaining vertices (N at once so the loads overlap).
struct PersistEmit {
    unsigned long long *sup;
    const int32_t *sub;
    unsigned long long pairs;
    template <int N>
    __device__ __forceinline__ void many(const int32_t (&k)[N], const uint32_t (&c)[N]) {
        bool live[N];
#pragma unroll
        for (int u = 0; u < N; u++) live[u] = k[u] >= 0 && __ldcg(sub + k[u]) < 0;
#pragma unroll
        for (int u = 0; u < N; u++)
            if (live[u]) {
                pairs++;
                atomicAdd(&sup[k[u]], 0ull - choose2(c[u]));
            }
    }
};

struct PersistMids {
    const int32_t *adj_s;
    const int64_t *off_o;
    const int32_t *len_o;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        const int32_t y = adj_s[q];
        beg = off_o[y];
        len = __ldcg(len_o + y);
    }
};

// Entries below `key` of the ascending working list L[0..n).
__device__ __forceinline__ int32_t lower_bound_l2(const int32_t *L, int32_t n, int32_t key) {
    int32_t lo = 0, hi = n;
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (__ldcg(L + mid) < key)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Middle vertices of up to GROUP anchors as one virtual list; the staging
// thread records which anchor its middle vertex belongs to.
struct PersistGroup {
    int64_t q0[GROUP];
    int32_t x[GROUP], kb[GROUP], ke[GROUP], part[GROUP], off[GROUP + 1], pre[GROUP + 1];
    uint8_t slot[PT];
};

struct GroupMids {
    PersistMids M;
    const int32_t *adj_o;
    PersistGroup *g;
    int nb;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        int a = 0;
        while (a + 1 < nb && g->pre[a + 1] <= q) a++;
        M.seg(g->q0[a] + (q - g->pre[a]), beg, len);
        if (g->part[a] >= 0 && len > 64) {
            // a long list and one window of several: only its keys in the
            // window (a short list is walked whole, the visits filter)
            const int32_t lo = lower_bound_l2(adj_o + beg, len, g->kb[a]);
            len = lower_bound_l2(adj_o + beg + lo, len - lo, g->ke[a]);
            beg += lo;
        }
        g->slot[threadIdx.x] = (uint8_t)a;
    }
};

struct GroupVisit {
    DenseSlice *eng;
    const PersistGroup *g;
    __device__ __forceinline__ void operator()(int k, int32_t key) {
        // keys outside the window belong to the anchor's other items or (past
        // the last one) are assigned vertices still in the lists
        const int a = g->slot[k];
        if (key >= g->kb[a] && key < g->ke[a] && key != g->x[a]) eng->add(g->off[a] + key - g->kb[a]);
    }
};

// One item alone in its pass: its constants stay in registers.
struct OneMids {
    PersistMids M;
    const int32_t *adj_o;
    int64_t q0;
    int32_t kb, ke;
    bool sliced;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        M.seg(q0 + q, beg, len);
        if (sliced && len > 64) {
            const int32_t lo = lower_bound_l2(adj_o + beg, len, kb);
            len = lower_bound_l2(adj_o + beg + lo, len - lo, ke);
            beg += lo;
        }
    }
};

struct OneVisit {
    DenseSlice *eng;
    int32_t x, kb, ke;
    __device__ __forceinline__ void operator()(int, int32_t key) {
        if (key >= kb && key < ke && key != x) eng->add(key - kb);
    }
};

struct OneEmit {
    PersistEmit *e;
    int32_t kb;
    template <int N>
    __device__ __forceinline__ void many(const int32_t (&k)[N], const uint32_t (&c)[N]) {
        int32_t kk[N];
#pragma unroll
        for (int u = 0; u < N; u++) kk[u] = k[u] >= 0 ? k[u] + kb : -1;
        e->template many<N>(kk, c);
    }
};

struct GroupEmit {
    PersistEmit *e;
    const PersistGroup *g;
    int nb;
    template <int N>
    __device__ __forceinline__ void many(const int32_t (&k)[N], const uint32_t (&c)[N]) {
        int32_t kk[N];
#pragma unroll
        for (int u = 0; u < N; u++) {
            int a = 0;
            while (a + 1 < nb && g->off[a + 1] <= k[u]) a++;
            kk[u] = k[u] >= 0 ? g->kb[a] + k[u] - g->off[a] : -1;
        }
        e->template many<N>(kk, c);
    }
};

// Position of every lane with `take` in a list counted by *cnt.
__device__ __forceinline__ int warp_slot(bool take, int32_t *cnt) {
    const unsigned bal = __ballot_sync(0xffffffffu, take);
    if (!bal) return 0;
    const int leader = __ffs(bal) - 1;
    int pos = 0;
    if ((threadIdx.x & 31) == leader) pos = atomicAdd(cnt, __popc(bal));
    return __shfl_sync(0xffffffffu, pos, leader) + __popc(bal & lanemask_lt());
}

// Drops the vertices assigned before `range` from every working list (one
// warp per list, in place: the write position never passes the read
// position); those that the running scan assigns to `range` stay.
__device__ void compact_working_lists(const PersistArgs &a, int32_t range, int64_t warp,
                                      int64_t nwarps, int lane) {
    for (int64_t y = warp; y < a.n_o; y += nwarps) {
        const int64_t b = a.off_o[y];
        const int32_t l = __ldcg(a.len_o + y);
        int32_t w = 0;
        for (int32_t r0 = 0; r0 < l; r0 += 128) {
            int32_t x[4];
            bool keep[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int32_t r = r0 + 32 * u + lane;
                x[u] = r < l ? __ldcg(a.adj_o + b + r) : -1;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int32_t sb = x[u] >= 0 ? __ldcg(a.sub + x[u]) : 0;
                keep[u] = x[u] >= 0 && (sb < 0 || sb == range);
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const unsigned bal = __ballot_sync(0xffffffffu, keep[u]);
                if (keep[u]) a.adj_o[b + w + __popc(bal & lanemask_lt())] = x[u];
                w += __popc(bal);
            }
            __syncwarp();
        }
        if (lane == 0) a.len_o[y] = w;
    }
}

// Bits of a range's histogram that a CTA gathers in its dense counters.
struct HistSmem {
    unsigned long long *w;
    uint32_t *c;
    __device__ __forceinline__ void add(unsigned long long v, unsigned long long weight) {
        const int b = log_bucket_of(v);
        atomicAdd(&c[b], 1u);
        if (weight) atomicAdd(&w[b], weight);
    }
    // Adds the gathered buckets to the global histogram and clears them.
    __device__ __forceinline__ void flush(unsigned long long *gw, uint32_t *gc) {
        for (int b = threadIdx.x; b < NBUCKET; b += PT) {
            const uint32_t n = c[b];
            if (n == 0) continue;
            const unsigned long long s = w[b];
            atomicAdd(gc + b, n);
            if (s) atomicAdd(gw + b, s);
            c[b] = 0;
            w[b] = 0;
        }
    }
};

__device__ __forceinline__ PersistAnchor load_anchor(const PersistAnchor *p) {
    PersistAnchor an;
    const int4 lo = __ldcg((const int4 *)p), hi = __ldcg((const int4 *)p + 1);
    an.q0 = ((int64_t)(uint32_t)lo.x) | ((int64_t)lo.y << 32);
    an.x = lo.z;
    an.deg = lo.w;
    an.kb = hi.x;
    an.w = hi.y;
    an.part = hi.z;
    an.wedges = (uint32_t)hi.w;
    return an;
}

// Updates of the anchors listed in classes [c0, c1] (na[c] each), a group of
// at least `need` warps per anchor: as many as leave every anchor a group.
// words: FP_WARPS * FP_WORDS zeroed counter words, zero again on return. cw, cm,
// ca: wedges (all lanes), middle vertices and anchors (lane 0 of a group's
// first warp).
__device__ __forceinline__ void group_items(const PersistArgs &a, const PersistMids &M,
                                            uint32_t *words, int c0, int c1, const int (&na)[3],
                                            int need, PersistEmit &emit, unsigned long long &cw,
                                            unsigned long long &cm, unsigned long long &ca) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int n = 0;
    for (int c = c0; c <= c1; c++) n += na[c];
    int g = need;
    while (g < FP_WARPS && (int64_t)n * 2 * g <= (int64_t)FP_WARPS * gridDim.x) g *= 2;
    const int grp = warp / g, part = warp & (g - 1);
    uint32_t *w = words + grp * g * FP_WORDS;
    for (int i = grp * gridDim.x + blockIdx.x; i < n; i += gridDim.x * (FP_WARPS / g)) {
        int c = c0, j = i;
        while (j >= na[c]) j -= na[c++];
        const PersistAnchor an = load_anchor(a.Lg + (size_t)c * a.n + j);
        const FpPlan pl = fp_plan(an.deg, an.wedges, an.w);
        const uint32_t wmask = (1u << pl.lw) - 1u;
        const int32_t ke = an.kb + an.w;
        // keys past the window are assigned vertices still in the lists
        if (pl.bits) {
            auto add = [&](int32_t key) {
                cw++;
                if (key < an.kb || key >= ke || key == an.x) return;
                const int32_t k = key - an.kb;
                atomicAdd(&w[k & wmask], 1u << ((k >> pl.lw) * pl.bits));
            };
            warp_walk<4, KeysL2>(M, an.q0, an.q0 + an.deg, a.adj_o, add, part, g);
        } else {
            auto add = [&](int32_t key) {
                cw++;
                if (key >= an.kb && key < ke && key != an.x) fp_table_add(w, wmask, key - an.kb);
            };
            warp_walk<4, KeysL2>(M, an.q0, an.q0 + an.deg, a.adj_o, add, part, g);
        }
        fp_sync(grp, g);
        for (uint32_t sl = part * 32 + lane; sl <= wmask / 4; sl += 32 * g) {
            const uint4 v = ((const uint4 *)w)[sl];
            if (!(v.x | v.y | v.z | v.w)) continue;
            ((uint4 *)w)[sl] = make_uint4(0, 0, 0, 0);
            const uint32_t e[4] = {v.x, v.y, v.z, v.w};
            if (pl.bits == 0) {
                int32_t k[4];
                uint32_t cc[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    cc[u] = e[u] & 1023u;
                    k[u] = cc[u] >= 2 ? an.kb + (int32_t)(e[u] >> 10) - 1 : -1;
                }
                emit.many<4>(k, cc);
                continue;
            }
#pragma unroll
            for (int x = 0; x < 4; x++) {
                uint32_t f = fp_repeats(e[x], pl.bits);
                while (f) {
                    int32_t k[4];
                    uint32_t cc[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int b = f ? __ffs(f) - 1 : 0;
                        cc[u] = (e[x] >> b) & (0xffffffffu >> (32 - pl.bits));
                        k[u] = f ? an.kb + (int32_t)(4 * sl + x) + ((b / pl.bits) << pl.lw) : -1;
                        f &= f - 1;
                    }
                    emit.many<4>(k, cc);
                }
            }
        }
        fp_sync(grp, g);
        if (part == 0 && lane == 0) {
            cm += (unsigned long long)an.deg;
            ca++;
        }
    }
    __syncthreads();
}

template <int FORM>
__global__ void __launch_bounds__(PT, 2) k_cd_persist(PersistArgs a) {
    constexpr bool WIDE = FORM == PERSIST_GROUPS, LISTS = FORM == PERSIST_LISTS;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_ok, s_nt, s_idx, s_nb, s_pick, s_first, s_last, s_nF, s_due;
    __shared__ unsigned long long s_tmp[33], s_goal, s_wrem, s_peeled;
    __shared__ uint32_t s_tmpc[33];
    __shared__ double s_tgt;
    __shared__ PersistGroup s_g;
    __shared__ uint32_t s_tier[8];  // a CTA's counters of a round by lists, per tier
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // global numbers with the CTA index fastest: a few items spread over CTAs
    const int gwarp = warp * gridDim.x + blockIdx.x, nwarps = (PT / 32) * gridDim.x;
    const int32_t gthread = blockIdx.x * PT + threadIdx.x, nthreads = gridDim.x * PT;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    // One graph: the scan for the activeSet also gathers the histogram of the
    // vertices it leaves, so that the scan which ends a range (it finds
    // nothing) starts the next one. In a union the scans are long and the
    // rounds many: a pass of its own per range.
    const bool fused = a.part_of == nullptr;
    DenseSlice H;
    unsigned char *p = H.bind(smem, &s_nt);
    Chunk ch;
    ch.beg = (int64_t *)p;
    ch.pre = (int32_t *)(ch.beg + PT);
    ch.tmp = ch.pre + PT + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    H.clear_all();
    HistSmem hist{(unsigned long long *)H.cnt, (uint32_t *)(H.cnt + 2 * NBUCKET)};
    PersistDev *pd = a.pd;
    CdDev *st = a.st;
    // the loop's state, the same in every CTA
    int mode = pd->mode, range = pd->range, sk = pd->sk, nrec = pd->nrec, hk = pd->hk;
    int dgm_passes = pd->dgm_passes;
    bool first = mode == PERSIST_PEEL, compact = false;
    unsigned long long hi = pd->hi, peeled = pd->peeled, peeled_at_dgm = pd->peeled_at_dgm;
    // last remaining vertex when the range began (one graph)
    int32_t last = fused && mode != PERSIST_RANGE ? a.n - 1 : -1;
    if (threadIdx.x < 8) s_tier[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        s_ok = 1;
        s_wrem = pd->wrem_prev;
        s_tgt = pd->tgt_prev;
    }
    unsigned target = 0;
    int stop = PERSIST_DONE;
    PersistMids M{a.adj_s, a.off_o, a.len_o};
    __syncthreads();
    // Buffers of histogram number k; the next one's are cleared meanwhile
    // (number k - 1 may still be read by a CTA that has yet to choose a bound).
    auto clear_next = [&](int k) {
        const size_t z = (size_t)((k + 1) % 3);
        for (int32_t b = gthread; b < NBUCKET; b += nthreads) {
            a.hist_w[z * NBUCKET + b] = 0;
            a.hist_c[z * NBUCKET + b] = 0;
        }
        for (int32_t b = gthread; b < a.nparts; b += nthreads) a.plast[z * a.nparts + b] = -1;
    };
    for (;;) {
        if (mode == PERSIST_RANGE) {
            if (range >= a.P) break;
            if (!fused || hk == 0) {
                // ---- histogram of the remaining supports
                int32_t *plast = a.plast + (size_t)(hk % 3) * a.nparts;
                for (int32_t b0 = blockIdx.x * PT; b0 < a.n; b0 += 4 * nthreads) {
                    int32_t x[4], sb[4];
                    unsigned long long v[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        x[u] = b0 + u * nthreads + threadIdx.x;
                        sb[u] = x[u] < a.n ? __ldcg(a.sub + x[u]) : 0;
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) v[u] = sb[u] < 0 ? __ldcg(a.sup + x[u]) : 0;
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const bool live = sb[u] < 0;
                        if (live)
                            hist.add(v[u], a.wfull[x[u]] - (unsigned long long)(a.off_s[x[u] + 1] -
                                                                                a.off_s[x[u]]));
                        const int32_t pt = live && a.part_of ? a.part_of[x[u]] : 0;
                        const unsigned act = __ballot_sync(0xffffffffu, live);
                        if (act) {
                            const int32_t p0 = __shfl_sync(0xffffffffu, pt, __ffs(act) - 1);
                            if (__all_sync(0xffffffffu, !live || pt == p0)) {
                                if (lane == 31 - __clz(act)) atomicMax(plast + p0, x[u]);
                            } else if (live) {
                                atomicMax(plast + pt, x[u]);
                            }
                        }
                    }
                }
                __syncthreads();
                hist.flush(a.hist_w + (size_t)(hk % 3) * NBUCKET, a.hist_c + (size_t)(hk % 3) * NBUCKET);
                clear_next(hk);
                hk++;
                if (!grid_barrier(pd, target, &s_ok)) return;
            }
            // ---- findHi with the adaptive target, as k_cd_select
            const unsigned long long *gw = a.hist_w + (size_t)((hk - 1) % 3) * NBUCKET;
            const uint32_t *gc = a.hist_c + (size_t)((hk - 1) % 3) * NBUCKET;
            constexpr int PER = (NBUCKET + PT - 1) / PT;
            static_assert(NBUCKET % PER == 0 && PER == 4, "vector loads of the histogram");
            unsigned long long w[PER] = {}, wsum = 0;
            uint32_t c[PER] = {}, csum = 0;
            if (threadIdx.x * PER < NBUCKET) {
                const uint4 c4 = __ldcg((const uint4 *)(gc + threadIdx.x * PER));
                const ulonglong2 w0 = __ldcg((const ulonglong2 *)(gw + threadIdx.x * PER));
                const ulonglong2 w1 = __ldcg((const ulonglong2 *)(gw + threadIdx.x * PER) + 1);
                c[0] = c4.x, c[1] = c4.y, c[2] = c4.z, c[3] = c4.w;
                w[0] = w0.x, w[1] = w0.y, w[2] = w1.x, w[3] = w1.y;
            }
            if (fused) last = __ldcg(a.plast + (hk - 1) % 3);
#pragma unroll
            for (int j = 0; j < PER; j++) {
                wsum += w[j];
                csum += c[j];
            }
            // one scan of both sums: warps, then the warps' totals in every thread
            unsigned long long wi = wsum;
            uint32_t ci = csum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long yw = __shfl_up_sync(0xffffffffu, wi, o);
                const uint32_t yc = __shfl_up_sync(0xffffffffu, ci, o);
                if (lane >= o) {
                    wi += yw;
                    ci += yc;
                }
            }
            if (lane == 31) {
                s_tmp[warp] = wi;
                s_tmpc[warp] = ci;
            }
            if (threadIdx.x == 0) {
                s_pick = s_first = NBUCKET;
                s_last = -1;
            }
            __syncthreads();
            unsigned long long wrun = wi - wsum, wtot = 0;
            uint32_t crun = ci - csum, ctot = 0;
#pragma unroll
            for (int k = 0; k < PT / 32; k++) {
                if (k < warp) {
                    wrun += s_tmp[k];
                    crun += s_tmpc[k];
                }
                wtot += s_tmp[k];
                ctot += s_tmpc[k];
            }
            if (ctot == 0) break;  // nothing remains
            if (threadIdx.x == 0) {
                // one thread: 64-bit floating point is slow on this chip
                double s_prev = 1.0;
                if (range > 0) {
                    const unsigned long long covered = s_wrem - wtot;
                    if (covered > 0) s_prev = fmin(1.0, s_tgt / (double)covered);
                }
                s_tgt = s_prev * (double)wtot / (double)(a.P - range);
                s_wrem = wtot;
                s_goal = target_weight(s_tgt);
            }
            __syncthreads();
            const unsigned long long goal = s_goal;
            int mine = NBUCKET, lo_b = NBUCKET, hi_b = -1;
#pragma unroll
            for (int j = 0; j < PER; j++) {
                const int b = threadIdx.x * PER + j;
                wrun += w[j];
                crun += c[j];
                if (c[j]) {
                    lo_b = min(lo_b, b);
                    hi_b = b;
                    if (wrun >= goal || (a.range_cap > 0 && crun >= (uint32_t)a.range_cap))
                        mine = min(mine, b);
                }
            }
            if (hi_b >= 0) {
                atomicMin(&s_first, lo_b);
                atomicMax(&s_last, hi_b);
                if (mine < NBUCKET) atomicMin(&s_pick, mine);
            }
            __syncthreads();
            int b = s_pick;
            if (goal == 0) b = s_first;
            if (b >= NBUCKET) b = s_last;
            const unsigned long long top = log_bucket_top(b);
            hi = top == ~0ull ? ~0ull : top + 1ull;
            first = true;
            mode = PERSIST_SCAN;
        }
        if (mode == PERSIST_SCAN) sk++;
        PersistDev::Set *set = &pd->set[sk % 3];
        if (mode == PERSIST_SCAN) {
            if (lead) pd->set[(sk + 1) % 3] = PersistDev::Set{};
            // ---- activeSet: remaining vertices with support < hi; a range's
            // first scan sees the supports the range began with
            const int32_t *plast = a.plast + (size_t)((hk + 2) % 3) * a.nparts;
            // a range's first scan takes at least one vertex: not its last
            const bool gather = fused && !first;
            unsigned long long fw = 0, fe = 0, uw = 0;
            int32_t live_last = -1;
            for (int32_t b0 = blockIdx.x * PT; b0 < a.n; b0 += 4 * nthreads) {
                int32_t x[4], sb[4];
                unsigned long long v[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    x[u] = b0 + u * nthreads + threadIdx.x;
                    sb[u] = x[u] < a.n ? __ldcg(a.sub + x[u]) : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; u++) v[u] = sb[u] < 0 ? __ldcg(a.sup + x[u]) : ~0ull;
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const bool live = sb[u] < 0, take = live && v[u] < hi;
                    if (first && live) a.init[x[u]] = v[u];
                    if (gather && live && !take) {
                        hist.add(v[u], a.wfull[x[u]] - (unsigned long long)(a.off_s[x[u] + 1] -
                                                                            a.off_s[x[u]]));
                        live_last = max(live_last, x[u]);
                    }
                    if (!__any_sync(0xffffffffu, take)) continue;
                    PersistAnchor an{0, x[u], 0, 0, 0, -1, 0};
                    int cls = -1;
                    unsigned long long wf = 0;
                    if (take) {
                        wf = a.wfull[x[u]];
                        an.q0 = a.off_s[x[u]];
                        an.deg = (int32_t)(a.off_s[x[u] + 1] - an.q0);
                        if (fused) {
                            an.w = last + 1;
                        } else {
                            const int32_t pt = a.part_of[x[u]];
                            an.kb = a.pfirst[pt];
                            an.w = __ldcg(plast + pt) - an.kb + 1;
                        }
                        a.sub[x[u]] = range;
                        fw += wf;
                        fe += (unsigned long long)an.deg;
                        if (v[u]) uw += wf;
                        if (WIDE && v[u] && wf > (unsigned long long)a.warp_max_w &&
                            wf <= GROUP_MAX_W) {
                            an.wedges = (uint32_t)wf;
                            const FpPlan pl = fp_plan(an.deg, an.wedges, an.w);
                            // a round waits for its longest walk
                            const int load = max((int)(wf >> 10), an.deg >> 6);
                            cls = pl.lw > 14              ? -1
                                  : pl.g == 1 && load < 1 ? 0
                                  : pl.g <= 4 && load < 4 ? 1
                                                          : 2;
                        }
                    }
                    if (LISTS && take) {
                        // rank bits and first vertex of its graph
                        const int32_t pt = fused ? 0 : a.part_of[x[u]];
                        an.kb = a.pfirst[pt];
                        an.part = fp_rank_bits(a.pfirst[pt + 1] - an.kb);
                        an.w = wf <= (unsigned long long)a.warp_max_w ? 0 : 4;  // tier
                    }
                    const bool small =
                        take && v[u] && (LISTS || wf <= (unsigned long long)a.warp_max_w);
                    const bool big = take && v[u] && !small && cls < 0;
                    const int pf = warp_slot(take, &set->nF);
                    const int pw = warp_slot(small, &set->nLw);
                    if (take) a.F[pf] = x[u];
                    if (small) a.Lw[pw] = an;
#pragma unroll
                    for (int c = 0; WIDE && c < 3; c++) {
                        const int pg = warp_slot(cls == c, &set->nG[c]);
                        if (cls == c) a.Lg[(size_t)c * a.n + pg] = an;
                    }
                    const int32_t win = an.w;
                    for (int j = 0; __any_sync(0xffffffffu, big && j * DENSE_KEYS < win); j++) {
                        const bool has = big && j * DENSE_KEYS < win;
                        const int pb = warp_slot(has, &set->nLd);
                        if (has) {
                            PersistAnchor it = an;
                            it.kb += j * DENSE_KEYS;
                            it.w = min(DENSE_KEYS, win - j * DENSE_KEYS);
                            it.part = win > DENSE_KEYS ? j : -1;
                            a.Ld[pb] = it;
                        }
                    }
                }
            }
            if (__any_sync(0xffffffffu, fe != 0)) {
                fw = warp_sum(fw);
                fe = warp_sum(fe);
                uw = warp_sum(uw);
                if (lane == 0) {
                    if (fw) atomicAdd(&set->front_w, fw);
                    if (fe) atomicAdd(&st->peeled_edges, fe);
                    if (fe) atomicAdd(&set->front_e, fe);
                    if (uw) atomicAdd(&st->wedges, uw);
                    if (uw) atomicAdd(&set->upd_w, uw);
                }
            }
            if (gather) {
                const size_t k = (size_t)(hk % 3);
                live_last = -warp_min(-live_last);
                if (lane == 0 && live_last >= 0) atomicMax(a.plast + k, live_last);
                __syncthreads();
                hist.flush(a.hist_w + k * NBUCKET, a.hist_c + k * NBUCKET);
                clear_next(hk);
                hk++;
            }
            // assigned vertices of earlier ranges leave the lists
            if (compact) compact_working_lists(a, range, gwarp, nwarps, lane);
            compact = false;
            if (!grid_barrier(pd, target, &s_ok)) return;
            if (threadIdx.x == 0) {
                const int nF = __ldcg(&set->nF);
                const unsigned long long now = peeled + __ldcg(&set->front_e);
                bool due = false;
                if (nF == 0) {
                    // the range is done: is a compaction due? (as cd_run)
                    due = a.dgm && range + 1 < a.P &&
                          (double)(now - peeled_at_dgm) >=
                              a.dgm_frac * (double)((unsigned long long)a.m - peeled_at_dgm);
                } else if (first && a.huc) {
                    // a recount instead of the range's first updates?
                    const unsigned long long crcnt = *a.crcnt;
                    due = crcnt > 0 && (double)__ldcg(&set->front_w) > a.huc_factor * (double)crcnt;
                }
                s_nF = nF;
                s_due = due ? 1 : 0;
                s_peeled = now;
            }
            __syncthreads();
            peeled = s_peeled;
            if (s_nF == 0) {
                compact = s_due != 0;
                if (compact) {
                    peeled_at_dgm = peeled;
                    dgm_passes++;
                }
                range++;
                mode = PERSIST_RANGE;
                continue;
            }
            mode = PERSIST_PEEL;
            if (s_due) {
                stop = PERSIST_RECOUNT;
                break;
            }
        }
        // ---- peel: updates of the listed anchors
        first = false;
        // the CTA's first item comes with the counters when there is one per CTA
        PersistAnchor pre{0, 0, 0, 0, 0, -1, 0};
        if (threadIdx.x == 0 && (int32_t)blockIdx.x < a.n) pre = load_anchor(a.Ld + blockIdx.x);
        const int32_t nW = __ldcg(&set->nLw), nD = __ldcg(&set->nLd), nF = __ldcg(&set->nF);
        PersistEmit emit{a.sup, a.sub, 0};
        unsigned long long cw = 0, cm = 0, ca = 0;
        if (LISTS && nW > 0) {
            // a group of warps per anchor: as many as leave every anchor a group.
            // The counters are those of the walks this saves (their lists are
            // kept and compacted as ever): sums of the working lists' lengths.
            int g = 1;
            while (g < PT / 32 && (int64_t)nW * 2 * g <= nwarps) g *= 2;
            const int grp = warp / g, part = warp & (g - 1);
            for (int i = grp * gridDim.x + blockIdx.x; i < nW; i += nwarps / g) {
                const PersistAnchor an = load_anchor(a.Lw + i);
                const unsigned long long q = __ldg(a.list + an.x);
                // (the first lengths are on their way while the list is read)
                int j1 = part * 32 + lane;
                uint32_t walk =
                    j1 < an.deg ? (uint32_t)__ldcg(a.len_o + __ldg(a.adj_s + an.q0 + j1)) : 0u;
                const uint32_t *e = a.pool + (q >> 24);
                const int len = (int)(q & 0xffffffu);
                const uint32_t rmask = (1u << an.part) - 1u;
                for (int j0 = part * 32 + lane; j0 < len; j0 += 128 * g) {
                    uint32_t c[4];
                    int32_t k[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int j = j0 + u * 32 * g;
                        c[u] = j < len ? __ldg(e + j) : 0u;
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        k[u] = c[u] ? an.kb + (int32_t)(c[u] & rmask) : -1;
                        c[u] >>= an.part;
                    }
                    emit.many<4>(k, c);
                }
                for (j1 += 32 * g; j1 < an.deg; j1 += 32 * g)
                    walk += (uint32_t)__ldcg(a.len_o + __ldg(a.adj_s + an.q0 + j1));
                walk = __reduce_add_sync(0xffffffffu, walk);
                const uint32_t pr = __reduce_add_sync(0xffffffffu, (uint32_t)emit.pairs);
                emit.pairs = 0;
                if (lane == 0) {
                    uint32_t *t = s_tier + an.w;  // 0: the warp tier's, 4: the windows'
                    atomicAdd(t, walk);
                    if (pr) atomicAdd(t + 1, pr);
                    if (part == 0) {
                        atomicAdd(t + 2, (uint32_t)an.deg);
                        atomicAdd(t + 3, 1u);
                    }
                }
            }
            __syncthreads();
            if (threadIdx.x < 8 && s_tier[threadIdx.x]) {
                unsigned long long *to[4] = {st->tier_w, st->tier_p, st->tier_m, st->tier_a};
                atomicAdd(to[threadIdx.x & 3] + (threadIdx.x & 4), (unsigned long long)s_tier[threadIdx.x]);
                s_tier[threadIdx.x] = 0;
            }
        }
        if (!LISTS && nW > 0) {
            WarpTable T{H.cnt + warp * (2 * WARP_SLOTS), H.cnt + warp * (2 * WARP_SLOTS) + WARP_SLOTS};
            for (int i = gwarp; i < nW;) {
                const PersistAnchor an = load_anchor(a.Lw + i);
                auto add = [&](int32_t k) {
                    cw++;
                    if (k != an.x) T.add(k);
                };
                warp_walk<4, KeysL2>(M, an.q0, an.q0 + an.deg, a.adj_o, add);
                __syncwarp();
                T.flush_clear(emit, lane);
                __syncwarp();
                cm += (unsigned long long)an.deg;
                ca++;
                if (nW <= nwarps) break;
                if (lane == 0) i = nwarps + atomicAdd(&set->workW, 1);
                i = __shfl_sync(0xffffffffu, i, 0);
            }
            cw = warp_sum(cw);
            const unsigned long long pr = warp_sum(emit.pairs);
            emit.pairs = 0;
            if (lane == 0 && ca) {
                atomicAdd(&st->tier_w[0], cw);
                atomicAdd(&st->tier_m[0], cm);
                atomicAdd(&st->tier_a[0], ca);
                if (pr) atomicAdd(&st->tier_p[0], pr);
            }
            cw = cm = ca = 0;
            __syncthreads();  // the tables' words become dense counters again
        }
        const int nG[3] = {WIDE ? __ldcg(&set->nG[0]) : 0, WIDE ? __ldcg(&set->nG[1]) : 0,
                           WIDE ? __ldcg(&set->nG[2]) : 0};
        if (WIDE && nG[0] + nG[1] + nG[2] > 0) {
            // in one go when the widest class leaves every anchor a group
            const int top = nG[2] ? 2 : nG[1] ? 1 : 0;
            if ((int64_t)(nG[0] + nG[1] + nG[2]) << (2 * top) <= (int64_t)FP_WARPS * gridDim.x) {
                group_items(a, M, H.cnt, 0, top, nG, 1 << (2 * top), emit, cw, cm, ca);
            } else {
                for (int c = top; c >= 0; c--)
                    if (nG[c]) group_items(a, M, H.cnt, c, c, nG, 1 << (2 * c), emit, cw, cm, ca);
            }
            cw = warp_sum(cw);
            if (lane == 0 && cw) {
                atomicAdd(&st->tier_w[4], cw);
                if (ca) {
                    atomicAdd(&st->tier_m[4], cm);
                    atomicAdd(&st->tier_a[4], ca);
                }
            }
            cw = cm = ca = 0;
        }
        // items per fetch: more than one only when the round has more items
        // than CTAs
        const int G = max(1, min(a.group, nD / (int)gridDim.x));
        for (int base = blockIdx.x * G; !LISTS && base < nD;) {
            const int gcount = min(G, nD - base);
            for (int i0 = 0; i0 < gcount;) {
                if (warp == 0) {
                    // the leading items whose windows fit side by side
                    PersistAnchor an{0, 0, 0, 0, 0, -1, 0};
                    if (i0 + lane < gcount)
                        an = G == 1 && base == (int)blockIdx.x ? pre : load_anchor(a.Ld + base + i0 + lane);
                    int32_t wi = an.w, di = an.deg;
#pragma unroll
                    for (int o = 1; o < GROUP; o <<= 1) {
                        const int32_t yw = __shfl_up_sync(0xffffffffu, wi, o);
                        const int32_t yd = __shfl_up_sync(0xffffffffu, di, o);
                        if (lane >= o) {
                            wi += yw;
                            di += yd;
                        }
                    }
                    const bool fits = i0 + lane < gcount && (lane == 0 || wi <= DENSE_KEYS);
                    const int nb = __popc(__ballot_sync(0xffffffffu, fits));
                    if (lane < nb) {
                        s_g.q0[lane] = an.q0;
                        s_g.x[lane] = an.x;
                        s_g.kb[lane] = an.kb;
                        s_g.ke[lane] = an.kb + an.w;
                        s_g.part[lane] = an.part;
                        s_g.off[lane + 1] = wi;
                        s_g.pre[lane + 1] = di;
                    }
                    if (lane == 0) {
                        s_g.off[0] = s_g.pre[0] = 0;
                        s_nb = nb;
                    }
                    // an anchor in several items counts once
                    const unsigned whole = __ballot_sync(0xffffffffu, lane < nb && an.part <= 0);
                    int32_t dw = lane < nb && an.part <= 0 ? an.deg : 0;
                    dw = warp_sum(dw);
                    cm += (unsigned long long)dw;
                    ca += __popc(whole);
                }
                __syncthreads();
                const int nb = s_nb;
                H.set_width(s_g.off[nb]);
                if (nb == 1) {
                    OneMids OM{M, a.adj_o, s_g.q0[0], s_g.kb[0], s_g.ke[0], s_g.part[0] >= 0};
                    OneVisit v{&H, s_g.x[0], s_g.kb[0], s_g.ke[0]};
                    cw += cta_walk<true, KeysL2>(OM, 0, s_g.pre[1], a.adj_o, ch, v);
                    OneEmit em{&emit, s_g.kb[0]};
                    H.sweep<true, true>(em);
                } else {
                    GroupMids GM{M, a.adj_o, &s_g, nb};
                    GroupVisit v{&H, &s_g};
                    cw += cta_walk<true, KeysL2>(GM, 0, s_g.pre[nb], a.adj_o, ch, v);
                    GroupEmit em{&emit, &s_g, nb};
                    H.sweep<true, true>(em);
                }
                __syncthreads();
                H.reset_scalars();
                i0 += nb;
                __syncthreads();
            }
            if (nD <= (int)gridDim.x * G) break;
            if (threadIdx.x == 0) s_idx = (int)gridDim.x * G + atomicAdd(&set->workD, G);
            __syncthreads();
            base = s_idx;
        }
        {
            const unsigned long long pr = warp_sum(emit.pairs);
            if (lane == 0 && pr) atomicAdd(&st->tier_p[4], pr);
            if (threadIdx.x == 0 && cw) {
                atomicAdd(&st->tier_w[4], cw);
                if (cm) atomicAdd(&st->tier_m[4], cm);
                if (ca) atomicAdd(&st->tier_a[4], ca);
            }
        }
        if (!grid_barrier(pd, target, &s_ok)) return;
        if (lead) {
            a.rec[nrec] = PersistRound{range, nF, hi,
                                       {__ldcg(&st->tier_a[0]), __ldcg(&st->tier_a[4])},
                                       {__ldcg(&st->tier_w[0]), __ldcg(&st->tier_w[4])}};
        }
        nrec++;
        mode = PERSIST_SCAN;
        if (nrec == a.rec_cap) {
            stop = PERSIST_RECORDS_FULL;
            break;
        }
    }
    if (lead) {
        pd->mode = mode;
        pd->stop = stop;
        pd->range = range;
        pd->sk = sk;
        pd->peeled = peeled;
        pd->nrec = nrec;
        pd->hk = hk;
        pd->dgm_passes = dgm_passes;
        pd->hi = hi;
        pd->peeled_at_dgm = peeled_at_dgm;
        pd->wrem_prev = s_wrem;
        pd->tgt_prev = s_tgt;
    }
}

constexpr size_t persist_smem() { return DenseSlice::bytes() + chunk_bytes(PT); }

}  // namespace

// Groups of warps pay where the mean walk is short: with several windows below
// the 8,192 wedges their tables hold (100,000 x 30,000, 1M edges, 2,000 wedges:
// 11.9 against 14.3 ms for the step; 40,000 x 400,000, 3M edges, 22,000: 23.6
// against 22.1; uniform graphs of 1M and 5M edges 0.8 against 2.2, 1.0 against
// 2.9), with one below 1,024 (2,000 x 500, 20k edges, 400: 2.2 against
// 2.4 the whole call; 5,000 x 20,000, 200k edges, 3,800: 7.8 against 6.8).
bool cd_persist_wide(const Decomp &D) {
    const uint64_t mean = D.n > 0 ? D.wedges_bup / (uint64_t)D.n : 0;
    return !D.parts && mean < (D.n > DENSE_KEYS ? 8192u : 1024u);
}

// Lists pay where a vertex's key space is at most two windows and the walks of
// all vertices at once (5 ms per 10^9 wedges; with the working lists compacted
// between ranges the rounds walk a third to a half of them) cost less than what
// the rounds save: 2 to 5 us each, of some 400, or 1,300 in a large union.
// 5,000 x 20,000, 200k edges: the whole call 5.7 ms, 7.0 without; 30,000 x 9,000,
// 300k, from the host 7.2 / 9.7; 2,000 x 500, 20k, 1.8 / 2.3; 256 packed graphs
// (1.9 10^9 wedges) 36 / 44; 40,000 x 400,000, 3M (9 10^8) 23.5 / 25.4; but 36,000
// x 1M, 10M (over 2 10^9) 44 / 42. Larger sides count a walk in slices and lose
// more: 120,000 x 40,000, 3M, 36 / 30 for the step; 140,000 x 14,000, 2M, 60 / 31.
// Sides of several windows with short walks keep the groups (100,000 x 30,000
// uniform, 1M edges: 1.1 / 0.8). Large unions: 24 graphs of 3.7 10^9 wedges 35.2 ms
// by lists, 35.8 by windows: the line may lie at 3 10^9 as well as above, and the
// counters of a round by lists are 32 bits wide. Not beside other units of the serving engine
// (list_bound): the walks take every SM, and the other units' cooperative
// launches wait for them (24 requests of 10k-1M edges: 57.4 / 56.4).
bool cd_persist_by_lists(const Decomp &D) {
    // (the counters of a round by lists are 32 bits wide)
    if (D.list_bound || D.max_deg_s >= 65535 ||
        D.wedges_bup + (uint64_t)D.m > (D.parts ? 3000000000ull : 1200000000ull))
        return false;
    if (!D.parts)
        return D.n <= 2 * DENSE_KEYS && (D.n <= DENSE_KEYS || !cd_persist_wide(D));
    for (size_t i = 0; i + 1 < D.parts->size(); i++)
        if ((*D.parts)[i + 1] - (*D.parts)[i] > DENSE_KEYS) return false;
    return true;
}

bool cd_persist_fits(const Decomp &D) {
    if (D.max_deg_s >= 65535) return false;  // counts may need 32 bits
    if (!D.parts) {
        // several windows walk a long list once per window: only while the
        // rounds are short (120,000 x 40,000 with 3M edges, 1.9 10^9 wedges,
        // 4 windows: 35.3 ms here, 30.8 by the per-round kernels; 40,000 x
        // 400,000 with 3M edges, 9 10^8, 2 windows: 21.5 against 29.3), and
        // past PERSIST_SLICES only where groups count the short walks
        // (500,000 x 120,000 uniform, 5M edges, 14 windows: 0.9 against 3.1)
        const int64_t windows = ceil_div(D.n, DENSE_KEYS);
        return windows == 1 ||
               (windows <= (cd_persist_wide(D) ? PERSIST_WIDE_SLICES : PERSIST_SLICES) &&
                (double)windows * (double)D.wedges_bup <= 3e9);
    }
    for (size_t i = 0; i + 1 < D.parts->size(); i++)
        if ((*D.parts)[i + 1] - (*D.parts)[i] > DENSE_KEYS) return false;
    return true;
}

static const void *persist_kernel(int form) {
    return form == PERSIST_LISTS    ? (const void *)k_cd_persist<PERSIST_LISTS>
           : form == PERSIST_GROUPS ? (const void *)k_cd_persist<PERSIST_GROUPS>
                                    : (const void *)k_cd_persist<PERSIST_WINDOWS>;
}

int cd_persist_group(const Decomp &D) {
    const uint64_t w = (uint64_t)D.max_deg_s * (uint64_t)D.max_deg_o;  // an anchor's, at most
    return w > 0 ? (int)std::max<uint64_t>(1, std::min<uint64_t>(GROUP, GROUP_W / w)) : GROUP;
}

int cd_persist_grid(int64_t m, int form) {
    const void *kernel = persist_kernel(form);
    allow_max_smem(kernel);
    int occ = 0;
    RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, PT, persist_smem()));
    if (occ < 1) fail(RECEIPT_ERR_INTERNAL, "the one-launch form does not fit an SM");
    // One CTA per 4,096 edges: fewer leave a round's anchors queueing (30,000 x
    // 9,000, 300k edges: 14.4 ms a call with 8,192 edges per CTA, 10.8 with
    // 4,096, 10.5 with 2,048), more only wait at the barriers while other
    // streams could use their SMs (24 requests of 10k-1M edges through the
    // serving loop: 64 / 70 / 118 ms). At least 16: the smallest sides' rounds
    // have that many anchors.
    return (int)std::min<int64_t>(num_sms() * std::min(occ, 2), std::max<int64_t>(16, m / 4096));
}

void cd_persist_launch(const PersistArgs &a, int grid, int form, cudaStream_t s) {
    void *args[] = {(void *)&a};
    RC_CUDA(cudaMemsetAsync(&a.pd->bar, 0, sizeof(unsigned), s));
    RC_CUDA(cudaLaunchCooperativeKernel(persist_kernel(form), dim3(grid), dim3(PT), args,
                                        persist_smem(), s));
    RC_LAUNCH();
}

}  // namespace receipt
