// Graph build (Algorithm 1, steps 1-3): duplicate removal, relabelling of
// each side in descending order of degree, and the CSR of both sides with
// neighbour lists sorted ascending by the new labels.
//
// The paper relabels all of W = U u V in one label space. Here each side
// keeps its own dense local ids (rank by descending degree, ties by original
// id), and `below[x]` records how many vertices of the OTHER side come
// before x in the single global order (descending degree, U before V on a
// tie, then id). For an end point ep on side A and a middle vertex mp on
// side B, "label(ep) < label(mp)" is then exactly "ep < below_B[mp]".
#include "common.cuh"
#include "internal.cuh"

namespace receipt {

namespace {

__global__ void k_validate_pack(const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                                int64_t m, int32_t nu, int32_t nv, int bits_v,
                                uint64_t *__restrict__ keys, unsigned long long *bad) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long nbad = 0;
    for (; i < m; i += stride) {
        int32_t u = eu[i], v = ev[i];
        if (u < 0 || u >= nu || v < 0 || v >= nv) {
            nbad++;
            u = 0;
            v = 0;
        }
        keys[i] = ((uint64_t)u << bits_v) | (uint64_t)v;
    }
    nbad = warp_sum(nbad);
    if ((threadIdx.x & 31) == 0 && nbad) atomicAdd(bad, nbad);
}

// Duplicate removal from sorted keys, a tile of DD_TILE keys a block: first the
// tiles' counts of distinct keys, then the keys to their places and V's
// degrees (original ids). Every warp owns consecutive keys.
constexpr int DD_THREADS = 256;
constexpr int DD_ITEMS = 8;
constexpr int DD_TILE = DD_THREADS * DD_ITEMS;

__device__ __forceinline__ void dd_load(const uint64_t *__restrict__ keys, int64_t m, int64_t wbase,
                                        uint64_t (&k)[DD_ITEMS], unsigned (&heads)[DD_ITEMS]) {
    const int lane = threadIdx.x & 31;
    uint64_t before = wbase > 0 && wbase < m ? keys[wbase - 1] : ~0ull;
#pragma unroll
    for (int j = 0; j < DD_ITEMS; j++) {
        const int64_t g = wbase + j * 32 + lane;
        k[j] = g < m ? keys[g] : 0;
    }
#pragma unroll
    for (int j = 0; j < DD_ITEMS; j++) {
        uint64_t prev = __shfl_up_sync(0xffffffffu, k[j], 1);
        if (lane == 0) prev = before;
        before = __shfl_sync(0xffffffffu, k[j], 31);
        const int64_t g = wbase + j * 32 + lane;
        heads[j] = __ballot_sync(0xffffffffu, g < m && (g == 0 || k[j] != prev));
    }
}

__global__ void k_dedup_count(const uint64_t *__restrict__ keys, int64_t m,
                              uint32_t *__restrict__ tiles) {
    __shared__ uint32_t s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    uint64_t k[DD_ITEMS];
    unsigned heads[DD_ITEMS];
    dd_load(keys, m, (int64_t)blockIdx.x * DD_TILE + (threadIdx.x >> 5) * (32 * DD_ITEMS), k, heads);
    uint32_t c = 0;
#pragma unroll
    for (int j = 0; j < DD_ITEMS; j++) c += __popc(heads[j]);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_n, c);
    __syncthreads();
    if (threadIdx.x == 0) tiles[blockIdx.x] = s_n;
}

// V's hubs would take most of a plain count's time (degree 50,000 among 10M
// edges: 0.72 ms, 0.22 so): a block counts the ids it meets first in a shared
// table of DD_SLOTS, added at its end.
constexpr int DD_GROUP = 8;  // tiles a block
constexpr int DD_SLOTS = 2048;
__global__ void k_dedup_write(const uint64_t *__restrict__ keys, int64_t m,
                              const uint32_t *__restrict__ tiles, int64_t ntiles, uint64_t mask_v,
                              uint64_t *__restrict__ ukeys, uint32_t *__restrict__ deg_v) {
    __shared__ uint32_t s_w[2][DD_THREADS / 32];
    __shared__ uint32_t s_id[DD_SLOTS], s_cnt[DD_SLOTS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < DD_SLOTS; i += DD_THREADS) {
        s_id[i] = ~0u;
        s_cnt[i] = 0;
    }
    for (int t = 0; t < DD_GROUP; t++) {
        const int64_t tile = (int64_t)blockIdx.x * DD_GROUP + t;
        if (tile >= ntiles) break;
        uint64_t k[DD_ITEMS];
        unsigned heads[DD_ITEMS];
        dd_load(keys, m, tile * DD_TILE + warp * (32 * DD_ITEMS), k, heads);
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < DD_ITEMS; j++) c += __popc(heads[j]);
        if (lane == 0) s_w[t & 1][warp] = c;
        __syncthreads();
        uint32_t at = tiles[tile];
        for (int w = 0; w < warp; w++) at += s_w[t & 1][w];
#pragma unroll
        for (int j = 0; j < DD_ITEMS; j++) {
            if (heads[j] >> lane & 1u) {
                ukeys[at + __popc(heads[j] & lanemask_lt())] = k[j];
                const uint32_t v = (uint32_t)(k[j] & mask_v);
                const uint32_t h = (v * 2654435761u) >> 21;
                uint32_t id = ((volatile uint32_t *)s_id)[h];
                if (id == ~0u) {
                    id = atomicCAS(&s_id[h], ~0u, v);
                    if (id == ~0u) id = v;
                }
                if (id == v)
                    atomicAdd(&s_cnt[h], 1u);
                else
                    atomicAdd(&deg_v[v], 1u);
            }
            at += __popc(heads[j]);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < DD_SLOTS; i += DD_THREADS)
        if (s_cnt[i]) atomicAdd(&deg_v[s_id[i]], s_cnt[i]);
}
static_assert(DD_SLOTS == 1 << 11, "hash of 11 bits");

// First of the sorted distinct keys of every u (nu + 1 entries).
__global__ void k_u_starts(const uint64_t *__restrict__ ukeys, const uint32_t *__restrict__ mu,
                           int32_t nu, int bits_v, uint32_t *__restrict__ ustart) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u > nu) return;
    uint32_t lo = 0, hi = *mu;
    const uint64_t want = (uint64_t)u << bits_v;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (ukeys[mid] < want)
            lo = mid + 1;
        else
            hi = mid;
    }
    ustart[u] = lo;
}

// Degrees of U from the starts, and both sides' largest degrees (block
// maxima): mx[0] U, mx[1] V.
__global__ void k_degrees(const uint32_t *__restrict__ ustart, int32_t nu, int32_t nv,
                          uint32_t *__restrict__ deg, unsigned *__restrict__ mx) {
    unsigned a = 0, b = 0;
    const int64_t n = (int64_t)nu + nv, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        if (i < nu) {
            const uint32_t d = ustart[i + 1] - ustart[i];
            deg[i] = d;
            a = max(a, d);
        } else {
            b = max(b, deg[i]);
        }
    }
    a = __reduce_max_sync(0xffffffffu, a);
    b = __reduce_max_sync(0xffffffffu, b);
    if ((threadIdx.x & 31) == 0) {
        if (a) atomicMax(&mx[0], a);
        if (b) atomicMax(&mx[1], b);
    }
}

// Sort keys of both sides' vertices: side, then maxdeg - deg, so that an
// ascending stable sort gives descending degrees, ties in ascending original
// id (the input order, in the low 32 bits).
__global__ void k_degree_keys(const uint32_t *__restrict__ deg, int32_t nu, int32_t nv,
                              uint32_t maxdeg, int db, uint64_t *__restrict__ key) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)nu + nv) return;
    const uint64_t side = i >= nu;
    key[i] = (((side << db) | (uint64_t)(maxdeg - deg[i])) << 32) | (uint32_t)(side ? i - nu : i);
}

__global__ void k_relabel_maps(const uint64_t *__restrict__ key, int32_t nu, int32_t nv,
                               const uint32_t *__restrict__ deg, int32_t *__restrict__ new2old_u,
                               int32_t *__restrict__ new2old_v, int32_t *__restrict__ old2new,
                               int64_t *__restrict__ deg_new) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)nu + nv) return;
    const int32_t o = (int32_t)(uint32_t)key[p];
    const int64_t base = p < nu ? 0 : nu;
    (p < nu ? new2old_u : new2old_v)[p - base] = o;
    old2new[base + o] = (int32_t)(p - base);
    deg_new[p] = deg[base + o];
}

// Offsets of both sides from the scanned degrees, and below[x] = number of
// other-side vertices ahead of x in the global order. On side U (U wins ties):
// #{v : deg_v > deg_x}. On side V: #{u : deg_u >= deg_y}. The degrees are in
// descending order on each side.
__global__ void k_offsets_below(const int64_t *__restrict__ deg_new, const int64_t *__restrict__ pre,
                                int32_t nu, int32_t nv, int64_t m, int64_t *__restrict__ off_u,
                                int64_t *__restrict__ off_v, int32_t *__restrict__ below_u,
                                int32_t *__restrict__ below_v) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p == 0) {
        off_u[nu] = m;
        off_v[nv] = m;
    }
    if (p >= (int64_t)nu + nv) return;
    const bool u = p < nu;
    const int64_t d = deg_new[p];
    const int64_t *other = u ? deg_new + nu : deg_new;
    // first index whose degree is <= d (U) or < d (V)
    int32_t lo = 0, hi = u ? nv : nu;
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo) / 2;
        const bool ahead = u ? other[mid] > d : other[mid] >= d;
        if (ahead)
            lo = mid + 1;
        else
            hi = mid;
    }
    if (u) {
        off_u[p] = pre[p];
        below_u[p] = lo;
    } else {
        off_v[p - nu] = pre[p] - m;
        below_v[p - nu] = lo;
    }
}

// Relabelled edges grouped by U's new labels: a vertex's edges move as one
// block to its new place. key = v << bu | u.
__global__ void k_relabel_edges(const uint64_t *__restrict__ ukeys, int64_t m, int bits_v,
                                uint64_t mask_v, const uint32_t *__restrict__ ustart,
                                const int32_t *__restrict__ o2n_u, const int32_t *__restrict__ o2n_v,
                                const int64_t *__restrict__ off_u, int bu, uint64_t *__restrict__ key) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const uint64_t k = ukeys[i];
    const int64_t uo = (int64_t)(k >> bits_v);
    const int32_t u = o2n_u[uo], v = o2n_v[k & mask_v];
    key[off_u[u] + (i - ustart[uo])] = ((uint64_t)v << bu) | (uint64_t)u;
}

// Prefix lengths (the wedges that Algorithm 1 walks from an edge, see count.cu)
// of up to WALK_SAMPLES edges a side, evenly spaced; counting chooses its form by
// their mean. A warp per edge, which probes 32 places a step: a thread's binary
// searches took 12 us, a hundredth of a build and count of 1M edges.
constexpr int WALK_SAMPLES = 1 << 11;
struct WalkSide {
    const int64_t *off, *off_o;
    const int32_t *adj, *adj_o, *below_o;
    int32_t n;
};
// Entries of the ascending a[0, n) that are <= key. One warp.
template <typename T>
__device__ __forceinline__ int64_t warp_upper_bound(const T *__restrict__ a, int64_t n, T key) {
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
    while (hi - lo > 0) {
        const int64_t step = (hi - lo + 31) / 32, i = lo + step * lane;
        const unsigned le = __ballot_sync(0xffffffffu, i < hi && a[i] <= key);
        const int c = __popc(le);  // a[lo + step (c - 1)] <= key < a[lo + step c]
        if (c == 0) return lo;
        hi = imin64(hi, lo + step * c);
        lo += step * (c - 1) + 1;
    }
    return lo;
}
// sum[0]: the lengths, sum[1]: blocks done; the last one leaves the sum in
// host memory (a copy would take as long as the kernel).
__global__ void __launch_bounds__(256) k_sample_walks(WalkSide a, WalkSide b, int64_t m, int32_t samples,
                                                      unsigned long long *__restrict__ sum,
                                                      unsigned long long *__restrict__ host) {
    __shared__ unsigned long long s_len;
    if (threadIdx.x == 0) s_len = 0;
    __syncthreads();
    const int32_t i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i < samples) {
        const WalkSide &S = blockIdx.y ? b : a;
        const int64_t q = (2 * (int64_t)i + 1) * m / (2 * (int64_t)samples);
        const int32_t mp = S.adj[q];
        const int64_t p0 = S.off_o[mp], p1 = S.off_o[mp + 1];
        const int32_t below = S.below_o[mp];
        // the start point: the last one whose list begins at or before q
        const int32_t sp = (int32_t)warp_upper_bound<int64_t>(S.off, S.n, q) - 1;
        const int64_t len = warp_upper_bound<int32_t>(S.adj_o + p0, p1 - p0, min(sp, below) - 1);
        if ((threadIdx.x & 31) == 0 && len) atomicAdd(&s_len, (unsigned long long)len);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_len) atomicAdd(sum, s_len);
        __threadfence();
        if (atomicAdd(sum + 1, 1ull) == (unsigned long long)gridDim.x * gridDim.y - 1) {
            *host = atomicAdd(sum, 0ull);
            __threadfence_system();
        }
    }
}

inline unsigned blocks_for(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// Builds a graph; the device arrays live in one allocation owned by g.
receipt_graph *build_graph(const int32_t *d_eu, const int32_t *d_ev, int64_t m, int32_t nu,
                           int32_t nv, int dedup, cudaStream_t s) {
    if (nu < 0 || nv < 0 || m < 0) fail(RECEIPT_ERR_INVALID, "negative size");
    if (m >= (int64_t)INT32_MAX) fail(RECEIPT_ERR_OVERFLOW, "m must be below 2^31");
    if (m > 0 && (!d_eu || !d_ev)) fail(RECEIPT_ERR_INVALID, "null edge pointer");
    if (m > 0 && ((int64_t)nu == 0 || nv == 0)) fail(RECEIPT_ERR_INVALID, "edges on an empty side");
    const int bu = bits_for(nu > 0 ? (uint64_t)(nu - 1) : 0);
    const int bv = bits_for(nv > 0 ? (uint64_t)(nv - 1) : 0);
    const uint64_t mask_v = bv ? ((1ull << bv) - 1) : 0;
    const uint64_t mask_u = bu ? ((1ull << bu) - 1) : 0;

    // scalars: [0] bad ids, [1] max deg U and V (read back), [2], [3] k_sample_walks
    DevBuf<unsigned long long> scal(4, s);
    scal.zero();
    DevBuf<uint64_t> keys(m, s);
    if (m > 0) {
        k_validate_pack<<<std::min<unsigned>(blocks_for(m), 4096), 256, 0, s>>>(
            d_eu, d_ev, m, nu, nv, bv, keys.get(), scal.get());
        RC_LAUNCH();
    }
    radix_sort(keys, m, 0, bu + bv, s);
    const int64_t tiles = (m + DD_TILE - 1) / DD_TILE;
    DevBuf<uint32_t> tile_at(tiles + 1, s);  // distinct keys of the tiles before
    DevBuf<uint64_t> ukeys(m, s);
    DevBuf<uint32_t> ustart((int64_t)nu + 1, s), deg((int64_t)nu + nv, s);  // deg: U, then V
    deg.zero();
    tile_at.zero();
    if (m > 0) {
        k_dedup_count<<<(unsigned)tiles, DD_THREADS, 0, s>>>(keys.get(), m, tile_at.get());
        RC_LAUNCH();
        scan_exclusive<uint32_t>(tile_at.get(), tile_at.get(), tiles + 1, s);
        k_dedup_write<<<(unsigned)((tiles + DD_GROUP - 1) / DD_GROUP), DD_THREADS, 0, s>>>(
            keys.get(), m, tile_at.get(), tiles, mask_v, ukeys.get(), deg.get() + nu);
        RC_LAUNCH();
    }
    // number of unique edges, read together with the checks
    unsigned long long h[4] = {0, 0, 0, 0};
    uint32_t distinct = 0;
    unsigned *dmax = reinterpret_cast<unsigned *>(scal.get() + 1);
    k_u_starts<<<blocks_for((int64_t)nu + 1), 256, 0, s>>>(ukeys.get(), tile_at.get() + tiles, nu, bv,
                                                          ustart.get());
    RC_LAUNCH();
    if (nu + (int64_t)nv > 0) {
        k_degrees<<<std::min<unsigned>(blocks_for((int64_t)nu + nv), 1024), 256, 0, s>>>(
            ustart.get(), nu, nv, deg.get(), dmax);
        RC_LAUNCH();
    }
    RC_CUDA(cudaMemcpyAsync(h, scal.get(), sizeof(h), cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaMemcpyAsync(&distinct, tile_at.get() + tiles, 4, cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    if (h[0]) fail(RECEIPT_ERR_INVALID, std::to_string(h[0]) + " edge ids out of range");
    const int64_t mu = distinct;
    if (!dedup && mu != m) fail(RECEIPT_ERR_INVALID, "duplicate edges with dedup == 0");
    const uint32_t maxdeg_u = (uint32_t)(h[1] & 0xffffffffu);
    const uint32_t maxdeg_v = (uint32_t)(h[1] >> 32);

    // one allocation for every array the graph keeps
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    size_t sz_off_u = al(8 * ((size_t)nu + 1)), sz_off_v = al(8 * ((size_t)nv + 1));
    size_t sz_adj = al(4 * (size_t)(mu > 0 ? mu : 1));
    size_t sz_id_u = al(4 * (size_t)(nu > 0 ? nu : 1)), sz_id_v = al(4 * (size_t)(nv > 0 ? nv : 1));
    size_t total = sz_off_u + sz_off_v + 2 * sz_adj + 2 * sz_id_u + 2 * sz_id_v;
    receipt_graph *g = new receipt_graph();
    g->nu = nu;
    g->nv = nv;
    g->m = mu;
    RC_CUDA(cudaGetDevice(&g->device));
    char *base = nullptr;
    if (cudaMallocAsync((void **)&base, total, s) != cudaSuccess) {
        cudaGetLastError();
        delete g;
        fail(RECEIPT_ERR_OOM, "graph allocation failed");
    }
    g->owned = base;
    char *p = base;
    auto take = [&](size_t b) {
        char *r = p;
        p += b;
        return r;
    };
    Side &SU = g->side[0];
    Side &SV = g->side[1];
    SU.n = nu;
    SV.n = nv;
    SU.off = (int64_t *)take(sz_off_u);
    SV.off = (int64_t *)take(sz_off_v);
    SU.adj = (int32_t *)take(sz_adj);
    SV.adj = (int32_t *)take(sz_adj);
    SU.new2old = (int32_t *)take(sz_id_u);
    SV.new2old = (int32_t *)take(sz_id_v);
    SU.below = (int32_t *)take(sz_id_u);
    SV.below = (int32_t *)take(sz_id_v);
    g->max_deg[0] = (int32_t)maxdeg_u;
    g->max_deg[1] = (int32_t)maxdeg_v;

    try {
        unsigned long long *walks = (unsigned long long *)pinned_scratch(8);
        *walks = 0;
        // relabel both sides: one stable sort by (side, maxdeg - deg)
        const int64_t nn = (int64_t)nu + nv;
        DevBuf<int32_t> o2n(nn, s);
        DevBuf<int64_t> dn(nn, s), pre(nn, s);
        if (nn > 0) {
            const uint32_t mx = std::max(maxdeg_u, maxdeg_v);
            const int db = bits_for(mx);
            DevBuf<uint64_t> dk(nn, s);
            k_degree_keys<<<blocks_for(nn), 256, 0, s>>>(deg.get(), nu, nv, mx, db, dk.get());
            RC_LAUNCH();
            // the sides are in order already
            radix_sort(dk, nn, 32, 32 + db + (nu > 0 && nv > 0), s);
            k_relabel_maps<<<blocks_for(nn), 256, 0, s>>>(dk.get(), nu, nv, deg.get(), SU.new2old,
                                                          SV.new2old, o2n.get(), dn.get());
            RC_LAUNCH();
            scan_exclusive<int64_t>(dn.get(), pre.get(), nn, s);
        }
        k_offsets_below<<<blocks_for(std::max<int64_t>(nn, 1)), 256, 0, s>>>(
            dn.get(), pre.get(), nu, nv, mu, SU.off, SV.off, SU.below, SV.below);
        RC_LAUNCH();
        if (mu > 0) {
            // Grouped by u, a stable sort by v gives V's lists; those, stably
            // sorted by u, give U's.
            k_relabel_edges<<<blocks_for(mu), 256, 0, s>>>(ukeys.get(), mu, bv, mask_v, ustart.get(),
                                                           o2n.get(), o2n.get() + nu, SU.off, bu,
                                                           keys.get());
            RC_LAUNCH();
            ukeys.release();
            radix_sort(keys, mu, bu, bu + bv, s, RadixField{SV.adj, 0, mask_u});
            radix_sort(keys, mu, 0, bu, s, RadixField{SU.adj, bu, mask_v}, false);
            const int32_t samples = (int32_t)std::min<int64_t>(mu, WALK_SAMPLES);
            k_sample_walks<<<dim3(blocks_for(samples, 8), 2), 256, 0, s>>>(
                WalkSide{SU.off, SV.off, SU.adj, SV.adj, SV.below, nu},
                WalkSide{SV.off, SU.off, SV.adj, SU.adj, SU.below, nv}, mu, samples, scal.get() + 2,
                walks);
            RC_LAUNCH();
        }
        RC_CUDA(cudaStreamSynchronize(s));
        g->count_walks =
            mu > WALK_SAMPLES ? (uint64_t)((double)*walks * ((double)mu / WALK_SAMPLES)) : *walks;
    } catch (...) {
        cudaStreamSynchronize(s);
        cudaFreeAsync(g->owned, s);
        delete g;
        throw;
    }
    return g;
}

// The graph's memory goes back to the stream-ordered pool without a device
// synchronisation. Every entry point has finished its work on the graph when
// it returns, so ordering the free on the legacy stream is safe.
void destroy_graph(receipt_graph *g) {
    if (!g) return;
    if (g->owned) {
        int prev = -1;
        cudaGetDevice(&prev);
        if (prev != g->device) cudaSetDevice(g->device);
        cudaFreeAsync(g->owned, 0);
        if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
    }
    delete g;
}

}  // namespace receipt
