// Updates of a large activeSet through the other side's hubs.
//
// The peel update subtracts from every remaining x' the sum over the anchors
// x of C(c(x, x'), 2), c = shared neighbours. On heavy-tailed graphs nearly
// all wedges pass through a few middle vertices of huge degree: the first
// HUBS (local ids are in descending order of degree). With c = a + b, a
// counting the hubs among the shared neighbours and b the others,
//
//   C(c, 2) = C(a, 2) + (C(b, 2) + a b).
//
// Hub part. Summed over the anchors, C(a, 2) counts, for every pair h' < h of
// hubs adjacent to x', the anchors adjacent to both:
//   sum_x C(a(x, x'), 2) = sum_{h' < h in N_x'} G[h, h'],
//   G[h, h'] = anchors adjacent to h and h',
// one small matrix per round and a quadratic form of every remaining vertex's
// 256-bit hub mask, which runs on the tensor cores (k_hub_quad): no wedge
// through a hub is walked. All numbers are integers below 2^24 in every
// 32-bit accumulation, so the result is exact.
//
// Rest. The other middle vertices' wedges are pulled instead of pushed: the
// anchors adjacent to each of them are listed once per round, and every
// remaining x' walks its own neighbours' lists and aggregates b(x, x') over
// the activeSet's index space (a few thousand keys, whatever the side's
// size): no key slices, and one addition to sup[x'] in place of one atomic
// per pair. a(x, x') is a population count of two masks. The HEAVY vertices
// of highest degree would walk too much by themselves; for them every anchor
// counts the bits of its neighbours' masks over those vertices.
//
// Measured (us a round on average, 40M-edge graph with 800,000 vertices on the
// side, 5,000 anchors a round): pull 75 (8 lanes) + 245 (warps) + 390 (CTAs),
// heavy 62, quadratic forms 45 + 70 and the Gram matrix 7 beside them. The pull
// is bound by the L1 (one 32-byte mask per wedge; 68 to 74% of its throughput in
// the larger two kernels) and by the chain of dependent loads of a vertex. The step
// took 664 ms by the per-anchor tiers alone (1.26 10^11 wedges walked) and takes
// 328 so (1.2 10^10); 10M-edge graph 120.6 -> 79.5 ms, 3M edges in 25 subsets
// 17.9 -> 12.0.
#include <cuda_fp16.h>

#include <algorithm>

#include "cd.cuh"

namespace receipt {

namespace {

constexpr int HUBS = HubPath::HUBS;
constexpr int HW = HUBS / 32;  // words of a hub mask
constexpr int HEAVY = 256;     // side-s vertices updated anchor by anchor
constexpr int NT = HUBS / 8, KT = HUBS / 16;
// (k tile, n tile) pairs below or on the diagonal, n tiles of one k tile
// together: the strictly lower triangle of G
constexpr int TILES = KT * NT - KT * (KT - 1);
static_assert(HUBS == 256 && HW == 8, "masks are two 16-byte loads");
__host__ __device__ constexpr int tile_index(int kt, int nt) {
    return NT * kt - kt * (kt - 1) + (nt - 2 * kt);
}
constexpr int DIGIT = 11;  // bits of G per fp16 operand (integers up to 2^11 are exact)

struct Mask {
    uint32_t w[HW];
};
__device__ __forceinline__ Mask load_mask(const uint32_t *__restrict__ p) {
    const uint4 lo = __ldg((const uint4 *)p), hi = __ldg((const uint4 *)p + 1);
    return Mask{{lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w}};
}
__device__ __forceinline__ uint32_t common(const Mask &a, const Mask &b) {
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < HW; i++) c += __popc(a.w[i] & b.w[i]);
    return c;
}

// mask[x]: bit y for every neighbour y < 256 of x (a prefix of its ascending
// list), its length in plen[x]. One warp per list.
__global__ void k_prefix_masks(const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                               int32_t n, uint32_t *__restrict__ mask, int32_t *__restrict__ plen) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = w0; x < n; x += nw) {
        const int64_t q0 = off[x], q1 = off[x + 1];
        uint32_t mine = 0;  // word `lane` of the mask (lanes 0..7)
        int32_t len = 0;
        for (int64_t qb = q0; qb < q1; qb += 32) {
            const int32_t y = qb + lane < q1 ? adj[qb + lane] : HUBS;
            const unsigned in = __ballot_sync(0xffffffffu, y < HUBS);
            len += __popc(in);
#pragma unroll
            for (int w = 0; w < HW; w++) {
                const uint32_t v =
                    __reduce_or_sync(0xffffffffu, (y >> 5) == w ? 1u << (y & 31) : 0u);
                if (lane == w) mine |= v;
            }
            if (in != 0xffffffffu) break;
        }
        if (lane < HW) mask[x * HW + lane] = mine;
        if (lane == 0 && plen) plen[x] = len;
    }
}

// out[0]: sum of d (d - 1) over the hubs; out[1]: degree of the first vertex
// of side s that is not heavy.
__global__ void k_hub_probe(const int64_t *__restrict__ off_o, int32_t n_o,
                            const int64_t *__restrict__ off_s, int32_t n,
                            unsigned long long *__restrict__ out) {
    const int y = threadIdx.x;
    if (y == 0) out[1] = n > HEAVY ? (unsigned long long)(off_s[HEAVY + 1] - off_s[HEAVY]) : 0;
    unsigned long long d = y < n_o ? (unsigned long long)(off_o[y + 1] - off_o[y]) : 0;
    d = warp_sum(d * (d ? d - 1 : 0));
    if ((threadIdx.x & 31) == 0 && d) atomicAdd(out, d);
}

// Where every anchor's edges past the hubs begin in the round's flat list of
// such edges (one CTA), and the round's counters to zero.
__global__ void __launch_bounds__(1024) k_hub_begin(HubArgs a) {
    __shared__ int32_t tmp[33];
    __shared__ int32_t s_run;
    const int32_t nA = a.st->nLb;
    if (threadIdx.x == 0) s_run = 0;
    if (threadIdx.x < TILES / 32 + 1) a.hd->flags[threadIdx.x] = 0;
    __syncthreads();
    constexpr int U = 8;  // consecutive anchors per thread and step
    for (int32_t b = 0; b < nA; b += 1024 * U) {
        const int32_t i0 = b + threadIdx.x * U;
        int32_t x[U], d[U], sum = 0;
#pragma unroll
        for (int u = 0; u < U; u++) x[u] = i0 + u < nA ? a.A[i0 + u] : -1;
#pragma unroll
        for (int u = 0; u < U; u++)
            d[u] = x[u] >= 0 ? (int32_t)(a.off_s[x[u] + 1] - a.off_s[x[u]]) - a.plen[x[u]] : 0;
#pragma unroll
        for (int u = 0; u < U; u++) sum += d[u];
        int32_t tot;
        int32_t at = s_run + block_exclusive_scan<int32_t>(sum, tmp, &tot);
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (i0 + u < nA) a.aoff[i0 + u] = at;
            at += d[u];
        }
        if (threadIdx.x == 0) s_run += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.aoff[nA] = s_run;
        HubDev &h = *a.hd;
        h.nA = nA;
        h.nE = s_run;
        h.nR = h.nQs = h.nQ = h.nMid = h.nBig = h.nTouch = h.cursor = h.work = h.work_mid = 0;
        atomicAdd(&a.st->tier_a[1], (unsigned long long)nA);
        atomicAdd(&a.st->tier_m[1], (unsigned long long)s_run);
    }
}

// Counts the anchors adjacent to every middle vertex past the hubs; an edge's
// place in its middle vertex's list is the count it found.
__global__ void k_hub_count(HubArgs a) {
    const int32_t nE = a.hd->nE, nA = a.hd->nA;
    // (64-bit positions: one past the last step may exceed 2^31)
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x; b < nE; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = b + threadIdx.x;
        bool fresh = false;
        int32_t y = 0;
        if (e < nE) {
            int32_t lo = 0, hi = nA - 1;
            while (lo < hi) {
                const int32_t mid = (lo + hi + 1) >> 1;
                if (a.aoff[mid] <= e)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            const int32_t x = a.A[lo];
            y = a.adj_s[a.off_s[x] + a.plen[x] + (e - a.aoff[lo])];
            const int32_t k = atomicAdd(&a.cb[y].x, 1);
            fresh = k == 0;
            a.ey[e] = y;
            a.ek[e] = make_int2(lo, k);
        }
        warp_append(fresh, y, &a.hd->nTouch, a.touch);
    }
}

__global__ void k_hub_base(HubArgs a) {
    const int32_t n = a.hd->nTouch;
    const int lane = threadIdx.x & 31;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = b + threadIdx.x;
        const int32_t y = t < n ? a.touch[t] : -1;
        const int32_t c = y >= 0 ? a.cb[y].x : 0;
        int32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        int32_t base = 0;
        if (lane == 31) base = atomicAdd(&a.hd->cursor, inc);
        base = __shfl_sync(0xffffffffu, base, 31);
        if (y >= 0) a.cb[y].y = base + inc - c;
    }
}

__global__ void k_hub_fill(HubArgs a) {
    const int32_t nE = a.hd->nE;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nE;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int2 k = a.ek[e];
        a.alist[a.cb[a.ey[e]].y + k.y] = k.x;
    }
}

__global__ void k_hub_clear(HubArgs a) {
    const int32_t n = a.hd->nTouch;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x)
        a.cb[a.touch[t]] = make_int2(0, 0);
}

// The anchors' masks side by side, and their transpose: cols[h] has one bit
// per anchor. One warp per 32 anchors.
__global__ void k_hub_cols(HubArgs a) {
    const int lane = threadIdx.x & 31;
    const int32_t nA = a.st->nLb;
    const int32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (int32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g * 32 < nA; g += nw) {
        const int32_t i = g * 32 + lane;
        Mask m = {};
        if (i < nA) {
            m = load_mask(a.mask + (size_t)a.A[i] * HW);
            uint4 *o = (uint4 *)(a.amask + (size_t)i * HW);
            o[0] = make_uint4(m.w[0], m.w[1], m.w[2], m.w[3]);
            o[1] = make_uint4(m.w[4], m.w[5], m.w[6], m.w[7]);
        }
#pragma unroll
        for (int w = 0; w < HW; w++) {
            uint32_t mine = 0;
#pragma unroll
            for (int b = 0; b < 32; b++) {
                const uint32_t v = __ballot_sync(0xffffffffu, (m.w[w] >> b) & 1u);
                if (lane == b) mine = v;
            }
            a.cols[(size_t)(w * 32 + lane) * a.colw + g] = mine;
        }
    }
}

// G[h, h'] for h' < h: one CTA per 16 x 16 pairs, population counts of two
// columns. Stored as the B operands (k = h', n = h) of k_hub_quad's
// mma.m16n8k16, fragment by fragment: low digit, then the rest.
__global__ void __launch_bounds__(1024) k_hub_gram(HubArgs a) {
    __shared__ uint32_t ca[16][257], cb[16][257];
    __shared__ uint32_t s_v[4][256];
    int th = 0, r = blockIdx.x;
    while (r > th) r -= ++th;  // block -> (th, r), r <= th
    // four groups of threads, each a quarter of the words of a step
    const int grp = threadIdx.x >> 8, i = (threadIdx.x >> 4) & 15, j = threadIdx.x & 15;
    const int32_t W = (a.st->nLb + 31) >> 5;
    uint32_t v = 0;
    for (int32_t w0 = 0; w0 < W; w0 += 256) {
        const int32_t nw = min(256, W - w0);
        for (int t = threadIdx.x; t < 16 * 256; t += 1024) {
            const int row = t >> 8, c = t & 255;
            const bool in = c < nw;
            ca[row][c] = in ? a.cols[(size_t)(th * 16 + row) * a.colw + w0 + c] : 0u;
            cb[row][c] = in ? a.cols[(size_t)(r * 16 + row) * a.colw + w0 + c] : 0u;
        }
        __syncthreads();
        const int e = min(64, nw - grp * 64);
#pragma unroll 8
        for (int c = 0; c < e; c++) v += __popc(ca[i][grp * 64 + c] & cb[j][grp * 64 + c]);
        __syncthreads();
    }
    s_v[grp][threadIdx.x & 255] = v;
    __syncthreads();
    if (grp) return;
    v = s_v[0][threadIdx.x] + s_v[1][threadIdx.x] + s_v[2][threadIdx.x] + s_v[3][threadIdx.x];
    const int h = th * 16 + i, h2 = r * 16 + j;
    if (h2 >= h) v = 0;
    if (h2 < h) a.gtri[h * (h - 1) / 2 + h2] = v;
    const int nt = h >> 3, kt = r, idx = tile_index(kt, nt);
    const int fl = (h & 7) * 4 + ((j & 7) >> 1);  // lane that holds (k = j, n = h & 7)
    const size_t at = (size_t)idx * 128 + fl * 4 + (j >> 3) * 2 + (j & 1);
    __half *B = (__half *)a.gram;
    B[at] = __uint2half_rn(v & ((1u << DIGIT) - 1u));
    B[(size_t)TILES * 128 + at] = __uint2half_rn(v >> DIGIT);
    if (v >> DIGIT) atomicOr(&a.hd->flags[idx >> 5], 1u << (idx & 31));
}

// Rows of the quadratic form with at most this many hubs add up their entries
// of G one by one; the others go through the tensor cores, where 16 rows share
// the work of the tiles in which any of them has a hub.
constexpr int SPARSE_ROW = 24;

// Remaining vertices with a hub pair (rows of the quadratic form, sparse or
// not) and those that pull: not heavy, with neighbours past the hubs
// (one atomic per list and 1,024 vertices: with one per warp the three
// counters took 20 us a round on a million vertices).
__global__ void __launch_bounds__(256) k_hub_rows(HubArgs a) {
    __shared__ int32_t s_n[3], s_at[3];
    const int lane = threadIdx.x & 31;
    constexpr int U = 4;
    for (int64_t b = (int64_t)blockIdx.x * (256 * U); b < a.n; b += (int64_t)gridDim.x * (256 * U)) {
        if (threadIdx.x < 3) s_n[threadIdx.x] = 0;
        __syncthreads();
        int32_t x[U], pl[U], d[U];
        int which[U], pos[3][U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = b + u * 256 + threadIdx.x;
            x[u] = i < a.n && a.sub[i] < 0 ? (int32_t)i : -1;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            pl[u] = x[u] >= 0 ? a.plen[x[u]] : 0;
            d[u] = x[u] >= 0 ? (int32_t)(a.off_s[x[u] + 1] - a.off_s[x[u]]) : 0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            which[u] = (pl[u] >= 2 && pl[u] <= SPARSE_ROW ? 1 : 0) | (pl[u] > SPARSE_ROW ? 2 : 0) |
                       (x[u] >= HEAVY && d[u] > pl[u] ? 4 : 0);
#pragma unroll
            for (int l = 0; l < 3; l++) {
                const unsigned bal = __ballot_sync(0xffffffffu, which[u] >> l & 1);
                int at = 0;
                if (lane == 0 && bal) at = atomicAdd(&s_n[l], __popc(bal));
                pos[l][u] = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & lanemask_lt());
            }
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            int32_t *cnt = threadIdx.x == 0 ? &a.hd->nQs : threadIdx.x == 1 ? &a.hd->nQ : &a.hd->nR;
            s_at[threadIdx.x] = s_n[threadIdx.x] ? atomicAdd(cnt, s_n[threadIdx.x]) : 0;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (which[u] & 1) a.Qs[s_at[0] + pos[0][u]] = x[u];
            if (which[u] & 2) a.Q[s_at[1] + pos[1][u]] = x[u];
            if (which[u] & 4) a.R[s_at[2] + pos[2][u]] = x[u];
        }
    }
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// sup[x'] -= sum over h' < h in N_x' of G[h, h'] for every sparse row: one
// thread per row, G's triangle in shared memory.
constexpr int TRI = HUBS * (HUBS - 1) / 2;
__global__ void __launch_bounds__(1024, 1) k_hub_quad_sparse(HubArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *G = (uint32_t *)smem;
    const int32_t n = a.hd->nQs;
    if ((int32_t)blockIdx.x * 1024 >= n) return;
    for (int t = threadIdx.x; t < TRI / 4; t += 1024) ((uint4 *)G)[t] = ((const uint4 *)a.gtri)[t];
    __syncthreads();
    for (int32_t i = blockIdx.x * 1024 + threadIdx.x; i < n; i += gridDim.x * 1024) {
        const int32_t x = a.Qs[i];
        const int32_t *L = a.adj_s + a.off_s[x];
        const int32_t len = a.plen[x];
        unsigned long long q = 0;
        for (int32_t j = 1; j < len; j++) {
            const int32_t h = L[j];
            const uint32_t *row = G + h * (h - 1) / 2;
            for (int32_t k = 0; k < j; k++) q += row[L[k]];
        }
        if (q) atomicAdd(&a.sup[x], 0ull - q);
    }
}
static_assert(TRI % 4 == 0, "vector copy of the triangle");

// The same for the other rows. A warp takes
// 16 rows: Y = M G (M: the rows' masks as 0/1 halves, made in registers from
// the bits), then every row adds up the columns of Y whose bit it has. (With
// all rows here the 10M-edge graph's rounds took 158 us, with the sparse rows
// apart 48 + 60 side by side: their tiles are mostly checks.) Tiles
// in which none of the 16 rows has a bit are skipped. Two digits of G, the
// second only in the tiles flagged as having one. Exact: a digit is below
// 2^11, an entry of Y at most 256 x 2^11 = 2^19, 16 of them 2^23.
constexpr int QUAD_THREADS = 512;
__global__ void __launch_bounds__(QUAD_THREADS, 1) k_hub_quad(HubArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint2 *B = (uint2 *)smem;  // [2][TILES][32]
    __shared__ uint32_t s_flag[TILES / 32 + 1];
    __shared__ int s_any;
    const int32_t nQ = a.hd->nQ;
    const int lane = threadIdx.x & 31;
    const int32_t w0 = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int32_t nw = (QUAD_THREADS / 32) * gridDim.x;
    if ((int32_t)blockIdx.x * 16 >= nQ) return;
    if (threadIdx.x == 0) s_any = 0;
    __syncthreads();
    if (threadIdx.x < TILES / 32 + 1) {
        s_flag[threadIdx.x] = a.hd->flags[threadIdx.x];
        if (s_flag[threadIdx.x]) s_any = 1;
    }
    __syncthreads();
    const int nd = s_any ? 2 : 1;
    for (int t = threadIdx.x; t < nd * TILES * 16; t += QUAD_THREADS)
        ((uint4 *)B)[t] = ((const uint4 *)a.gram)[t];
    __syncthreads();
    const int g = lane >> 2, c2 = (lane & 3) * 2;
    for (int32_t t = w0; t * 16 < nQ; t += nw) {
        const int32_t i0 = t * 16 + g, i1 = i0 + 8;
        const int32_t x0 = i0 < nQ ? a.Q[i0] : -1, x1 = i1 < nQ ? a.Q[i1] : -1;
        Mask m0 = {}, m1 = {};
        if (x0 >= 0) m0 = load_mask(a.mask + (size_t)x0 * HW);
        if (x1 >= 0) m1 = load_mask(a.mask + (size_t)x1 * HW);
        uint32_t U[HW], ntm = 0;  // bits any row has; n tiles with one
#pragma unroll
        for (int w = 0; w < HW; w++) {
            U[w] = __reduce_or_sync(0xffffffffu, m0.w[w] | m1.w[w]);
#pragma unroll
            for (int b = 0; b < 4; b++) ntm |= ((U[w] >> (8 * b)) & 0xffu) ? 1u << (4 * w + b) : 0u;
        }
        unsigned long long q0 = 0, q1 = 0;
        for (int d = 0; d < nd; d++) {
            const uint2 *Bd = B + (size_t)d * TILES * 32 + lane;
#pragma unroll
            for (int part = 0; part < NT / 8; part++) {  // 8 n tiles at a time
                if (!((ntm >> (8 * part)) & 0xffu)) continue;
                float acc[8][4];
#pragma unroll
                for (int j = 0; j < 8; j++)
#pragma unroll
                    for (int k = 0; k < 4; k++) acc[j][k] = 0.f;
#pragma unroll
                for (int kt = 0; kt < KT; kt++) {
                    if (2 * kt >= 8 * (part + 1)) break;
                    if (!((U[kt >> 1] >> ((kt & 1) * 16)) & 0xffffu)) continue;
                    const uint32_t r0 = m0.w[kt >> 1] >> ((kt & 1) * 16),
                                   r1 = m1.w[kt >> 1] >> ((kt & 1) * 16);
                    // two bits -> two halves 0.0 / 1.0
                    auto pair = [](uint32_t bits) {
                        return (((bits & 3u) * 0x8001u) & 0x10001u) * 0x3c00u;
                    };
                    const uint32_t A[4] = {pair(r0 >> c2), pair(r1 >> c2), pair(r0 >> (c2 + 8)),
                                           pair(r1 >> (c2 + 8))};
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int nt = 8 * part + j;
                        if (nt < 2 * kt) continue;
                        const int idx = tile_index(kt, nt);
                        if (!((ntm >> nt) & 1u)) continue;
                        if (d && !((s_flag[idx >> 5] >> (idx & 31)) & 1u)) continue;
                        mma16816(acc[j], A, Bd[idx * 32]);
                    }
                }
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const int nt = 8 * part + j;
                    const uint32_t b0 = m0.w[nt >> 2] >> ((nt & 3) * 8 + c2),
                                   b1 = m1.w[nt >> 2] >> ((nt & 3) * 8 + c2);
                    s0 += (b0 & 1u) ? acc[j][0] : 0.f;
                    s0 += (b0 & 2u) ? acc[j][1] : 0.f;
                    s1 += (b1 & 1u) ? acc[j][2] : 0.f;
                    s1 += (b1 & 2u) ? acc[j][3] : 0.f;
                }
                q0 += (unsigned long long)(uint32_t)s0 << (DIGIT * d);
                q1 += (unsigned long long)(uint32_t)s1 << (DIGIT * d);
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            q0 += __shfl_xor_sync(0xffffffffu, q0, o);
            q1 += __shfl_xor_sync(0xffffffffu, q1, o);
        }
        if ((lane & 3) == 0) {
            if (q0) atomicAdd(&a.sup[x0], 0ull - q0);
            if (q1) atomicAdd(&a.sup[x1], 0ull - q1);
        }
    }
}

// ---- pull: wedges x' - y - x through middle vertices y past the hubs.
// Eight lanes per x' while its list has at most PULL8_DEG entries and its
// wedges at most PULL8_W; otherwise a warp, up to PULL_DEG entries and PULL_W
// wedges; otherwise a CTA. Every kernel finds the wedge count first and hands
// larger vertices on: the chain of dependent loads of one vertex (list, its
// entries, their anchors, the anchors' masks) is ~4 us however few its wedges
// are, so what counts is how many vertices are under way at once.
constexpr int PULL8_DEG = 64, PULL8_W = 64, PULL8_SLOTS = 128;
constexpr int PULL_DEG = 1024, PULL_W = 1024, PULL_SLOTS = 2048;

struct PullMids {
    const int32_t *adj_s;
    const int2 *cb;
    __device__ __forceinline__ void seg(int64_t q, int64_t &beg, int32_t &len) const {
        const int2 c = __ldg(cb + adj_s[q]);
        beg = c.y;
        len = c.x;
    }
};

// Occurrences of every anchor among one vertex's wedges. An occurrence adds
// the number of earlier ones: over b occurrences that is C(b, 2), so nothing
// has to be read back from the table. Open addressing at load <= 1/2, one word
// per slot: (anchor + 1) << 16 | count, 0 = empty.
struct PackedTable {
    uint32_t *slot;
    uint32_t mask;  // slots in use - 1
    __device__ __forceinline__ uint32_t add(int32_t key) {
        const uint32_t k = ((uint32_t)key + 1u) << 16;
        uint32_t h = (hash_key(key) >> 16) & mask;
        for (uint32_t p = 0; p <= mask; p++) {
            uint32_t cur = ((volatile uint32_t *)slot)[h];
            if (cur == 0) {
                cur = atomicCAS(&slot[h], 0u, k | 1u);
                if (cur == 0) return 0;
            }
            if ((cur ^ k) < 65536u) return atomicAdd(&slot[h], 1u) & 0xffffu;
            h = (h + 1) & mask;
        }
        return 0;
    }
};

__global__ void __launch_bounds__(256) k_hub_pull8(HubArgs a) {
    __shared__ __align__(16) uint32_t s_tab[32][PULL8_SLOTS];
    const int lane = threadIdx.x & 31, l8 = lane & 7, g8 = lane >> 3;
    const int grp = threadIdx.x >> 3;
    PackedTable T{s_tab[grp], PULL8_SLOTS - 1};
    for (int i = l8; i < PULL8_SLOTS; i += 8) T.slot[i] = 0;
    __syncwarp();
    const int32_t nR = a.hd->nR;
    const int32_t nw = (gridDim.x * blockDim.x) >> 5;
    unsigned long long cw = 0, cp = 0;
    for (int32_t b = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; b < nR; b += nw * 4) {
        const int32_t i = b + g8;
        int32_t x = 0, deg = 0;
        int64_t q0 = 0;
        if (i < nR) {
            x = a.R[i];
            q0 = a.off_s[x] + a.plen[x];
            deg = (int32_t)(a.off_s[x + 1] - q0);
        }
        bool on = deg > PULL_DEG;  // handed on, to which list
        bool wide = on, warp_sized = !on && deg > PULL8_DEG;
        if (deg > PULL8_DEG) deg = 0;
        int2 c[PULL8_DEG / 8];
        int32_t W = 0;
#pragma unroll
        for (int s = 0; s < PULL8_DEG / 8; s++) {
            c[s] = make_int2(0, 0);
            const int k = s * 8 + l8;
            if (k < deg) c[s] = __ldg(a.cb + a.adj_s[q0 + k]);
            W += c[s].x;
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) W += __shfl_xor_sync(0xffffffffu, W, o);
        if (W > PULL8_W) {
            wide |= W > PULL_W;
            warp_sized |= W <= PULL_W;
            W = 0;
        }
        warp_append(l8 == 0 && warp_sized, x, &a.hd->nMid, a.mid);
        warp_append(l8 == 0 && wide, x, &a.hd->nBig, a.big);
        if (!__any_sync(0xffffffffu, W > 0)) continue;
        uint32_t dec = 0;  // at most 64 x (256 + 63)
        if (W > 0) {
            const Mask mx = load_mask(a.mask + (size_t)x * HW);
#pragma unroll
            for (int s = 0; s < PULL8_DEG / 8; s++)
                for (int32_t k = 0; k < c[s].x; k++) {
                    const int32_t key = __ldg(a.alist + c[s].y + k);
                    const Mask ma = load_mask(a.amask + (size_t)key * HW);
                    dec += T.add(key);
                    dec += common(mx, ma);
                }
        }
        __syncwarp();
        if (W > 0)
            for (int i = l8; i < PULL8_SLOTS / 4; i += 8)
                ((uint4 *)T.slot)[i] = make_uint4(0, 0, 0, 0);
        __syncwarp();
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) dec += __shfl_xor_sync(0xffffffffu, dec, o);
        if (l8 == 0 && W > 0) {
            cw += (unsigned long long)W;
            if (dec) {
                cp++;
                atomicAdd(&a.sup[x], 0ull - (unsigned long long)dec);
            }
        }
    }
    cw = warp_sum(cw);
    cp = warp_sum(cp);
    if (lane == 0) {
        if (cw) atomicAdd(&a.st->tier_w[1], cw);
        if (cp) atomicAdd(&a.st->tier_p[1], cp);
    }
}

__global__ void __launch_bounds__(128) k_hub_pull_warp(HubArgs a) {
    __shared__ __align__(16) uint32_t s_tab[4][PULL_SLOTS];
    const int lane = threadIdx.x & 31;
    PackedTable T{s_tab[threadIdx.x >> 5], PULL_SLOTS - 1};
    for (int i = lane; i < PULL_SLOTS; i += 32) T.slot[i] = 0;
    __syncwarp();
    const int32_t n = a.hd->nMid;
    const int32_t nw = (gridDim.x * blockDim.x) >> 5;
    unsigned long long cw = 0, cp = 0;
    for (int32_t i = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; i < n;) {
        const int32_t x = a.mid[i];
        const int64_t q0 = a.off_s[x] + a.plen[x], q1 = a.off_s[x + 1];
        const Mask mx = load_mask(a.mask + (size_t)x * HW);
        int32_t W = 0;
        for (int64_t q = q0 + lane; q < q1; q += 32) W += __ldg(&a.cb[a.adj_s[q]].x);
        W = warp_sum(W);
        if (W > PULL_W) {
            if (lane == 0) a.big[atomicAdd(&a.hd->nBig, 1)] = x;
        } else if (W > 0) {
            // table of the smallest power of two that keeps the load at 1/2
            const uint32_t slots = max(64u, 2u << (32 - __clz(W - 1)));
            T.mask = slots - 1;
            uint32_t dec = 0;  // at most 1,024 x (256 + 1,023)
            for (int64_t qb = q0; qb < q1; qb += 32) {
                int2 c = make_int2(0, 0);
                if (qb + lane < q1) c = __ldg(a.cb + a.adj_s[qb + lane]);
                int32_t inc = c.x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += v;
                }
                const int32_t total = __shfl_sync(0xffffffffu, inc, 31), ex = inc - c.x;
                constexpr int U = 4;  // keys and masks of a lane in flight
                for (int32_t j0 = 0; j0 < total; j0 += 32 * U) {
                    int32_t key[U];
                    Mask ma[U];
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const int32_t j = j0 + u * 32 + lane;
                        int lo = 0;
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1) {
                            const int32_t e = __shfl_sync(0xffffffffu, ex, lo + step);
                            if (e <= j) lo += step;
                        }
                        const int32_t b = __shfl_sync(0xffffffffu, c.y, lo);
                        const int32_t e0 = __shfl_sync(0xffffffffu, ex, lo);
                        key[u] = j < total ? __ldg(a.alist + b + (j - e0)) : -1;
                    }
#pragma unroll
                    for (int u = 0; u < U; u++)
                        ma[u] = load_mask(a.amask + (size_t)max(key[u], 0) * HW);
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (key[u] >= 0) {
                            dec += T.add(key[u]);
                            dec += common(mx, ma[u]);
                        }
                }
            }
            dec = __reduce_add_sync(0xffffffffu, dec);
            for (uint32_t t = lane; t < slots / 4; t += 32)
                ((uint4 *)T.slot)[t] = make_uint4(0, 0, 0, 0);
            __syncwarp();
            cw += (unsigned long long)W;
            if (lane == 0 && dec) {
                cp++;
                atomicAdd(&a.sup[x], 0ull - (unsigned long long)dec);
            }
        }
        if (n <= nw) break;
        if (lane == 0) i = nw + atomicAdd(&a.hd->work_mid, 1);
        i = __shfl_sync(0xffffffffu, i, 0);
    }
    if (lane == 0) {
        if (cw) atomicAdd(&a.st->tier_w[1], cw);
        if (cp) atomicAdd(&a.st->tier_p[1], cp);
    }
}

// Two 16-bit counters per word over the activeSet's index space: key k < half
// in the low half of word k, the others in the high half of word k - half.
// As in PackedTable, an occurrence adds the number of earlier ones.
struct PullVisit {
    uint32_t *cnt;
    int32_t half;
    const uint32_t *amask;
    Mask mx;
    unsigned long long dec;
    template <int N>
    __device__ __forceinline__ void many(const int (&)[N], const int32_t (&key)[N]) {
        uint32_t d = 0;
#pragma unroll
        for (int u0 = 0; u0 < N; u0 += 4) {
            Mask ma[4];
#pragma unroll
            for (int u = 0; u < 4; u++)
                ma[u] = load_mask(amask + (size_t)max(key[u0 + u], 0) * HW);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int32_t k = key[u0 + u];
                if (k < 0) continue;
                const bool hi = k >= half;
                const uint32_t old = atomicAdd(&cnt[hi ? k - half : k], hi ? 0x10000u : 1u);
                d += (hi ? old >> 16 : old & 0xffffu) + common(mx, ma[u]);
            }
        }
        dec += d;
    }
};

// One CTA per x' with more wedges. The counters are sized for the activeSet
// (a few thousand keys: several CTAs per SM, whose barrier-separated phases
// overlap) and cleared whole after the walk.
constexpr int PULL_THREADS = 256;
__global__ void __launch_bounds__(PULL_THREADS) k_hub_pull_cta(HubArgs a, int32_t words) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_idx;
    __shared__ unsigned long long s_dec;
    const int32_t nBig = a.hd->nBig;
    if ((int32_t)blockIdx.x >= nBig) return;
    uint32_t *cnt = (uint32_t *)smem;
    Chunk ch;
    ch.beg = (int64_t *)(cnt + words);
    ch.pre = (int32_t *)(ch.beg + PULL_THREADS);
    ch.tmp = ch.pre + PULL_THREADS + 1;
    ch.len = chunk_len_ptr(ch.tmp);
    const int32_t half = (a.hd->nA + 1) >> 1, half4 = (half + 3) >> 2;
    for (int i = threadIdx.x; i < half4; i += PULL_THREADS) ((uint4 *)cnt)[i] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) s_dec = 0;
    __syncthreads();
    PullMids M{a.adj_s, a.cb};
    unsigned long long cw = 0, cp = 0;
    for (int idx = blockIdx.x; idx < nBig;) {
        const int32_t x = a.big[idx];
        PullVisit v{cnt, half, a.amask, load_mask(a.mask + (size_t)x * HW), 0};
        cw += cta_walk(M, a.off_s[x] + a.plen[x], a.off_s[x + 1], a.alist, ch, v);
        for (int i = threadIdx.x; i < half4; i += PULL_THREADS)
            ((uint4 *)cnt)[i] = make_uint4(0, 0, 0, 0);
        unsigned long long dec = v.dec;
        dec = warp_sum(dec);
        if ((threadIdx.x & 31) == 0 && dec) atomicAdd(&s_dec, dec);
        if (threadIdx.x == 0) s_idx = (int)gridDim.x + atomicAdd(&a.hd->work, 1);
        __syncthreads();
        idx = s_idx;
        if (threadIdx.x == 0) {
            if (s_dec) {
                cp++;
                atomicAdd(&a.sup[x], 0ull - s_dec);
            }
            s_dec = 0;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (cw) atomicAdd(&a.st->tier_w[1], cw);
        if (cp) atomicAdd(&a.st->tier_p[1], cp);
    }
}

// ---- the HEAVY vertices of highest degree, anchor by anchor: lane l of a
// warp counts b(x, x') for x' = 32 w + l, w < 8, from the masks of the
// anchor's middle vertices over those vertices. Anchors of many edges take a
// whole CTA (partial counts in shared memory): from 256 / 1,024 / 8,192 edges on the
// coarse-grained step of the 40M-edge graph takes 333 / 334 / 345 ms, of a 6M-edge
// one with hubs on both sides 84.6 / 85.0 / 86.7.
constexpr int HEAVY_DEG = 1024;
__global__ void __launch_bounds__(512) k_hub_heavy(HubArgs a) {
    __shared__ unsigned long long s_dec[HEAVY];
    __shared__ int32_t s_b[HEAVY];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t nA = a.hd->nA;
    for (int t = threadIdx.x; t < HEAVY; t += 512) {
        s_dec[t] = 0;
        s_b[t] = 0;
    }
    __syncthreads();
    unsigned long long dec[8] = {};
    int32_t b[8];
    // counts of edges e0 + 4 step, step += stride, up to e1
    auto count = [&](int32_t e0, int32_t e1, int32_t first, int32_t stride) {
        for (int64_t e = e0 + first * 4; e < e1; e += stride * 4) {
            // lane: word (lane & 7) of the mask of edge e + (lane >> 3)
            const int64_t k = e + (lane >> 3);
            const uint32_t word =
                k < e1 ? __ldg(a.heavy + (size_t)a.ey[k] * HW + (lane & 7)) : 0u;
            if (!__any_sync(0xffffffffu, word)) continue;
#pragma unroll
            for (int s = 0; s < 32; s++) {
                const uint32_t v = __shfl_sync(0xffffffffu, word, s);
                b[s & 7] += (v >> lane) & 1u;
            }
        }
    };
    auto finish = [&](int32_t i) {
        const Mask ma = load_mask(a.amask + (size_t)i * HW);
#pragma unroll
        for (int w = 0; w < 8; w++) {
            const int32_t x = w * 32 + lane;
            if (b[w] > 0 && x < a.n) {
                const uint32_t m = common(ma, load_mask(a.mask + (size_t)x * HW));
                dec[w] += (unsigned long long)b[w] * m + choose2((unsigned long long)b[w]);
            }
        }
    };
    const int32_t gw = warp * gridDim.x + blockIdx.x, nw = 16 * gridDim.x;
    for (int32_t i = gw; i < nA; i += nw) {
        const int32_t e0 = a.aoff[i], e1 = a.aoff[i + 1];
        if (e1 - e0 > HEAVY_DEG || e1 == e0) continue;
#pragma unroll
        for (int w = 0; w < 8; w++) b[w] = 0;
        count(e0, e1, 0, 1);
        finish(i);
    }
    for (int32_t i = blockIdx.x; i < nA; i += gridDim.x) {
        const int32_t e0 = a.aoff[i], e1 = a.aoff[i + 1];
        if (e1 - e0 <= HEAVY_DEG) continue;
#pragma unroll
        for (int w = 0; w < 8; w++) b[w] = 0;
        count(e0, e1, warp, 16);
#pragma unroll
        for (int w = 0; w < 8; w++)
            if (b[w]) atomicAdd(&s_b[w * 32 + lane], b[w]);
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int w = 0; w < 8; w++) {
                b[w] = s_b[w * 32 + lane];
                s_b[w * 32 + lane] = 0;
            }
            finish(i);
        }
        __syncthreads();
    }
#pragma unroll
    for (int w = 0; w < 8; w++)
        if (dec[w]) atomicAdd(&s_dec[w * 32 + lane], dec[w]);
    __syncthreads();
    for (int t = threadIdx.x; t < HEAVY; t += 512)
        if (s_dec[t] && a.sub[t] < 0) atomicAdd(&a.sup[t], 0ull - s_dec[t]);
}

constexpr size_t quad_smem() { return (size_t)2 * TILES * 256; }

}  // namespace

size_t HubPath::bytes(int64_t m, int64_t n, int64_t n_o) {
    return 16 * (size_t)m + (4 * HW + 24) * (size_t)n + (4 * HW + 12) * (size_t)n_o +
           (size_t)MAX_ANCHORS * (4 * HW + 4 + HUBS / 8) + 4 * (size_t)TRI + 512 * (size_t)TILES;
}

bool HubPath::init(const Decomp &D, cudaStream_t s) {
    const Side &S = *D.S, &O = *D.O;
    const int32_t n = D.n;
    if (!(mask_.try_alloc((size_t)n * HW, s) && plen_.try_alloc(n, s) &&
          heavy_.try_alloc((size_t)O.n * HW, s) && cb_.try_alloc(O.n, s) && touch_.try_alloc(O.n, s) &&
          Qs_.try_alloc(n, s) && Q_.try_alloc(n, s) && mid_.try_alloc(n, s) && R_.try_alloc(n, s) &&
          big_.try_alloc(n, s) && gtri_.try_alloc(TRI, s) && aoff_.try_alloc(MAX_ANCHORS + 1, s) &&
          amask_.try_alloc((size_t)MAX_ANCHORS * HW, s) &&
          cols_.try_alloc((size_t)HUBS * (MAX_ANCHORS / 32), s) &&
          gram_.try_alloc((size_t)2 * TILES * 64, s) && ey_.try_alloc(D.m, s) && ek_.try_alloc(D.m, s) &&
          alist_.try_alloc(D.m, s) && hd_.try_alloc(1, s))) {
        for (DevBuf<uint32_t> *b : {&mask_, &heavy_, &amask_, &cols_, &gram_, &gtri_}) b->release();
        for (DevBuf<int32_t> *b : {&plen_, &touch_, &Qs_, &Q_, &R_, &mid_, &big_, &aoff_, &ey_, &alist_})
            b->release();
        for (DevBuf<int2> *b : {&cb_, &ek_}) b->release();
        return false;
    }
    for (cudaEvent_t &e : ev_) RC_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    cb_.zero();
    hd_.zero();
    const int grid = num_sms() * 16;
    k_prefix_masks<<<grid, 256, 0, s>>>(S.off, S.adj, n, mask_.get(), plen_.get());
    RC_LAUNCH();
    k_prefix_masks<<<grid, 256, 0, s>>>(O.off, O.adj, O.n, heavy_.get(), nullptr);
    RC_LAUNCH();
    allow_max_smem((const void *)k_hub_quad_sparse);
    allow_max_smem((const void *)k_hub_quad);
    allow_max_smem((const void *)k_hub_pull_cta);
    return true;
}

void HubPath::round(const Decomp &D, CdDev *st, const int32_t *A, int32_t nF, cudaStream_t s) {
    const int sms = num_sms();
    const HubArgs a{D.n,         D.S->off,    D.S->adj,    D.sup,        D.sub,       st,
                    A,           mask_.get(), plen_.get(), heavy_.get(), cb_.get(),   touch_.get(),
                    Qs_.get(),   Q_.get(),    R_.get(),    mid_.get(),   big_.get(),  aoff_.get(),
                    amask_.get(), cols_.get(), MAX_ANCHORS / 32, gram_.get(), gtri_.get(), ey_.get(), ek_.get(), alist_.get(), hd_.get()};
    // three branches: the hub part (columns, Gram matrix, quadratic forms),
    // the heavy vertices, the pull; their decrements are atomic
    cudaStream_t sq = tier_stream(0), sh = tier_stream(1);
    struct ForkGuard {  // left by an error, the buffers wait for the branches
        cudaStream_t q, h;
        bool joined = false;
        ~ForkGuard() {
            if (joined) return;
            cudaStreamSynchronize(q);
            cudaStreamSynchronize(h);
        }
    } fg{sq, sh};
    k_hub_begin<<<1, 1024, 0, s>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaEventRecord(ev_[0], s));
    RC_CUDA(cudaStreamWaitEvent(sq, ev_[0], 0));
    k_hub_cols<<<sms, 256, 0, sq>>>(a);
    RC_LAUNCH();
    k_hub_rows<<<std::min(ceil_div(D.n, 1024), sms * 8), 256, 0, sq>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaEventRecord(ev_[1], sq));
    k_hub_gram<<<(HUBS / 16) * (HUBS / 16 + 1) / 2, 1024, 0, sq>>>(a);
    RC_LAUNCH();
    k_hub_quad_sparse<<<sms, 1024, TRI * 4, sq>>>(a);
    RC_LAUNCH();
    k_hub_quad<<<sms, QUAD_THREADS, quad_smem(), sq>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaEventRecord(ev_[2], sq));
    k_hub_count<<<sms * 8, 256, 0, s>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaEventRecord(ev_[3], s));
    k_hub_base<<<sms * 4, 256, 0, s>>>(a);
    RC_LAUNCH();
    k_hub_fill<<<sms * 8, 256, 0, s>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaStreamWaitEvent(sh, ev_[1], 0));
    RC_CUDA(cudaStreamWaitEvent(sh, ev_[3], 0));
    k_hub_heavy<<<sms, 512, 0, sh>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaEventRecord(ev_[4], sh));
    RC_CUDA(cudaStreamWaitEvent(s, ev_[1], 0));
    k_hub_pull8<<<sms * 8, 256, 0, s>>>(a);
    RC_LAUNCH();
    k_hub_pull_warp<<<sms * 6, 128, 0, s>>>(a);
    RC_LAUNCH();
    {
        // counters for at most nF anchors, as many CTAs as fit
        const int32_t words = (((nF + 1) >> 1) + 3) & ~3;
        const size_t smem = (size_t)words * 4 + chunk_bytes(PULL_THREADS);
        int occ = 1;
        RC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_hub_pull_cta, PULL_THREADS,
                                                              smem));
        k_hub_pull_cta<<<sms * std::max(1, occ), PULL_THREADS, smem, s>>>(a, words);
    }
    RC_LAUNCH();
    k_hub_clear<<<sms * 4, 256, 0, s>>>(a);
    RC_LAUNCH();
    RC_CUDA(cudaStreamWaitEvent(s, ev_[2], 0));
    RC_CUDA(cudaStreamWaitEvent(s, ev_[4], 0));
    fg.joined = true;
}

HubPath::~HubPath() {
    for (cudaEvent_t e : ev_)
        if (e) cudaEventDestroy(e);
}

bool HubPath::suits(const Decomp &D, cudaStream_t s) {
    if (D.m == 0) return false;
    DevBuf<unsigned long long> w(2, s);
    w.zero();
    k_hub_probe<<<1, HUBS, 0, s>>>(D.O->off, D.O->n, D.S->off, D.n, w.get());
    RC_LAUNCH();
    unsigned long long h[2] = {0, 0};
    RC_CUDA(cudaMemcpyAsync(h, w.get(), sizeof(h), cudaMemcpyDeviceToHost, s));
    RC_CUDA(cudaStreamSynchronize(s));
    return 2 * h[0] >= D.wedges_bup && h[1] < 65535;
}

}  // namespace receipt
