// Device primitives used by the CSR build and the fine-grained setup:
// an exclusive prefix scan (reduce, scan of tile totals, scan-and-add) and a
// stable LSD radix sort (tile histograms, offsets, stable scatter ranked by
// warp match).
#include <cstdio>

#include "common.cuh"

namespace receipt {

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 16;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
__global__ void k_tile_sums(const T *__restrict__ in, int64_t n, T *__restrict__ sums) {
    __shared__ T tmp[33];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    T s = 0;
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        int64_t g = base + i;
        if (g < n) s += in[g];
    }
    T tot;
    block_exclusive_scan<T>(s, tmp, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// `in` may be `out`: a block reads its tile before it writes it, and no other.
template <typename T>
__global__ void k_tile_scan(const T *in, T *out, int64_t n, const T *__restrict__ offsets) {
    __shared__ T tile[SCAN_TILE];
    __shared__ T tmp[33];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        int64_t g = base + i;
        tile[i] = g < n ? in[g] : T(0);
    }
    __syncthreads();
    T loc[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        loc[j] = s;
        s += tile[threadIdx.x * SCAN_ITEMS + j];
    }
    T tot;
    T pre = block_exclusive_scan<T>(s, tmp, &tot);
    T off = (offsets ? offsets[blockIdx.x] : T(0)) + pre;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) tile[threadIdx.x * SCAN_ITEMS + j] = loc[j] + off;
    __syncthreads();
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        int64_t g = base + i;
        if (g < n) out[g] = tile[i];
    }
}

}  // namespace

template <typename T>
void scan_exclusive(const T *d_in, T *d_out, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (tiles == 1) {
        k_tile_scan<T><<<1, SCAN_THREADS, 0, s>>>(d_in, d_out, n, nullptr);
        RC_LAUNCH();
        return;
    }
    DevBuf<T> sums(tiles, s), offs(tiles, s);
    k_tile_sums<T><<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(d_in, n, sums.get());
    RC_LAUNCH();
    scan_exclusive<T>(sums.get(), offs.get(), tiles, s);
    k_tile_scan<T><<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(d_in, d_out, n, offs.get());
    RC_LAUNCH();
}

template void scan_exclusive<int64_t>(const int64_t *, int64_t *, int64_t, cudaStream_t);
template void scan_exclusive<uint64_t>(const uint64_t *, uint64_t *, int64_t, cudaStream_t);
template void scan_exclusive<uint32_t>(const uint32_t *, uint32_t *, int64_t, cudaStream_t);
template void scan_exclusive<int32_t>(const int32_t *, int32_t *, int64_t, cudaStream_t);

// ---------------------------------------------------------------------
// Radix sort
//
// Three launches a pass: digit counts of every tile, offsets (a block per 32
// digits runs down the tiles), scatter. Small sorts are bound by launches and
// by each kernel's dependent steps, large ones by the scatter's writes of
// whole sectors; so digits have up to RS_MAX_BITS bits, as even as the key's
// bits allow (a pass fewer for 17 to 20 and 33 to 40 bits than with 8), and
// tiles shrink while there are few of them. The scatter matches each key's
// digit once within its warp. The last pass can write int32 fields of the keys
// instead of (or beside) the keys. 10M keys: 0.16 ms a pass (0.13 the scatter's
// writes); 10 bits against 8: a 10M-edge build 2.55 / 2.79 ms, with 8 keys a
// thread 2.64. Before, with 8-bit digits, a general scan a pass and three sorts
// of whole edges a build: builds of 20k / 1M / 10M / 40M edges 0.49 / 1.27 /
// 5.05 / 22.3 ms, now 0.27 / 0.55 / 2.6 / 9.3.
// ---------------------------------------------------------------------
namespace {

constexpr int RS_WARPS = 8;
constexpr int RS_THREADS = RS_WARPS * 32;
constexpr int RS_MAX_BITS = 10;

template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint64_t *__restrict__ keys, int64_t n,
                                                        int shift, uint32_t dmask, int D,
                                                        uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[1 << RS_MAX_BITS];
    for (int i = threadIdx.x; i < D; i += RS_THREADS) h[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * (RS_THREADS * ITEMS);
    uint64_t k[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const int64_t g = base + j * RS_THREADS + threadIdx.x;
        k[j] = g < n ? keys[g] : 0;
    }
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const int64_t g = base + j * RS_THREADS + threadIdx.x;
        if (g < n) atomicAdd(&h[(uint32_t)(k[j] >> shift) & dmask], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < D; d += RS_THREADS) hist[(int64_t)blockIdx.x * D + d] = h[d];
}

// Column sums of hist[ntiles][D] become exclusive prefixes down the tiles;
// total[d]: keys of digit d. A block per 32 digits.
__global__ void __launch_bounds__(1024) k_rs_offsets(uint32_t *__restrict__ hist, int ntiles, int D,
                                                     uint32_t *__restrict__ total) {
    __shared__ uint32_t s[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (ntiles + 31) / 32;
    const int r0 = min(warp * per, ntiles), r1 = min(r0 + per, ntiles);
    uint32_t *col = hist + blockIdx.x * 32 + lane;
    uint32_t sum = 0;
#pragma unroll 4
    for (int r = r0; r < r1; r++) sum += col[(int64_t)r * D];
    s[warp][lane] = sum;
    __syncthreads();
    // warp w scans digit w's 32 partial sums
    const uint32_t v = s[lane][warp];
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    s[lane][warp] = inc - v;
    if (lane == 31) total[blockIdx.x * 32 + warp] = inc;
    __syncthreads();
    uint32_t run = s[warp][lane];
#pragma unroll 4
    for (int r = r0; r < r1; r++) {
        const uint32_t c = col[(int64_t)r * D];
        col[(int64_t)r * D] = run;
        run += c;
    }
}

template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS)
    k_rs_scatter(const uint64_t *__restrict__ kin, uint64_t *__restrict__ kout, RadixField out,
                 int64_t n, int shift, uint32_t dmask, int D, const uint32_t *__restrict__ hist,
                 const uint32_t *__restrict__ total) {
    extern __shared__ uint32_t smem[];
    __shared__ uint32_t tmp[33];
    uint32_t *gbase = smem;                         // D: output position of the tile's first key
    uint16_t *wcnt = (uint16_t *)(smem + D);        // [warp][D]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < RS_WARPS * D / 2; i += RS_THREADS) ((uint32_t *)wcnt)[i] = 0;
    const int64_t wbase = ((int64_t)blockIdx.x * RS_WARPS + warp) * (32 * ITEMS);
    uint64_t k[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const int64_t g = wbase + j * 32 + lane;
        k[j] = g < n ? kin[g] : 0;
    }
    // digits' first positions: scan of the totals, plus the tiles before
    {
        const int per = (D + RS_THREADS - 1) / RS_THREADS;  // 1 to 4
        uint32_t t[4], sum = 0;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int d = threadIdx.x * per + e;
            t[e] = e < per && d < D ? total[d] : 0;
            sum += t[e];
        }
        uint32_t run = block_exclusive_scan<uint32_t>(sum, tmp, nullptr);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int d = threadIdx.x * per + e;
            if (e < per && d < D) gbase[d] = run + hist[(int64_t)blockIdx.x * D + d];
            run += t[e];
        }
    }
    __syncthreads();
    uint16_t *cnt = wcnt + warp * D;
    uint16_t rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const bool in = wbase + j * 32 + lane < n;
        const uint32_t d = (uint32_t)(k[j] >> shift) & dmask;
        const unsigned peers = __match_any_sync(0xffffffffu, in ? (int)d : -1);
        const unsigned before = in ? cnt[d] : 0;
        __syncwarp();
        if (in && (__ffs(peers) - 1) == lane) cnt[d] = (uint16_t)(before + __popc(peers));
        __syncwarp();
        rank[j] = (uint16_t)(before + __popc(peers & lanemask_lt()));
    }
    __syncthreads();
    for (int d = threadIdx.x; d < D; d += RS_THREADS) {
        unsigned run = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; w++) {
            const unsigned c = wcnt[w * D + d];
            wcnt[w * D + d] = (uint16_t)run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        if (wbase + j * 32 + lane >= n) continue;
        const uint32_t d = (uint32_t)(k[j] >> shift) & dmask;
        const uint32_t pos = gbase[d] + cnt[d] + rank[j];
        if (kout) kout[pos] = k[j];
        if (out.dst) out.dst[pos] = (int32_t)((k[j] >> out.shift) & out.mask);
    }
}

__global__ void k_field(const uint64_t *__restrict__ key, int64_t n, RadixField out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out.dst[i] = (int32_t)((key[i] >> out.shift) & out.mask);
}

template <int ITEMS>
void radix_sort_tiles(DevBuf<uint64_t> &keys, int64_t n, int begin_bit, int end_bit, RadixField out,
                      bool want_keys, cudaStream_t s) {
    const int passes = (end_bit - begin_bit + RS_MAX_BITS - 1) / RS_MAX_BITS;
    const int64_t ntiles = (n + RS_THREADS * ITEMS - 1) / (RS_THREADS * ITEMS);
    const int dmax = 1 << RS_MAX_BITS;
    DevBuf<uint64_t> other(passes > 1 || want_keys ? n : 1, s);
    DevBuf<uint32_t> hist(ntiles * dmax, s), total(dmax, s);
    int shift = begin_bit;
    for (int p = 0; p < passes; p++) {
        const int bits = (end_bit - shift + passes - p - 1) / (passes - p);
        const int D = std::max(32, 1 << bits);
        const uint32_t dmask = (1u << bits) - 1u;
        const bool last = p == passes - 1;
        k_rs_hist<ITEMS><<<(unsigned)ntiles, RS_THREADS, 0, s>>>(keys.get(), n, shift, dmask, D,
                                                                 hist.get());
        RC_LAUNCH();
        k_rs_offsets<<<D / 32, 1024, 0, s>>>(hist.get(), (int)ntiles, D, total.get());
        RC_LAUNCH();
        k_rs_scatter<ITEMS><<<(unsigned)ntiles, RS_THREADS, 4 * D + 2 * RS_WARPS * D, s>>>(
            keys.get(), last && !want_keys ? nullptr : other.get(), last ? out : RadixField{}, n,
            shift, dmask, D, hist.get(), total.get());
        RC_LAUNCH();
        if (!last || want_keys) std::swap(keys, other);
        shift += bits;
    }
}

}  // namespace

void radix_sort(DevBuf<uint64_t> &keys, int64_t n, int begin_bit, int end_bit, cudaStream_t s,
                RadixField out, bool want_keys) {
    if (n >= (int64_t)UINT32_MAX) fail(RECEIPT_ERR_OVERFLOW, "radix sort of 2^32 - 1 keys or more");
    if (n <= 0) return;
    if (n == 1 || end_bit <= begin_bit) {
        if (out.dst) {
            k_field<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(keys.get(), n, out);
            RC_LAUNCH();
        }
        return;
    }
    // 4,096 keys a tile, 1,024 while that leaves SMs without a tile
    if (n >= (1 << 21))
        radix_sort_tiles<16>(keys, n, begin_bit, end_bit, out, want_keys, s);
    else
        radix_sort_tiles<4>(keys, n, begin_bit, end_bit, out, want_keys, s);
}

}  // namespace receipt
