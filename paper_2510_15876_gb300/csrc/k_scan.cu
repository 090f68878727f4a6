// k_scan.cu -- exclusive prefix sum of uint32 counts (bin offsets of the
// counting sorts in ingest and reprojection), with the clearing and filling
// that the sort around it needs (ScanWith). Two launches: per-block sums, and
// a per-block scan whose prefix every block adds up from the sums before it
// (beyond kDirectBlocks blocks a launch between scans the sums first, so that
// the work does not grow with the square of their number). out has n + 1
// entries; out[n] is the total.
//
// Bound: HBM at large n (every array once, 256-bit accesses), launches at small
// n: with a launch of its own for the sums, 32-byte strided reads, and separate
// launches for the cursor copy, the clearing and the fill, a reprojection's
// share was nine operations (30 us at 1920x1080, 20 us at 128x128), now two
// (10 and 4.5 us).
#include "afr_internal.cuh"

namespace afr {
namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr size_t kDirectBlocks = 2048;   // 8.4M counts: a block reads at most 8 KB of sums

struct Items {
    uint32_t v[kScanItems];
};

__device__ __forceinline__ Items load_items(const uint32_t *p, size_t i, size_t n) {
    Items r;
    if (i + kScanItems <= n) {
        asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
              "=r"(r.v[7])
            : "l"(p + i)
            : "memory");   // not before grid_order's wait
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) r.v[k] = i + k < n ? p[i + k] : 0u;
    }
    return r;
}

__device__ __forceinline__ void store_items(uint32_t *p, size_t i, size_t n, const Items &r, bool wide = true) {
    if (wide && i + kScanItems <= n) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p + i), "r"(r.v[0]), "r"(r.v[1]),
                     "r"(r.v[2]), "r"(r.v[3]), "r"(r.v[4]), "r"(r.v[5]), "r"(r.v[6]), "r"(r.v[7])
                     : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k)
            if (i + k < n) p[i + k] = r.v[k];
    }
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Block-wide exclusive scan of one value per thread; returns the block total
// through *total.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *total) {
    __shared__ uint32_t warp_sums[kScanThreads / 32];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = warp_incl_scan(v);
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kScanThreads / 32 ? warp_sums[lane] : 0u;
        uint32_t wi = warp_incl_scan(w);
        if (lane < kScanThreads / 32) warp_sums[lane] = wi - w;
        if (lane == kScanThreads / 32 - 1) *total = wi;
    }
    __syncthreads();
    uint32_t r = warp_sums[warp] + incl - v;
    __syncthreads();
    return r;
}

// Sum of one value per thread, returned to every thread.
__device__ __forceinline__ uint32_t block_sum(uint32_t v) {
    __shared__ uint32_t ws[kScanThreads / 32];
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) t += ws[w];
    return t;
}

__global__ void __launch_bounds__(kScanThreads) k_block_sums(const uint32_t *in, size_t n, uint32_t *sums) {
    grid_order();
    const Items r = load_items(in, (size_t)blockIdx.x * kScanTile + (size_t)threadIdx.x * kScanItems, n);
    uint32_t acc = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) acc += r.v[k];
    const uint32_t t = block_sum(acc);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
}

// Scans nb block sums in place (exclusive) with one block.
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(uint32_t *sums, size_t nb) {
    grid_order();
    __shared__ uint32_t carry;
    __shared__ uint32_t tot;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (size_t base = 0; base < nb; base += kScanThreads) {
        size_t i = base + threadIdx.x;
        uint32_t v = i < nb ? sums[i] : 0u;
        uint32_t ex = block_excl_scan(v, &tot);
        if (i < nb) sums[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

// scanned: sums holds exclusive prefixes already; wide: out is 32-byte aligned
// (a caller's own array need not be)
__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(uint32_t *in, uint32_t *out, size_t n,
                                                              Fresh<uint32_t> sums, bool scanned, bool wide, ScanWith with) {
    grid_order();
    __shared__ uint32_t tot;
    const size_t base = (size_t)blockIdx.x * kScanTile + (size_t)threadIdx.x * kScanItems;
    Items r = load_items(in, base, n);
    uint32_t before = 0;
    if (!scanned)
        for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kScanThreads) before += sums[i];
    uint32_t acc = 0, most = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        acc += r.v[k];
        most = max(most, r.v[k]);
    }
    const uint32_t prefix = scanned ? sums[blockIdx.x] : block_sum(before);
    uint32_t ex = block_excl_scan(acc, &tot) + prefix;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const uint32_t c = r.v[k];
        r.v[k] = ex;
        ex += c;
    }
    if (with.crowded && most > with.crowded_from) *with.crowded = 1ull;
    store_items(out, base, n, r, wide);
    if (with.cursor) store_items(with.cursor, base, n, r);
    const Items zero{};
    if (with.clear_in) store_items(in, base, n, zero);
    if (with.fill) {
        Items f;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) f.v[k] = with.fill_value;
        store_items(with.fill, base, n, f);
    }
    if (threadIdx.x == 0) {
        if (blockIdx.x == gridDim.x - 1) out[n] = prefix + tot;
        if (blockIdx.x == 0) {
            if (with.counter_from) {
                *with.counter_to = *with.counter_from;
                *with.counter_from = 0ull;
            }
            if (with.counter_zero) *with.counter_zero = 0ull;
        }
    }
}

}  // namespace

size_t scan_tmp_elems(size_t n) { return (n + kScanTile - 1) / kScanTile + 2; }

cudaError_t scan_exclusive(uint32_t *in, uint32_t *out, size_t n, uint32_t *tmp, cudaStream_t s, const ScanWith &with) {
    size_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 0) {
        return cudaMemsetAsync(out, 0, sizeof(uint32_t), s);
    }
    const bool scanned = nb > kDirectBlocks, wide = reinterpret_cast<uintptr_t>(out) % 32 == 0;
    launch_next(k_block_sums, dim3((unsigned)nb), dim3(kScanThreads), 0, s, in, n, tmp);   // after the caller's counting
    if (scanned) launch_next(k_scan_sums, dim3(1), dim3(kScanThreads), 0, s, tmp, nb);
    launch_next(k_scan_tiles, dim3((unsigned)nb), dim3(kScanThreads), 0, s, in, out, n, tmp, scanned, wide, with);
    return cudaGetLastError();
}

}  // namespace afr
