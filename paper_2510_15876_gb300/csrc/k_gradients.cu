// k_gradients.cu -- sections 4 and 4.1 on the deep buffer.
//
//  pixel pass   (thread per pixel on queues staged in shared memory): age
//               weights exp(-3.47 a), weighted mean luminance and its weighted
//               spread (per-pixel moments for the tile variance), the sum of
//               the ages, and the temporal gradient over the queue sorted by
//               time.
//  tile pass    (block per tile, warp per small one): G_x, G_y from the four neighbours' means,
//               the gradient and age sums and the tile's luminance moments
//               (mean first, then the squares about it).
#include "afr_internal.cuh"

namespace afr {
namespace {

// ---- pixel pass ------------------------------------------------------------------
// A warp takes 32 pixels: it copies their times and colours (contiguous in
// memory) to shared memory with asynchronous 16-byte copies, and then each
// lane walks one pixel's slots, newest first by insertion (slot h - 1, h - 2,
// ... cyclically, h the head). Consecutive entries are the consecutive samples
// that the temporal gradient compares when times do not increase along the
// walk, the usual case; a queue out of time order is sorted (by time, newest
// first; equal times newest first by insertion), up to 16 entries by insertion on
// slot numbers in shared memory, more by a network in registers. Sequence numbers
// are not read: they fall along the walk.
//
// Every sum over a queue adds entry k to partial k mod L and the L partials in
// a tree, L = 2, 4 or 8 with the depth: short chains, and one order of rounding
// whatever the number of threads a pixel gets.
//
// Bound: HBM (20 bytes a slot in FP32 colours, 36 a pixel: 5.4 TB/s). A group of
// lanes a pixel spent the time on shuffles and read the sequence numbers too:
// 1920x1080x16 227 us, this one 135 us (with a runtime depth, weights kept in
// shared memory: 156 us; CTAs of two and four warps 135-164 us); 640x480x8 in
// FP16 32 -> 18 us. Depths 4, 8 and 16 have a kernel of their own, where every
// slot is at a constant offset and weights and deviations stay in registers.
//
// Shared memory of a warp: times (ts words a pixel), colours (cb bytes a
// pixel), slot order (b bytes a pixel) and, where b is not a compile-time
// constant, the weights (ts words a pixel; else they stay in registers).
// Strides are odd multiples of the access size where the copies allow it, so
// that lanes at one slot do not conflict.
constexpr int kPixelWarps = 1;

struct PixelLayout {
    int ts;       // words a pixel of the time and weight areas
    int cb;       // bytes a pixel of the colour area
    int bytes;    // of one warp
};

__host__ __device__ constexpr PixelLayout pixel_layout(int b, int csize, bool weights) {
    PixelLayout l{};
    l.ts = (b & 3) == 0 && ((b >> 2) & 1) == 0 ? b + 4 : b;   // 16-byte copies never cross a padded pixel
    l.cb = (b & 1) == 0 ? csize * b + 16 : csize * b;
    l.bytes = (32 * ((weights ? 8 : 4) * l.ts + l.cb + b) + 15) & ~15;
    return l;
}

__device__ __forceinline__ void copy16(uint32_t dst, const void *src, int bytes) {   // bytes < 16: the rest is zero
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Copies n bytes of 32 pixels' records from src (16-byte aligned) to dst,
// padding each pixel from `from` to `to` bytes (equal: one linear copy).
__device__ __forceinline__ void stage(char *dst, const char *src, int n, int from, int to) {
    const int lane = threadIdx.x & 31;
    const uint32_t d0 = (uint32_t)__cvta_generic_to_shared(dst);
    if (from == to) {
        for (int i = 16 * lane; i < n; i += 512) copy16(d0 + i, src + i, min(16, n - i));
        return;
    }
    const int per = from >> 4, dp = 32 / per, dr = 32 - dp * per;   // chunks a pixel; a step of 32 chunks in (pixels, chunks)
    int p = lane / per, r = lane - p * per;
    for (int i = 16 * lane; i < n; i += 512) {
        copy16(d0 + p * to + 16 * r, src + i, min(16, n - i));
        p += dp;
        r += dr;
        if (r >= per) {
            r -= per;
            ++p;
        }
    }
}

__device__ __forceinline__ float lum_diff(float3 a, float3 b) {   // L(a) - L(b) from the colour differences
    return fmaf(kLumB, __fsub_rn(a.z, b.z), fmaf(kLumG, __fsub_rn(a.y, b.y), kLumR * __fsub_rn(a.x, b.x)));
}

// Luminance differences carry the gradients: the spatial gradient is a
// difference of neighbouring pixel means and the temporal one a difference
// of consecutive luminances, both far smaller than the luminances. So each
// pixel takes the luminance of its newest sample, in double-float, as its
// reference L_r, and every sample its deviation d = L - L_r in FP32 from the
// colour differences (exact when the colours are within a factor 2, else
// rounded once), whose error scales with the pixel's spread of luminance,
// not its level. The mean is L_r + sum(w d) / sum(w), kept as (hi, lo); the
// temporal gradient takes each consecutive pair's difference from its colour
// differences; the age weights, the time steps and the variance moments are
// FP32.
// Sum of L partials: halves added pairwise.
template <int L>
__device__ __forceinline__ float tree_sum(float (&v)[L]) {
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < o; ++k) v[k] += v[k + o];
    return v[0];
}

// The slots of a queue of n entries (the newest in slot `first`, depth b <= N) by
// time, newest first, equal times newest first by insertion, to order[]. A
// bitonic network over keys in registers: a deep queue's insertion sort is a long
// chain of dependent loads, and the lanes' lengths differ. The gradient passes at
// 1280x720, 32 deep, times in random order: 409 us, by insertion 1084 (falling
// times 409 and 1255; in order 236); 24 deep 299 and 519.
template <int N>
__device__ __forceinline__ void sort_network(const float *ts, uint8_t *order, int b, int first, int n) {
    unsigned long long key[N];   // ascending: falling time, then the place in the queue
#pragma unroll
    for (int k = 0; k < N; ++k) {
        int s = first - k;
        if (s < 0) s += b;
        const uint32_t bits = k < n ? __float_as_uint(ts[s] + 0.f) : 0u;   // + 0: one zero
        const uint32_t up = bits ^ ((uint32_t)((int)bits >> 31) | 0x80000000u);   // order of the floats
        key[k] = k < n ? ((unsigned long long)~up << 32) | (uint32_t)k : ~0ull;
    }
#pragma unroll
    for (int k = 2; k <= N; k *= 2)
#pragma unroll
        for (int j = k / 2; j > 0; j /= 2)
#pragma unroll
            for (int i = 0; i < N; ++i)
                if ((i ^ j) > i) {
                    const bool swap = (key[i] > key[i ^ j]) == ((i & k) == 0);
                    const unsigned long long x = key[i], y = key[i ^ j];
                    key[i] = swap ? y : x;
                    key[i ^ j] = swap ? x : y;
                }
#pragma unroll
    for (int k = 0; k < N; ++k) {
        int s = first - (int)(uint32_t)key[k];
        if (s < 0) s += b;
        if (k < n) order[k] = (uint8_t)s;
    }
}

// Partials of a sum over a queue of depth b.
__host__ __device__ constexpr int partials(int b) { return b <= 8 ? 2 : b <= 16 ? 4 : 8; }

// B: the depth, or 0 for a depth known at run time; L: partials(depth).
template <int CT, int B, int L>
__global__ void __launch_bounds__(32 * kPixelWarps) k_pixel(int P, int b_run, float t_now,
                                                            const uint32_t *__restrict__ state,
                                                            const float *__restrict__ r_t,
                                                            const void *__restrict__ r_col, float2 *__restrict__ lbar,
                                                            float4 *__restrict__ pstat,
                                                            unsigned long long *__restrict__ total) {
    using CS = ColorStore<CT>;
    using T4 = typename CS::T;
    extern __shared__ __align__(16) char smem[];
    const int b = B ? B : b_run;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const PixelLayout l = pixel_layout(b, (int)sizeof(T4), B == 0);
    if (blockIdx.x == 0 && threadIdx.x == 0) *total = 0ull;   // the tile pass counts the samples
    const int p0 = (blockIdx.x * kPixelWarps + warp) * 32, np = min(32, P - p0);
    if (np <= 0) return;
    char *base = smem + warp * l.bytes;
    float *ts = reinterpret_cast<float *>(base);
    char *cs = base + 128 * l.ts;
    uint8_t *order = reinterpret_cast<uint8_t *>(cs + 32 * l.cb);
    float *ws = reinterpret_cast<float *>(base + l.bytes - (B ? 0 : 128 * l.ts));
    const char *src_t = reinterpret_cast<const char *>(r_t + (size_t)p0 * b),
               *src_c = reinterpret_cast<const char *>(reinterpret_cast<const T4 *>(r_col) + (size_t)p0 * b);
    if (B && np == 32) {   // whole: constant trip counts, no ends to check
        stage(base, src_t, 128 * B, 4 * B, 4 * l.ts);
        stage(cs, src_c, 32 * (int)sizeof(T4) * B, (int)sizeof(T4) * B, l.cb);
    } else {
        stage(base, src_t, 4 * np * b, 4 * b, 4 * l.ts);
        stage(cs, src_c, (int)sizeof(T4) * np * b, (int)sizeof(T4) * b, l.cb);
    }
    const int p = p0 + lane;
    const uint32_t st = lane < np ? __ldg(state + p) : 0u;
    const int n = (int)(st & 0xFFFFu), h = (int)(st >> 16);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    ts += lane * l.ts;
    ws += lane * l.ts;
    const T4 *col = reinterpret_cast<const T4 *>(cs + lane * l.cb);
    order += lane * b;
    const int first = h == 0 ? b - 1 : h - 1;   // newest slot
    const float3 cr = CS::widen(col[first]);
    float sw[L] = {}, swd[L] = {}, num[L] = {}, den[L] = {}, m2[L] = {}, age = 0.f, Tp = 0.f, wp = 0.f;
    float3 cp = cr;
    bool ordered = true;   // times do not increase along the walk
    float W[B ? B : 1], D[B ? B : 1];
#pragma unroll(B ? B / L : 1)
    for (int k0 = 0; k0 < b; k0 += L) {
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const int k = k0 + j;
            if (!B && k >= b) break;
            int s = h - 1 - k;
            if (s < 0) s += b;
            const float T = ts[s], a = fmaxf(t_now - T, 0.f), w = expf(-kAgeDecay * a);
            const float3 c = CS::widen(col[s]);
            const float d = lum_diff(c, cr), dl = fabsf(lum_diff(cp, c));
            if (B) {
                W[B ? k : 0] = w;
                D[B ? k : 0] = d;
            } else {
                ws[s] = w;
            }
            if (k < n) {
                sw[j] += w;
                swd[j] += w * d;
                age += a;
                if (k > 0) {   // entry k - 1 and the next older one
                    num[(j + L - 1) % L] += wp * dl;
                    den[(j + L - 1) % L] += wp * (Tp - T);
                    ordered = ordered && Tp >= T;
                }
            }
            Tp = T;
            wp = w;
            cp = c;
        }
    }
    if (!ordered) {
        if (L == 8) {
            sort_network<32>(ts, order, b, first, n);
        } else {
            int s = first;
            for (int k = 0; k < n; ++k) {
                const float T = ts[s];
                int j = k;
                while (j > 0 && ts[order[j - 1]] < T) {
                    order[j] = order[j - 1];
                    --j;
                }
                order[j] = (uint8_t)s;
                s = s == 0 ? b - 1 : s - 1;
            }
        }
#pragma unroll
        for (int j = 0; j < L; ++j) num[j] = den[j] = 0.f;
        float T = ts[order[0]];
        float3 c = CS::widen(col[order[0]]);
        for (int k0 = 0; k0 + 1 < n; k0 += L) {
#pragma unroll
            for (int j = 0; j < L; ++j) {
                if (k0 + j + 1 >= n) break;
                const int o = order[k0 + j + 1];
                const float To = ts[o], w = expf(-kAgeDecay * fmaxf(t_now - T, 0.f));
                const float3 co = CS::widen(col[o]);
                num[j] += w * fabsf(lum_diff(c, co));
                den[j] += w * (T - To);
                T = To;
                c = co;
            }
        }
    }
    const float tw = tree_sum(sw), delta = n > 0 ? tree_sum(swd) / tw : 0.f;   // mean - L_r
#pragma unroll(B ? B / L : 1)
    for (int k0 = 0; k0 < b; k0 += L) {
#pragma unroll
        for (int j = 0; j < L; ++j) {
            const int k = k0 + j;
            if (!B && k >= b) break;
            int s = h - 1 - k;
            if (s < 0) s += b;
            const float w = B ? W[B ? k : 0] : ws[s], dd = (B ? D[B ? k : 0] : lum_diff(CS::widen(col[s]), cr)) - delta;
            if (k < n) m2[j] += w * dd * dd;
        }
    }
    if (lane >= np) return;
    if (n == 0) {
        lbar[p] = make_float2(__int_as_float(0x7fc00000), 0.f);
        pstat[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        const dfloat mean = df_add(luminance_df(cr), {delta, 0.f});
        lbar[p] = make_float2(mean.h, mean.l);
        const float tn = tree_sum(num), td = tree_sum(den);
        pstat[p] = make_float4(tw, tree_sum(m2), (n >= 2 && td > 0.f) ? tn / td : 0.f, age);
    }
}

// ---- tile pass -------------------------------------------------------------------
// One block per statistics tile, a warp per row: G_x, G_y of each pixel from
// its neighbours' means (written to the gradient map) and the tile record:
// sample count, non-empty pixels, sums of gradients and ages, and the
// age-weighted luminance moments. The weights, the weighted means and then the
// weighted squares about the tile's mean are summed as double-floats, so the
// moments need no division per pixel and lose nothing in tiles of any size.
// Bound: the latency of a block's loads and sums. Merging per-pixel moments with
// Chan's formula, two divisions a merge, with FP64 merges of large tiles by one
// thread, took 63 us at 1920x1080, 20 us at 640x480 and 9.6 us at 128x128; this
// takes 28.6, 7.3 and 4.1 us (two and four blocks a SM: 30 us).
constexpr int kTileThreads = 256;
constexpr int kTileWarps = kTileThreads / 32;

// a + x for a running double-float sum: exact but for the rounding of the low part
__device__ __forceinline__ dfloat df_more(dfloat a, float x) {
    const dfloat s = two_sum(a.h, x);
    return {s.h, __fadd_rn(a.l, s.l)};
}

// Sum over the `width` lanes (a power of two) of each group of lanes.
template <int WIDTH>
__device__ __forceinline__ dfloat lanes_sum(dfloat v) {
#pragma unroll
    for (int o = WIDTH / 2; o > 0; o >>= 1)
        v = df_add(v, dfloat{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
    return v;
}

template <int WIDTH, typename T>
__device__ __forceinline__ T lanes_sum(T v) {
#pragma unroll
    for (int o = WIDTH / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The weights of samples 25 time units old and more are below the least normal
// number, and their products with the means would keep a few bits only. A power
// of two changes no other bit of the sums.
constexpr float kWeightScale = 4294967296.f;   // 2^32

// What one pixel adds to its tile.
struct PixelRead {
    float2 c, l, r, u, d;   // means of the pixel and its neighbours (itself past the border)
    float4 ps;
    uint32_t cnt;
};

__device__ __forceinline__ PixelRead read_pixel(int x, int y, int W, int H, const float2 *__restrict__ lbar,
                                                const float4 *__restrict__ pstat, const uint32_t *__restrict__ state) {
    const int p = y * W + x;
    PixelRead v;
    v.c = __ldg(lbar + p);
    v.l = __ldg(lbar + (x > 0 ? p - 1 : p));
    v.r = __ldg(lbar + (x + 1 < W ? p + 1 : p));
    v.u = __ldg(lbar + (y > 0 ? p - W : p));
    v.d = __ldg(lbar + (y + 1 < H ? p + W : p));
    v.ps = __ldg(pstat + p);
    v.cnt = __ldg(state + p) & 0xFFFFu;
    return v;
}

struct TileSums {
    uint32_t n = 0, ne = 0;
    float gx = 0.f, gy = 0.f, gt = 0.f;
    dfloat sw{0.f, 0.f}, swm{0.f, 0.f}, age{0.f, 0.f};
};

__device__ __forceinline__ void add_pixel(const PixelRead &v, int x, int y, int W, int H, float4 *__restrict__ grad,
                                          TileSums &t) {
    const int p = y * W + x;
    t.age = df_more(t.age, v.ps.w);   // of every buffered sample, too old for any weight or not
    if (isnan(v.c.x)) {
        grad[p] = make_float4(0.f, 0.f, 0.f, v.c.x);
        return;
    }
    // one-sided differences of the double-float means, rounded once
    const dfloat m{v.c.x, v.c.y};
    float sx = 0.f, sy = 0.f;
    int mx = 0, my = 0;
    if (x > 0 && !isnan(v.l.x)) { sx += fabsf(df_diff(m, {v.l.x, v.l.y})); ++mx; }
    if (x + 1 < W && !isnan(v.r.x)) { sx += fabsf(df_diff(m, {v.r.x, v.r.y})); ++mx; }
    if (y > 0 && !isnan(v.u.x)) { sy += fabsf(df_diff(m, {v.u.x, v.u.y})); ++my; }
    if (y + 1 < H && !isnan(v.d.x)) { sy += fabsf(df_diff(m, {v.d.x, v.d.y})); ++my; }
    const float gx = mx == 2 ? 0.5f * sx : sx, gy = my == 2 ? 0.5f * sy : sy;
    grad[p] = make_float4(gx, gy, v.ps.z, v.c.x);
    t.n += v.cnt;
    ++t.ne;
    t.gx += gx;
    t.gy += gy;
    t.gt += v.ps.z;
    const float w = v.ps.x * kWeightScale;
    t.sw = df_more(t.sw, w);
    const dfloat q = two_prod(w, v.c.x);
    t.swm = df_more(t.swm, q.h);
    t.swm.l += q.l;
}

// Tiles of up to 16 x 16 pixels: a warp a tile, PER pixels a lane, nothing shared
// but the count of a block's samples. A block a tile left most of its threads
// without a pixel: 1920x1080, 2 deep, both gradient passes, tiles of 1, 4, 8 and 16
// pixels a side 15965, 1077, 326 and 129 us; so 2249, 195, 103 and 89 (17 a side, a
// block a tile: 126).
template <int PER>
__global__ void __launch_bounds__(kTileThreads, 3) k_warp_tiles(int W, int H, int S, int ntx, int ntiles,
                                                             const float2 *__restrict__ lbar,
                                                             const float4 *__restrict__ pstat,
                                                             const uint32_t *__restrict__ state,
                                                             float4 *__restrict__ grad, TilePartial *__restrict__ tiles,
                                                             unsigned long long *__restrict__ total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tile = blockIdx.x * kTileWarps + warp;
    TileSums t;
    if (tile < ntiles) {   // warp-uniform
        const int x0 = (tile % ntx) * S, y0 = (tile / ntx) * S;
        const int tw = min(S, W - x0), A = tw * min(S, H - y0);
        float c[PER], w[PER], m[PER];   // mean, weight and spread of each pixel
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int k = min(32 * r + lane, A - 1), row = k / tw, x = x0 + k - row * tw, y = y0 + row;
            const PixelRead v = read_pixel(x, y, W, H, lbar, pstat, state);
            const bool in = 32 * r + lane < A;
            if (in) add_pixel(v, x, y, W, H, grad, t);
            c[r] = in ? v.c.x : __int_as_float(0x7fc00000);
            w[r] = v.ps.x;
            m[r] = v.ps.y;
        }
        t.n = __reduce_add_sync(0xffffffffu, t.n);
        t.ne = __reduce_add_sync(0xffffffffu, t.ne);
        const dfloat sw = lanes_sum<32>(t.sw), swm = lanes_sum<32>(t.swm), age = lanes_sum<32>(t.age);
        const dfloat mean = sw.h > 0.f ? df_div(swm, sw) : dfloat{0.f, 0.f};
        dfloat m2{0.f, 0.f};   // squares about the tile's mean
#pragma unroll
        for (int r = 0; r < PER; ++r)
            if (!isnan(c[r])) m2 = df_more(m2, fmaf(w[r] * (c[r] - mean.h), c[r] - mean.h, m[r]));
        m2 = lanes_sum<32>(m2);
        TilePartial out;
        out.sw = ((double)sw.h + (double)sw.l) / kWeightScale;
        out.mean = (double)mean.h + (double)mean.l;
        out.m2 = (double)m2.h + (double)m2.l;
        out.sgx = lanes_sum<32>(t.gx);
        out.sgy = lanes_sum<32>(t.gy);
        out.sgt = lanes_sum<32>(t.gt);
        out.n = t.n;
        out.nonempty = t.ne;
        out.age = __fadd_rn(age.h, age.l);
        out.pad[0] = out.pad[1] = 0u;
        if (lane == 0) tiles[tile] = out;
    }
    __shared__ uint32_t count[kTileWarps];
    if (lane == 0) count[warp] = t.n;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t n = 0;
        for (int k = 0; k < kTileWarps; ++k) n += count[k];
        if (n) atomicAdd(total, (unsigned long long)n);
    }
}

// SMALL: tiles of up to 32 x 32 pixels, four rows a warp: every load of a
// thread is issued before the first is used, and the second pass reads
// registers.
template <bool SMALL>
__global__ void __launch_bounds__(kTileThreads, 3) k_spatial_tiles(int W, int H, int S, int ntx,
                                                                const float2 *__restrict__ lbar,
                                                                const float4 *__restrict__ pstat,
                                                                const uint32_t *__restrict__ state,
                                                                float4 *__restrict__ grad,
                                                                TilePartial *__restrict__ tiles,
                                                                unsigned long long *__restrict__ total) {
    const int tile = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = (tile % ntx) * S, y0 = (tile / ntx) * S;
    const int x1 = min(W, x0 + S), y1 = min(H, y0 + S);
    constexpr int ROWS = SMALL ? 4 : 1;
    PixelRead v[ROWS];
    TileSums t;
    if (SMALL) {
        const int x = min(x0 + lane, x1 - 1);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) v[r] = read_pixel(x, min(y0 + warp + r * kTileWarps, y1 - 1), W, H, lbar, pstat, state);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int y = y0 + warp + r * kTileWarps;
            if (x0 + lane < x1 && y < y1) add_pixel(v[r], x, y, W, H, grad, t);
            else v[r].c.x = __int_as_float(0x7fc00000);   // no pixel
        }
    } else {
        for (int x = x0 + lane; x < x1; x += 32)
            for (int y = y0 + warp; y < y1; y += kTileWarps)
                add_pixel(read_pixel(x, y, W, H, lbar, pstat, state), x, y, W, H, grad, t);
    }
    __shared__ float2 shd[3][kTileWarps];
    __shared__ float shf[3][kTileWarps];
    __shared__ uint32_t shi[2][kTileWarps];
    __shared__ float tile_mean;
    t.n = __reduce_add_sync(0xffffffffu, t.n);
    t.ne = __reduce_add_sync(0xffffffffu, t.ne);
    t.gx = lanes_sum<32>(t.gx);
    t.gy = lanes_sum<32>(t.gy);
    t.gt = lanes_sum<32>(t.gt);
    t.sw = lanes_sum<32>(t.sw);
    t.swm = lanes_sum<32>(t.swm);
    t.age = lanes_sum<32>(t.age);
    if (lane == 0) {
        shi[0][warp] = t.n; shi[1][warp] = t.ne;
        shf[0][warp] = t.gx; shf[1][warp] = t.gy; shf[2][warp] = t.gt;
        shd[0][warp] = make_float2(t.sw.h, t.sw.l);
        shd[1][warp] = make_float2(t.swm.h, t.swm.l);
        shd[2][warp] = make_float2(t.age.h, t.age.l);
    }
    __syncthreads();
    TilePartial out;
    if (warp == 0) {   // eight lanes a quantity
        static_assert(kTileWarps == 8, "eight partials a quantity");
        const int q = min(lane >> 3, 2), w = lane & 7;
        const dfloat d = lanes_sum<8>(dfloat{shd[q][w].x, shd[q][w].y});
        const float f = lanes_sum<8>(shf[q][w]);
        const uint32_t i = lanes_sum<8>(shi[min(q, 1)][w]);
        auto take = [&](int k) { return dfloat{__shfl_sync(0xffffffffu, d.h, 8 * k), __shfl_sync(0xffffffffu, d.l, 8 * k)}; };
        const dfloat tw = take(0), tm = take(1), ta = take(2);
        const dfloat mean = tw.h > 0.f ? df_div(tm, tw) : dfloat{0.f, 0.f};
        out.sw = ((double)tw.h + (double)tw.l) / kWeightScale;
        out.mean = (double)mean.h + (double)mean.l;
        out.n = __shfl_sync(0xffffffffu, i, 0);
        out.nonempty = __shfl_sync(0xffffffffu, i, 8);
        out.sgx = __shfl_sync(0xffffffffu, f, 0);
        out.sgy = __shfl_sync(0xffffffffu, f, 8);
        out.sgt = __shfl_sync(0xffffffffu, f, 16);
        out.age = __fadd_rn(ta.h, ta.l);
        out.pad[0] = out.pad[1] = 0u;
        if (lane == 0) {
            tile_mean = mean.h;
            if (out.n) atomicAdd(total, (unsigned long long)out.n);
        }
    }
    __syncthreads();
    // squares about the tile's mean
    const float tm = tile_mean;
    dfloat m2{0.f, 0.f};
    auto square = [&](float c, float sw, float m) {
        if (!isnan(c)) m2 = df_more(m2, fmaf(sw * (c - tm), c - tm, m));
    };
    if (SMALL) {
#pragma unroll
        for (int r = 0; r < ROWS; ++r) square(v[r].c.x, v[r].ps.x, v[r].ps.y);
    } else {
        for (int x = x0 + lane; x < x1; x += 32)
            for (int y = y0 + warp; y < y1; y += kTileWarps) {
                const int p = y * W + x;
                const float2 ps = __ldg(reinterpret_cast<const float2 *>(pstat + p));
                square(__ldg(&lbar[p].x), ps.x, ps.y);
            }
    }
    m2 = lanes_sum<32>(m2);
    if (lane == 0) shd[0][warp] = make_float2(m2.h, m2.l);
    __syncthreads();
    if (warp == 0) {
        const dfloat d = lanes_sum<8>(dfloat{shd[0][lane & 7].x, shd[0][lane & 7].y});
        out.m2 = (double)d.h + (double)d.l;
        if (lane == 0) tiles[tile] = out;
    }
}

template <int CT, int B, int L>
void launch_depth(AfrContext *c, float t_now, unsigned long long *total, cudaStream_t s) {
    static_assert(B == 0 || L == partials(B), "one order of summation a depth");
    const PixelLayout l = pixel_layout(c->b, c->csize, B == 0);
    const int groups = (c->P + 31) / 32;
    k_pixel<CT, B, L><<<(groups + kPixelWarps - 1) / kPixelWarps, 32 * kPixelWarps, kPixelWarps * l.bytes, s>>>(
        c->P, c->b, t_now, c->r_state, c->r_t, c->r_col, c->lbar, c->pstat, total);
}

template <int CT>
void launch_pixel(AfrContext *c, float t_now, unsigned long long *total, cudaStream_t s) {
    switch (c->b) {
        case 4: launch_depth<CT, 4, 2>(c, t_now, total, s); break;
        case 8: launch_depth<CT, 8, 2>(c, t_now, total, s); break;
        case 16: launch_depth<CT, 16, 4>(c, t_now, total, s); break;
        default:
            if (partials(c->b) == 2) launch_depth<CT, 0, 2>(c, t_now, total, s);
            else if (partials(c->b) == 4) launch_depth<CT, 0, 4>(c, t_now, total, s);
            else launch_depth<CT, 0, 8>(c, t_now, total, s);
            break;
    }
}

}  // namespace

cudaError_t launch_gradients(AfrContext *c, float t_now, cudaStream_t s) {
    unsigned long long *total = tile_total(c);
    switch (c->ct) {
        case AFR_F32: launch_pixel<AFR_F32>(c, t_now, total, s); break;
        case AFR_F16: launch_pixel<AFR_F16>(c, t_now, total, s); break;
        default: launch_pixel<AFR_BF16>(c, t_now, total, s); break;
    }
    const int warps = (c->ntiles + kTileWarps - 1) / kTileWarps;
    if (c->S <= 8)
        k_warp_tiles<2><<<warps, kTileThreads, 0, s>>>(c->W, c->H, c->S, c->ntx, c->ntiles, c->lbar, c->pstat, c->r_state,
                                                       c->grad, c->tiles, total);
    else if (c->S <= 16)
        k_warp_tiles<8><<<warps, kTileThreads, 0, s>>>(c->W, c->H, c->S, c->ntx, c->ntiles, c->lbar, c->pstat, c->r_state,
                                                       c->grad, c->tiles, total);
    else if (c->S <= 32)
        k_spatial_tiles<true><<<c->ntiles, kTileThreads, 0, s>>>(c->W, c->H, c->S, c->ntx, c->lbar, c->pstat,
                                                                 c->r_state, c->grad, c->tiles, total);
    else
        k_spatial_tiles<false><<<c->ntiles, kTileThreads, 0, s>>>(c->W, c->H, c->S, c->ntx, c->lbar, c->pstat,
                                                                  c->r_state, c->grad, c->tiles, total);
    return cudaGetLastError();
}

}  // namespace afr
