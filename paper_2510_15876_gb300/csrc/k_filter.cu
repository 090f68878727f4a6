// k_filter.cu -- sections 5.1 and 5.2: filter widths from density and
// gradients, the normalised space-time Gaussian gather over each pixel's
// integer disc of frame bins, and its adjoint.
//
// Exponent shift. Every weight is 2^-E with E = d^2 ks + a^2 kt >= 0
// (ks = log2 e / (2 sigma_s^2), kt = log2 e / (2 sigma_t^2)). A pixel whose
// samples are all old under a narrow temporal filter has every E far above
// the FP32 range, so the kernel subtracts a per-pixel shift m: the minimum
// over the footprint's bins of a lower bound of E in that bin (the bin's
// nearest point to the pixel centre and its smallest a^2). Then E - m >= 0
// for every sample and E - m <= ((R+1)^2 - R^2 + ...) ks stays small for
// the sample that attains the bound, so the normalised colour is exact up to
// rounding whatever the ages; W is reported as S * 2^-m.
#include <type_traits>

#include "afr_internal.cuh"

namespace afr {
namespace {

struct Widths {
    float es, et, raw_s, raw_t, ss, st;
};

__device__ __forceinline__ Widths widths(float4 g, float V, float eps, const AfrParams &prm) {
    Widths w;
    float Gs = fmaxf(0.5f * (g.x + g.y), eps);
    float Gt = fmaxf(g.z, eps);
    w.es = cbrtf(V * Gt / Gs);
    w.et = cbrtf(V * (Gs * Gs) / (Gt * Gt));
    w.raw_s = fmaf(prm.alpha_s, w.es, prm.beta_s);
    w.raw_t = fmaf(prm.alpha_t, w.et, prm.beta_t);
    w.ss = fminf(fmaxf(w.raw_s, kSigmaSMin), prm.clamp_s);
    w.st = fminf(fmaxf(w.raw_t, kSigmaTMin), prm.clamp_t);
    return w;
}

__device__ __forceinline__ float tile_volume(int x, int y, int W, int H, int S, int ntx, float window,
                                             const TilePartial *__restrict__ tiles) {
    int tx = x / S, ty = y / S;
    float A = (float)(min(S, W - tx * S) * min(S, H - ty * S));
    float n = (float)__ldg(&tiles[ty * ntx + tx].n);   // an integer count
    return n > 0.f ? A * window / n : A * window;
}

// floor(sqrt(R^2 - dy^2)), |dy| <= R <= 8: the radicand is an integer, so half
// a unit added before the root keeps the approximation's error away from the
// integers.
__device__ __forceinline__ int half_width(int R, int dy) {
    float h;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(h) : "f"((float)(R * R - dy * dy) + 0.5f));
    return (int)h;
}

__device__ __forceinline__ float bin_gap(int d) {   // nearest distance from a pixel centre to a bin d away
    float g = fabsf((float)d) - 0.5f;
    return g > 0.f ? g : 0.f;
}

struct PixelFrame {
    float cx, cy, ks, kt, m;
    bool any;
};

// Per-pixel constants of the gather: centre, exponent scales and shift.
__device__ __forceinline__ PixelFrame pixel_frame(int x, int y, int W, int H, int R, float2 sg,
                                                  const uint32_t *__restrict__ amin2) {
    PixelFrame f;
    f.cx = (float)x + 0.5f;
    f.cy = (float)y + 0.5f;
    f.ks = kLog2e / (2.f * sg.x * sg.x);
    f.kt = kLog2e / (2.f * sg.y * sg.y);
    float m = INFINITY;
    for (int dy = -R; dy <= R; ++dy) {
        int row = y + dy;
        if (row < 0 || row >= H) continue;
        int hw = half_width(R, dy);
        int x0 = max(0, x - hw), x1 = min(W - 1, x + hw);
        float gy = bin_gap(dy);
        for (int bx = x0; bx <= x1; ++bx) {
            uint32_t a2 = __ldg(amin2 + (size_t)row * W + bx);
            if (a2 == 0x7f800000u) continue;   // empty bin
            float gx = bin_gap(bx - x);
            float lb = fmaf(fmaf(gx, gx, gy * gy), f.ks, __uint_as_float(a2) * f.kt);
            m = fminf(m, lb);
        }
    }
    f.any = m < INFINITY;
    f.m = f.any ? m : 0.f;
    return f;
}

// Filter widths of every pixel (unless KEEP: the widths already in the map
// are used) and the pixel's gather constants for the filter: -ks, -kt, the
// exponent shift m and the footprint radius.
//
// A block takes 32 x 8 pixels and keeps the smallest ages of their bins and the
// halo in shared memory. Bins at the same |dx| and |dy| from a pixel have the
// same distance term, and the bound grows with the age, so their ages are
// compared as integers first and the bound is evaluated once for each pair of
// offsets (15 instead of 49 at R = 4): the same minimum, bit for bit. RT: R at
// compile time (every load at a constant offset), or -1. Bound: issue. A
// thread a pixel with 49 global loads and bounds took 89 us at 1920x1080 (R 4)
// and 58 us at 1280x720 (R 5); this takes 34 and 20 us.
constexpr int kSigX = 32, kSigY = 8, kSigHalo = 8;
constexpr uint32_t kEmptyBin = 0x7f800000u;

template <bool KEEP, int RT>
__global__ void __launch_bounds__(kSigX * kSigY) k_sigma(int W, int H, int Rrun, int S, int ntx, float window, float eps,
                                                         AfrParams prm, const float4 *__restrict__ grad,
                                                         const TilePartial *__restrict__ tiles,
                                                         const uint32_t *__restrict__ amin2,
                                                         float2 *__restrict__ sigma, float4 *__restrict__ fconst) {
    grid_order();
    __shared__ uint32_t age[(kSigY + 2 * kSigHalo) * (kSigX + 2 * kSigHalo)];
    const int R = RT >= 0 ? RT : Rrun, pitch = kSigX + 2 * R;
    const int x0 = blockIdx.x * kSigX, y0 = blockIdx.y * kSigY, x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    for (int r = threadIdx.y; r < kSigY + 2 * R; r += kSigY) {
        const int row = y0 - R + r;
        for (int c = threadIdx.x; c < pitch; c += kSigX) {
            const int col = x0 - R + c;
            age[r * pitch + c] = row >= 0 && row < H && col >= 0 && col < W ? __ldg(amin2 + (size_t)row * W + col) : kEmptyBin;
        }
    }
    const bool in = x < W && y < H;
    const size_t p = (size_t)min(y, H - 1) * W + min(x, W - 1);
    float2 sg;
    if (KEEP) {
        sg = sigma[p];
    } else {
        const Widths w = widths(__ldg(grad + p), tile_volume(min(x, W - 1), min(y, H - 1), W, H, S, ntx, window, tiles), eps, prm);
        sg = make_float2(w.ss, w.st);
        if (in) sigma[p] = sg;
    }
    __syncthreads();
    if (!in) return;
    const float ks = kLog2e / (2.f * sg.x * sg.x), kt = kLog2e / (2.f * sg.y * sg.y);
    const uint32_t *own = age + (threadIdx.y + R) * pitch + threadIdx.x + R;
    float m = INFINITY;
#pragma unroll
    for (int v = 0; v <= R; ++v) {
        const float gy = bin_gap(v);
#pragma unroll
        for (int u = 0; u <= R; ++u) {
            if (u * u + v * v > R * R) continue;
            uint32_t a = min(own[v * pitch + u], own[v * pitch - u]);
            if (v) a = min(a, min(own[-v * pitch + u], own[-v * pitch - u]));
            const float gx = bin_gap(u);
            if (a != kEmptyBin) m = fminf(m, fmaf(fmaf(gx, gx, gy * gy), ks, __uint_as_float(a) * kt));
        }
    }
    fconst[p] = make_float4(-ks, -kt, m < INFINITY ? m : 0.f, __int_as_float(R));
}

// Section 6.2 in gather form: the next footprint radius of each pixel is the
// mean of the previous radii over its 3x3 neighbourhood (clipped at the
// border), times 4 below 4 samples, times 0.7 above 32 (no count: times 1),
// clamped; single precision with one rounding per operation, in the same
// order as a plain loop over the neighbourhood rows.
__device__ __forceinline__ float next_radius(int x, int y, int W, int H, const float *__restrict__ r_prev, int32_t n,
                                             float r_min, float r_max) {
    float sum = 0.f;
    int cnt = 0;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
            const int qx = x + dx, qy = y + dy;
            if (qx < 0 || qy < 0 || qx >= W || qy >= H) continue;
            sum = __fadd_rn(sum, __ldg(r_prev + (size_t)qy * W + qx));
            ++cnt;
        }
    const float mean = __fdiv_rn(sum, (float)cnt);
    const float f = n < 0 ? 1.f : n < 4 ? 4.f : n > 32 ? 0.7f : 1.f;
    float r = __fmul_rn(mean, f);
    if (r < r_min) r = r_min;
    if (r > r_max) r = r_max;
    return r;
}

// k_sigma for adaptive footprints: each pixel's next radius r, the widths, the
// gather constants of the disc of radius floor(r + 1/2), and the samples in it
// for the update after this one. (As a launch of its own the radius update
// took 17 us at 1920x1080 beside 63 us for the rest; together 58 us.)
template <bool KEEP>
__global__ void __launch_bounds__(kSigX * kSigY) k_sigma_adaptive(int W, int H, int S, int ntx, float window, float eps,
                                                                  AfrParams prm, const float4 *__restrict__ grad,
                                                                  const TilePartial *__restrict__ tiles,
                                                                  const uint32_t *__restrict__ amin2,
                                                                  const float *__restrict__ r_prev,
                                                                  float *__restrict__ r_next, float r_min, float r_max,
                                                                  const uint32_t *__restrict__ foff,
                                                                  int32_t *__restrict__ cov_n, float2 *__restrict__ sigma,
                                                                  float4 *__restrict__ fconst) {
    grid_order();
    const int x = blockIdx.x * kSigX + threadIdx.x, y = blockIdx.y * kSigY + threadIdx.y;
    if (x >= W || y >= H) return;
    const size_t p = (size_t)y * W + x;
    const float r = next_radius(x, y, W, H, r_prev, cov_n[p], r_min, r_max);
    r_next[p] = r;
    const int R = (int)floorf(__fadd_rn(r, 0.5f));
    float2 sg;
    if (KEEP) {
        sg = sigma[p];
    } else {
        const Widths w = widths(__ldg(grad + p), tile_volume(x, y, W, H, S, ntx, window, tiles), eps, prm);
        sg = make_float2(w.ss, w.st);
        sigma[p] = sg;
    }
    int32_t n = 0;
    for (int dy = max(-R, -y); dy <= min(R, H - 1 - y); ++dy) {
        const int hw = half_width(R, dy);
        const uint32_t *row = foff + (size_t)(y + dy) * W;
        n += (int32_t)(__ldg(row + min(W - 1, x + hw) + 1) - __ldg(row + max(0, x - hw)));
    }
    cov_n[p] = n;
    const PixelFrame f = pixel_frame(x, y, W, H, R, sg, amin2);
    fconst[p] = make_float4(-f.ks, -f.kt, f.m, __int_as_float(R));
}

__global__ void k_coverage_init(int P, float r0, float *__restrict__ r, int32_t *__restrict__ n) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
        r[p] = r0;
        n[p] = -1;
    }
}

// Forward gather. One warp owns a 2x2 block of pixels. The union of the four
// discs is, row by row of bins, one contiguous run of columns, and the frame
// view stores the records of consecutive bins of a row contiguously; so the
// union's records are (2R + 2) contiguous index ranges. Lanes enumerate the
// rows (range and count, from the tile's bin offsets in shared memory), a warp
// scan lays them out in one flat index space, and the gather runs a flat loop
// over it: lane l takes flat indices l, l + 32, ..., following its row with a
// cursor, so loads are coalesced and every lane runs the same trip count
// whatever the bin occupancy; a record is one 256-bit load, and the next one
// is loaded while the current one is summed. Which of the four discs hold a
// record's bin depends only on the bin's place in the union box and R: a table
// (0 in the disc, -inf outside, per pixel), shared by every block, is indexed
// by the place that the record carries (row * kPitch + column, less the place
// of the box's corner). The arithmetic runs on pixel pairs (same row) with
// paired FP32 instructions. Each lane accumulates the four pixels; the warp
// reduces them at the end. The per-pixel constants (-ks, -kt, shift) come from
// k_sigma.
//
// Bound: instruction issue and L1 (one launch at 960x540x16: 59% of issue
// slots, 66% of the L1 data pipe, 1588 warp instructions a block of which 31
// iterations take 44 each; 24 of the 44 are arithmetic). Records and row
// offsets in one place each, the shared disc table and the prefetch took the
// launch at 1920x1080x16 from 1600 to 1130 us (FP32 colours), 1280x720x8 with
// R = 5 from 607 to 407 us and 640x480x8 in FP16 from 185 to 122 us. Adaptive
// footprints, 1920x1080x16 with most radii at 1: 720 us with a table per block,
// 617 us keeping a warp's table while the radius stays, 562 us with shared
// tables of the small radii (the per-warp ones took 41 KB a CTA from L1); with one
// more for a tile's largest radius above those, 640x480x32 at radius 8 takes 1366
// us instead of 1693 (a table per block: 1310). The adaptive form spills 40 to 44
// bytes at its 80 registers, the fixed one 8 to 12. The shift
// table per block (disc + shift, no addition per record) measured 1655 us, its
// shared memory taken from L1; four CTAs a SM (64 registers, spills) 1183 us;
// a prefetch two records deep 1413 us (spills); CTAs of 12 or 24 warps
// 1317-1500 us.
constexpr int kMaxRows = 2 * 8 + 2;   // union rows (and columns) for R <= 8
constexpr int kWarps = 8;
constexpr int kMaxBatch = 64;         // contexts per batched launch

typedef unsigned long long f2;   // two floats in one 64-bit register pair

__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ uint32_t warp_incl_scan_u(uint32_t v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Reduces N per-lane values (N a power of two up to 32) across the warp:
// afterwards lane l holds the total of value l / (32 / N) with its log2(N) bits
// as they are (a transposed butterfly: N - 1 exchanges, then log2(32 / N)
// among the lanes that share a value).
template <int N>
__device__ __forceinline__ float warp_reduce(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = N / 2, o = 16; n > 0; n >>= 1, o >>= 1) {
        const bool hi = lane & o;
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
            if (k >= n) break;
            const float send = hi ? v[k] : v[k + n], stay = hi ? v[k + n] : v[k];
            v[k] = stay + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 16 / N; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// Constants and accumulators of the block's pixel pairs: pair j holds pixels
// (0, j) and (1, j).
struct PairConsts {
    f2 cx;               // (cx0, cx1)
    f2 cy[2];            // (cy_j, cy_j): row centres
    f2 nks[2], nkt[2], m[2];
};
// Weights of the block's four pixels for one record. in: 0 for each pixel
// whose disc holds the record's bin, else -inf; pixel k = 2 j + column in
// component k.
struct PairWeights {
    f2 d2[2], w[2];
};

__device__ __forceinline__ PairWeights pair_weights(const PairConsts &pc, float4 in, const FrameRec &q) {
    PairWeights r;
    const f2 dx = sub2(pk(q.p.x, q.p.x), pc.cx);
    const f2 sx = mul2(dx, dx);
    const f2 y = pk(q.p.y, q.p.y), a2 = pk(q.p.z, q.p.z);
    const f2 t[2] = {pk(in.x, in.y), pk(in.z, in.w)};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const f2 dy = sub2(y, pc.cy[j]);
        r.d2[j] = fma2(dy, dy, sx);
        const f2 e = fma2(r.d2[j], pc.nks[j], fma2(a2, pc.nkt[j], add2(pc.m[j], t[j])));
        float e0, e1;
        upk(e, e0, e1);
        r.w[j] = pk(ex2(e0), ex2(e1));
    }
    return r;
}

// What the gather sums. Forward: the weights (compensated for 16-bit colour
// storage) and the weighted colours.
template <bool KAHAN>
struct ForwardSums {
    f2 S[2], C[2], r[2], g[2], b[2];
    __device__ __forceinline__ ForwardSums() {
#pragma unroll
        for (int j = 0; j < 2; ++j) S[j] = C[j] = r[j] = g[j] = b[j] = 0ull;
    }
    __device__ __forceinline__ void add(const PairConsts &pc, float4 in, const FrameRec &q) {
        const PairWeights p = pair_weights(pc, in, q);
        const f2 cr = pk(q.c.x, q.c.x), cg = pk(q.c.y, q.c.y), cb = pk(q.c.z, q.c.z);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const f2 w = p.w[j];
            if (KAHAN) {
                const f2 v = sub2(w, C[j]);
                const f2 n = add2(S[j], v);
                C[j] = sub2(sub2(n, S[j]), v);
                S[j] = n;
            } else {
                S[j] = add2(S[j], w);
            }
            r[j] = fma2(w, cr, r[j]);
            g[j] = fma2(w, cg, g[j]);
            b[j] = fma2(w, cb, b[j]);
        }
    }
};

// Discs of the union box of a 2x2 block at footprint radius R: entry
// (v, u) = bin row by - R + v, column bx - R + u.
constexpr int kTables = 4;   // adaptive footprints: radii 1 .. kTables have a table each, a tile's largest radius above them one more
constexpr int kTableRows = kTables * (kTables + 3);
__host__ __device__ constexpr int table_row(int R) { return (R - 1) * (R + 2); }   // rows of the tables before R's
static_assert(table_row(kTables + 1) == kTableRows, "2R + 2 rows each");

__device__ __forceinline__ void fill_discs(float4 *in, int R) {
    for (int i = threadIdx.x; i < (2 * R + 2) * kPitch; i += blockDim.x) {
        const int v = i / kPitch - R, u = i % kPitch - R;
        float s[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int du = u - (k & 1), dv = v - (k >> 1);
            s[k] = du * du + dv * dv <= R * R ? 0.f : -INFINITY;
        }
        in[i] = make_float4(s[0], s[1], s[2], s[3]);
    }
}

// The same for pixels whose radii differ, for the bin at place t of the box of
// radius R.
__device__ __forceinline__ float4 own_discs(int t, int R, const int (&Rk)[4]) {
    const int v = t * 57 >> 10, u = t - v * kPitch;   // t / 18 for t < 18 * 18
    float s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int du = u - R - (k & 1), dv = v - R - (k >> 1);
        s[k] = du * du + dv * dv <= Rk[k] * Rk[k] ? 0.f : -INFINITY;
    }
    return make_float4(s[0], s[1], s[2], s[3]);
}

// A value in a register that the assembler cannot compute again from
// parameters and special registers inside a loop (a shuffle is opaque to it).
__device__ __forceinline__ uint32_t keep(uint32_t v) {
    asm volatile("shfl.sync.bfly.b32 %0, %0, 0, 0x1f, 0xffffffff;" : "+r"(v));
    return v;
}
template <typename T>
__device__ __forceinline__ T *keep(T *v) {
    const unsigned long long u = reinterpret_cast<unsigned long long>(v);
    const uint32_t lo = keep((uint32_t)u), hi = keep((uint32_t)(u >> 32));
    return reinterpret_cast<T *>(((unsigned long long)hi << 32) | lo);
}

// p + i as one multiply-add
template <typename T>
__device__ __forceinline__ const T *element(const T *p, int i) {
    unsigned long long a;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(a) : "r"(i), "n"((int)sizeof(T)), "l"(p));
    return reinterpret_cast<const T *>(a);
}

__device__ __forceinline__ uint32_t smem_at(const void *p) { return keep((uint32_t)__cvta_generic_to_shared(p)); }
__device__ __forceinline__ float4 lds4(uint32_t at) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at));
    return v;
}
__device__ __forceinline__ uint2 lds2(uint32_t at) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(at));
    return v;
}

// Row cursor of one lane of the gather: at is the shared address of the row
// table's entry (flat end, record index - flat index) for the row that holds
// the lane's flat index j + lane; end and base are that entry with the lane
// taken off.
struct Cursor {
    uint32_t at;
    int end, base;
};

__device__ __forceinline__ void step(Cursor &k, int j, int lane) {   // at most one row on
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ge.s32 p, %3, %1;\n\t"
        "@p add.u32 %0, %0, 8;\n\t"
        "@p ld.shared.v2.b32 {%1, %2}, [%0];\n\t"
        "@p sub.s32 %1, %1, %4;\n\t}"
        : "+r"(k.at), "+r"(k.end), "+r"(k.base) : "r"(j), "r"(lane));
}

template <bool ONE>
__device__ __forceinline__ void advance(Cursor &k, int j, int lane) {
    do step(k, j, lane);
    while (!ONE && __any_sync(0xffffffffu, j >= k.end));
}

// What the blocks of a CTA's tile share, loaded once: the gather constants of
// its pixels, and the bin offsets of every row of the tile and its halo, so
// that a block's row ranges cost two shared loads instead of a chain of global
// ones.
constexpr int kTilePixels = 128;              // (2 tbx) x (64 / tbx)
constexpr int kTileOffsets = 1008;            // the most of (64 / tbx + 2R) x (2 tbx + 2R + 1): tbx 2, R 8
struct TileSmem {
    float4 fc[kTilePixels];
    uint32_t off[kTileOffsets];
    uint2 rows[kWarps][kMaxRows];
};

// Offsets of the bins of rows y0 - R .. y0 + th + R - 1 at columns x0 - R ..
// x0 + tw + R (clamped to the row's first and last; rows outside the image
// are empty).
__device__ __forceinline__ void load_offsets(TileSmem &t, int W, int H, int R, int x0, int y0, int tw, int th,
                                             const uint32_t *__restrict__ foff) {
    const int cols = tw + 2 * R + 1;
    for (int r = threadIdx.x >> 5; r < th + 2 * R; r += blockDim.x >> 5) {
        const int row = y0 - R + r;
        for (int c = threadIdx.x & 31; c < cols; c += 32) {
            uint32_t v = 0;
            if (row >= 0 && row < H) v = __ldg(foff + (size_t)row * W + min(max(x0 - R + c, 0), W));
            t.off[r * cols + c] = v;
        }
    }
}

// Asks L2 for the tile's records (rows x cols of offsets) while the first
// blocks set up: they come from HBM, and a block's few iterations hide little of
// that (1.5% at R 4, 5% for adaptive footprints). Nothing past the cap records
// of the frame view is asked for, whatever the offsets say.
__device__ __forceinline__ void prefetch_tile(const TileSmem &t, int cols, int rows, const FrameRec *frec, uint32_t cap) {
    for (int r = threadIdx.x >> 5; r < rows; r += blockDim.x >> 5) {
        const uint32_t end = min(t.off[r * cols + cols - 1], cap);
        for (uint32_t i = t.off[r * cols] + 4u * (threadIdx.x & 31); i < end; i += 128u)   // 128-byte lines
            asm volatile("prefetch.global.L2 [%0];" ::"l"(frec + i));
    }
}

// Pixels past the right or bottom edge repeat the edge pixel (never stored).
__device__ __forceinline__ float4 load_const(int i, int W, int H, int x0, int y0, int tw,
                                             Fresh<float4> fconst) {
    return fconst[(size_t)min(y0 + i / tw, H - 1) * W + min(x0 + i % tw, W - 1)];
}

// Sums of one 2x2 pixel block by one warp: the block (lx, ly) of the tile at
// (x0, y0), tw pixels wide, whose offsets were loaded for footprints up to Rt.
// VAR: each pixel's footprint radius is read from its gather constants
// (adaptive footprints; most neighbouring ones have settled at one radius);
// otherwise every pixel uses Rt. tables_at: shared address of the disc tables
// (VAR: of radii 1 .. kTables, then of Rt if it is larger; else of Rt alone). frec:
// the frame view from this lane's record on.
template <bool VAR, class Sums>
__device__ __forceinline__ void gather_block(int Rt, int x0, int y0, int tw, int lx, int ly, const FrameRec *frec,
                                             const TileSmem &ts, uint32_t tables_at, uint2 *rows, uint32_t rows_at,
                                             const DebugCheck &dc, Sums &A) {
    const int lane = threadIdx.x & 31;
    const int bx = x0 + 2 * lx, by = y0 + 2 * ly;
    float4 fc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) fc[k] = ts.fc[(2 * ly + (k >> 1)) * tw + 2 * lx + (k & 1)];
    int R = Rt;
    bool same = true;
    const int Rk[4] = {__float_as_int(fc[0].w), __float_as_int(fc[1].w), __float_as_int(fc[2].w), __float_as_int(fc[3].w)};
    if (VAR) {
        R = max(max(Rk[0], Rk[1]), max(Rk[2], Rk[3]));   // the block's largest footprint
        same = min(min(Rk[0], Rk[1]), min(Rk[2], Rk[3])) == R;
    }
    // union rows: lane v (< 2R + 2) takes bin row by - R + v; the union of the
    // four discs' rows is one run of columns [bx - lo, bx + 1 + hi]
    uint32_t cnt = 0, first = 0;
    if (lane < 2 * R + 2) {
        const int v = lane - R;
        int lo, hi;
        if (!VAR || same) {   // of the two pixel rows, the nearer has the wider run
            lo = hi = half_width(R, v > 0 ? v - 1 : v);
        } else {
            lo = hi = -2;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int dv = v - (k >> 1);
                if (dv >= -Rk[k] && dv <= Rk[k]) {
                    const int h = half_width(Rk[k], dv);
                    lo = max(lo, h - (k & 1));
                    hi = max(hi, h + (k & 1) - 1);
                }
            }
        }
        if (lo + hi >= -1) {
            const uint32_t *o = ts.off + (2 * ly + v + Rt) * (tw + 2 * Rt + 1) + 2 * lx + Rt;
            first = o[-lo];
            const uint32_t last = o[hi + 2];
            cnt = last - first;
            if (!AFR_CHECK(last >= first && cnt <= dc.cap, dc.derr)) cnt = 0;
        }
    }
    const uint32_t incl = warp_incl_scan_u(cnt);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (lane < 2 * R + 2) rows[lane] = make_uint2(lane == 2 * R + 1 ? 0x7fffffffu : incl, first - (incl - cnt));
    // rows of 32 records or more between the first and the last: an iteration moves a lane at most one row on
    const bool one = __all_sync(0xffffffffu, cnt >= 32u || lane == 0 || lane >= 2 * R + 1);
    __syncwarp();
    PairConsts pc;
    pc.cx = pk((float)bx + 0.5f, (float)bx + 1.5f);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float cy = (float)(by + j) + 0.5f;
        pc.cy[j] = pk(cy, cy);
        pc.nks[j] = pk(fc[2 * j].x, fc[2 * j + 1].x);
        pc.nkt[j] = pk(fc[2 * j].y, fc[2 * j + 1].y);
        pc.m[j] = pk(fc[2 * j].z, fc[2 * j + 1].z);
    }
    const int origin = (by - R) * kPitch + bx - R;
    const bool table = !VAR || (same && R >= 1 && (R <= kTables || R == Rt));
    const uint32_t table_at = tables_at + (VAR && table ? table_row(min(R, kTables + 1)) * kPitch * 16u : 0u);
    const uint32_t tab = keep(table_at - (uint32_t)origin * 16u);   // + 16 place: the entry of a record's bin
    auto load = [&](int i) {   // record i + lane (i itself may be negative)
        const bool ok = AFR_CHECK((uint32_t)(i + lane) < dc.cap + kFramePad, dc.derr);
        FrameRec r = load_rec(element(frec, ok ? i : 0));   // not ok: another record read, weight 0
        if (!ok) r.p.w = __int_as_float(origin - 1);   // a place before the box
        return r;
    };
    auto add = [&](const FrameRec &r, auto from_table) {
        const int place = __float_as_int(r.p.w);
        const bool ok = AFR_CHECK(place >= origin && place < origin + (2 * R + 2) * kPitch, dc.derr);
        float4 d;
        if constexpr (decltype(from_table)::value) d = lds4(ok ? tab + (uint32_t)place * 16u : table_at);
        else d = own_discs(place - origin, R, Rk);
        if (!ok) d = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        A.add(pc, d, r);
    };
    // The last iteration's lanes past the end read on (the frame arrays end in
    // kFramePad records of padding) and are dropped before they are summed.
    auto gather = [&](auto one_row, auto from_table) {
        constexpr bool ONE = decltype(one_row)::value;
        const uint2 r0 = lds2(rows_at);
        Cursor k{rows_at, (int)r0.x - lane, (int)r0.y};
        FrameRec ra, rb;
        advance<false>(k, 0, lane);
        ra = load(k.base);
        int j = 32;
        for (; j + 32 < (int)total; j += 64) {
            advance<ONE>(k, j, lane);
            rb = load(j + k.base);
            add(ra, from_table);
            advance<ONE>(k, j + 32, lane);
            ra = load(j + 32 + k.base);
            add(rb, from_table);
        }
        if (j < (int)total) {
            advance<ONE>(k, j, lane);
            rb = load(j + k.base);
            add(ra, from_table);
            ra = rb;
            j += 32;
        }
        if (j - 32 + lane < (int)total) add(ra, from_table);
    };
    if (total) {
        if (!table) {
            if constexpr (VAR) gather(std::false_type{}, std::false_type{});
        } else if (one) {
            gather(std::true_type{}, std::true_type{});
        } else {
            gather(std::false_type{}, std::true_type{});
        }
    }
    __syncwarp();   // the next block overwrites the row table
}

// Tile pixel of a block that lane k = lane mod 4 stores.
__device__ __forceinline__ int block_pixel(int tw, int lx, int ly) {
    return (2 * ly + ((threadIdx.x >> 1) & 1)) * tw + 2 * lx + (threadIdx.x & 1);
}

// Normalised colours and weight sums of a block's pixels from its sums.
template <bool KAHAN>
__device__ __forceinline__ void store_block(const ForwardSums<KAHAN> &A, int W, int H, int bx, int by, float4 fc,
                                            float4 *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    float vals[16];   // sum q of pixel k at q * 4 + k (q: S, r, g, b)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        upk(KAHAN ? sub2(A.S[j], A.C[j]) : A.S[j], vals[2 * j], vals[2 * j + 1]);
        upk(A.r[j], vals[4 + 2 * j], vals[4 + 2 * j + 1]);
        upk(A.g[j], vals[8 + 2 * j], vals[8 + 2 * j + 1]);
        upk(A.b[j], vals[12 + 2 * j], vals[12 + 2 * j + 1]);
    }
    const float tot = warp_reduce(vals);
    float q[4];   // to lane k
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = __shfl_sync(0xffffffffu, tot, 2 * (4 * i + (lane & 3)));
    const int x = bx + (lane & 1), y = by + ((lane >> 1) & 1);
    if (lane < 4 && x < W && y < H) {
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q[0] > 0.f) {
            const float inv = 1.f / q[0];
            o = make_float4(q[1] * inv, q[2] * inv, q[3] * inv, q[0] * ex2(-fc.z));
        }
        out[(size_t)y * W + x] = o;
    }
}

// Tile of (2 * tbx) x (2 * 32 / tbx) pixels per CTA: 32 blocks of 2x2, four
// per warp; its upper 1 / 2^lsplit for images whose tiles would not fill the GPU.
template <bool KAHAN, bool VAR>
__global__ void __launch_bounds__(256, 3) k_filter(int W, int H, int R, int ltbx, int lsplit, Fresh<float4> fconst,
                                                   const uint32_t *__restrict__ foff, const FrameRec *frec,
                                                   float4 *__restrict__ out, DebugCheck dc) {
    grid_order();
    __shared__ TileSmem ts;
    __shared__ float4 discs[(VAR ? kTableRows + kMaxRows : kMaxRows) * kPitch];
    const int warp = threadIdx.x >> 5, tw = 2 << ltbx, th = 64 >> ltbx >> lsplit, pixels = tw * th;
    const int x0 = blockIdx.x * tw, y0 = blockIdx.y * th;
    const FrameRec *const frec0 = frec;
    frec = keep(frec + (threadIdx.x & 31));
    const uint32_t tables_at = smem_at(discs), rows_at = smem_at(ts.rows[warp]);
    int Rt = R;
    float4 fc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < pixels) {
        fc = load_const(threadIdx.x, W, H, x0, y0, tw, fconst);
        ts.fc[threadIdx.x] = fc;
    }
    if (VAR) {   // the tile's largest footprint
        Rt = 0;
        for (int r = 1; r <= 8 && __syncthreads_or(__float_as_int(fc.w) >= r && threadIdx.x < pixels); ++r) {
            Rt = r;
            if (r <= kTables) fill_discs(discs + table_row(r) * kPitch, r);
        }
        if (Rt > kTables) fill_discs(discs + kTableRows * kPitch, Rt);
    } else {
        fill_discs(discs, R);
    }
    load_offsets(ts, W, H, Rt, x0, y0, tw, th, foff);
    __syncthreads();
    prefetch_tile(ts, tw + 2 * Rt + 1, th + 2 * Rt, frec0, dc.cap);
    for (int blk = warp; blk < 32 >> lsplit; blk += kWarps) {
        const int lx = blk & ((1 << ltbx) - 1), ly = blk >> ltbx;
        if (x0 + 2 * lx >= W || y0 + 2 * ly >= H) continue;   // warp-uniform
        ForwardSums<KAHAN> A;
        gather_block<VAR>(Rt, x0, y0, tw, lx, ly, frec, ts, tables_at, ts.rows[warp], rows_at, dc, A);
        store_block(A, W, H, x0 + 2 * lx, y0 + 2 * ly, ts.fc[block_pixel(tw, lx, ly)], out);
    }
}

// ---- batched form ---------------------------------------------------------------
// Two launches reconstruct many contexts. k_batch_sigma computes the widths
// and gather constants of every pixel of every context (thread per pixel,
// full occupancy: the per-pixel work is bound by the latency of the footprint
// loads). k_batch, a persistent kernel, then takes tiles of (2 tbx) x
// (64 / tbx) pixels of any context from a work queue (one atomic counter, the
// next tile claimed while the current one runs), largest contexts first, and
// filters them. Tiles never wait for one another.

// owning context of a batch-wide index: the last c with first[c] <= v
__device__ __forceinline__ int batch_owner(const uint32_t *first, int nctx, uint32_t v) {
    int lo = 0, hi = nctx - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= v) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Widths of every pixel of the batch: each block takes chunks of
// kBatchSigmaChunk pixels of one context (chunks are numbered per context from
// BatchCtx::s0) and reads the context's record once per chunk.
__global__ void __launch_bounds__(256) k_batch_sigma(const BatchCtx *__restrict__ cs, int nctx, uint32_t nchunks) {
    __shared__ uint32_t first[kMaxBatch];      // first chunk of each context
    __shared__ BatchCtx ctx;
    for (int c = threadIdx.x; c < nctx; c += blockDim.x) first[c] = cs[c].s0;
    __syncthreads();
    for (uint32_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        if (threadIdx.x == 0) ctx = cs[batch_owner(first, nctx, ch)];
        __syncthreads();
        const int W = ctx.W, H = ctx.H, P = W * H;
        const int p0 = (int)(ch - ctx.s0) * kBatchSigmaChunk, p1 = min(P, p0 + kBatchSigmaChunk);
        for (int p = p0 + (int)threadIdx.x; p < p1; p += blockDim.x) {
            const int px = p % W, py = p / W;
            Widths w = widths(__ldg(ctx.grad + p), tile_volume(px, py, W, H, ctx.S, ctx.ntx, ctx.window, ctx.tiles),
                              ctx.eps, ctx.prm);
            const float2 sg = make_float2(w.ss, w.st);
            ctx.sigma[p] = sg;
            const PixelFrame f = pixel_frame(px, py, W, H, ctx.R, sg, ctx.amin2);
            ctx.fconst[p] = make_float4(-f.ks, -f.kt, f.m, __int_as_float(ctx.R));
        }
        __syncthreads();
    }
}

template <bool KAHAN>
__global__ void __launch_bounds__(256, 3) k_batch(const BatchCtx *__restrict__ cs, int nctx, uint32_t total,
                                                  uint32_t *queue) {
    __shared__ TileSmem ts;
    __shared__ float4 discs[kMaxRows * kPitch];   // of the current tile's footprint radius
    __shared__ uint32_t item_buf[2];            // current and next claimed tile
    const uint32_t tables_at = smem_at(discs), rows_at = smem_at(ts.rows[threadIdx.x >> 5]);
    int held = -1;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) item_buf[0] = atomicAdd(queue, 1u);
    __syncthreads();
    for (int it = 0;; ++it) {
        const uint32_t item = item_buf[it & 1];
        if (item >= total) break;
        if (threadIdx.x == 0) item_buf[(it + 1) & 1] = atomicAdd(queue, 1u);
        int lo = 0, hi = nctx - 1;                  // owning context: last c with cs[c].a0 <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&cs[mid].a0) <= item) lo = mid;
            else hi = mid - 1;
        }
        const BatchCtx &x = cs[lo];
        const FrameRec *frec = keep(x.frec + (threadIdx.x & 31));
        const uint32_t local = item - x.a0;
        const int band = (int)(local / (uint32_t)x.ntiles_x), tile = (int)(local % (uint32_t)x.ntiles_x);
        const int tbx = x.tbx, tw = 2 * tbx, th = 2 * (32 / tbx), x0 = tile * tw, y0 = band * th;
        // every thread is past the last tile's gather
        if (threadIdx.x < kTilePixels) ts.fc[threadIdx.x] = load_const(threadIdx.x, x.W, x.H, x0, y0, tw, x.fconst);
        load_offsets(ts, x.W, x.H, x.R, x0, y0, tw, th, x.foff);
        if (x.R != held) fill_discs(discs, x.R);
        held = x.R;
        __syncthreads();
        for (int blk = warp; blk < 32; blk += kWarps) {
            const int lx = blk % tbx, ly = blk / tbx;
            if (x0 + 2 * lx >= x.W || y0 + 2 * ly >= x.H) continue;
            ForwardSums<KAHAN> A;
            gather_block<false>(x.R, x0, y0, tw, lx, ly, frec, ts, tables_at, ts.rows[warp], rows_at,
                                DebugCheck{x.fcap, x.derr}, A);
            store_block(A, x.W, x.H, x0 + 2 * lx, y0 + 2 * ly, ts.fc[block_pixel(tw, lx, ly)], x.out);
        }
        __syncthreads();
    }
}

// ---- adjoint -------------------------------------------------------------------
// A pass over the pixels (the same gather as the forward pass, with more sums),
// then one over the records. Between them, what a record needs of each pixel:
// a plane of float4 (-ks, -kt, shift, g_r / S) and one of float2 (g_g / S,
// g_b / S), g the loss gradient of the pixel's colour (0 where it holds no
// sample).
struct Adjoint {
    float4 *k;
    float2 *g;
};
struct AdjointRead {   // for the pass launched just after
    Fresh<float4> k;
    Fresh<float2> g;
};

// Weighted sums of one pixel over the records of its disc, in frame order. The
// totals of the width gradients over an image cancel to a small part of their
// terms, so the terms' rounding shows in them: the order of every sum, here and
// over the image (32 x 4 pixels a partial), is fixed, whatever a thread or a
// CTA holds.
template <bool PARAMS>
struct PixelSums {
    float S = 0.f, sc[3] = {0.f, 0.f, 0.f}, Ds = 0.f, dsc[3] = {0.f, 0.f, 0.f}, Dt = 0.f, dtc[3] = {0.f, 0.f, 0.f};
    // fc: (-ks, -kt, shift); a record of finite colour outside the disc adds exact zeros
    __device__ __forceinline__ void add(float4 r, float4 c, float cx, float cy, float4 fc, bool in) {
        const float ddx = r.x - cx, ddy = r.y - cy;
        const float d2 = fmaf(ddx, ddx, ddy * ddy);
        const float e2 = ex2(fmaf(d2, fc.x, fmaf(r.z, fc.y, fc.z))), w = in ? e2 : 0.f;
        S += w;
        if (PARAMS) {
            const float ws = w * d2, wt = in ? w * r.z : 0.f;
            sc[0] = fmaf(w, c.x, sc[0]); sc[1] = fmaf(w, c.y, sc[1]); sc[2] = fmaf(w, c.z, sc[2]);
            Ds += ws; Dt += wt;
            dsc[0] = fmaf(ws, c.x, dsc[0]); dsc[1] = fmaf(ws, c.y, dsc[1]); dsc[2] = fmaf(ws, c.z, dsc[2]);
            dtc[0] = fmaf(wt, c.x, dtc[0]); dtc[1] = fmaf(wt, c.y, dtc[1]); dtc[2] = fmaf(wt, c.z, dtc[2]);
        }
    }
};

// The pixel pass: a thread takes kBwdRows pixels of a column and walks the
// union of their discs, so a record is read once for all of them. Bound: the
// sectors of L1 (a warp's lanes read records of neighbouring bins, one 32-byte
// sector each): 512x512x8, 325 us with a pixel a thread that also searched its
// exponent shift again, 217 us so (two rows a thread 237, four 302: registers),
// 207 with the next record loaded ahead and five CTAs a SM (235 when the
// compiler takes the registers for four), 211 with the check for sums that are not
// finite.
// The filter's gather, lanes over records, takes 176 us, but sums in another
// order. A small image gets a pixel a thread (the same sums): with three its few
// CTAs leave most of the GPU idle behind one thread's walk (parameter gradients,
// 8 deep: 128x128 72 -> 37 us, 256x256 129 -> 103; 352x288, 264 CTAs of three
// rows, 140 -> 147, so the line lies at one and a half CTAs a SM). So do the radii 0
// and 1, whose rows share no record or few: 512x512x8 29 -> 24 and 55 -> 52 us,
// 1024x768x4 77 -> 64 and 112 -> 97 (at radius 2 three rows are faster from depth 4 on).
constexpr int kBwdX = 32, kBwdY = 4;
constexpr int kBwdRows = 3;
constexpr int kPartRows = 4;   // rows of one partial
static_assert(kBwdY % kPartRows == 0, "a CTA holds whole partials");

// The sums of one pixel from the records of its own disc alone.
template <bool PARAMS>
__device__ __noinline__ void walk_own(int W, int H, int R, int x, int y, float4 fc, const uint32_t *foff,
                                      const FrameRec *frec, DebugCheck dc, PixelSums<PARAMS> &out) {
    PixelSums<PARAMS> s;
    for (int v = max(-R, -y); v <= min(R, H - 1 - y); ++v) {
        const uint32_t *row = foff + (size_t)(y + v) * W;
        const int hw = half_width(R, v);
        const uint32_t beg = __ldg(row + max(0, x - hw)), end = __ldg(row + min(W - 1, x + hw) + 1);
        if (!AFR_CHECK(beg <= end && end <= dc.cap, dc.derr)) continue;
        for (uint32_t e = beg; e < end; ++e) {
            const FrameRec q = load_rec(frec + e);
            s.add(q.p, q.c, (float)x + 0.5f, (float)y + 0.5f, fc, true);
        }
    }
    out = s;
}

template <bool PARAMS, int ROWS>
__global__ void __launch_bounds__(kBwdX * kBwdY, 5) k_bwd_pixel(
    int W, int H, int R, int S_, int ntx, float window, float eps, AfrParams prm, const float4 *__restrict__ grad,
    const TilePartial *__restrict__ tiles, const float2 *__restrict__ sigma, const float4 *__restrict__ fconst,
    const uint32_t *__restrict__ foff, const FrameRec *__restrict__ frec, const float4 *__restrict__ gout, Adjoint adj,
    float *__restrict__ bparam, DebugCheck dc) {
    grid_order();
    __shared__ float part[kBwdY * ROWS][6];
    const int x = blockIdx.x * kBwdX + threadIdx.x, y0 = (blockIdx.y * kBwdY + threadIdx.y) * ROWS;
    float4 fc[ROWS];
    PixelSums<PARAMS> A[ROWS];
    if (x < W && y0 < H) {
#pragma unroll
        for (int k = 0; k < ROWS; ++k) fc[k] = __ldg(fconst + (size_t)min(y0 + k, H - 1) * W + x);
        const float cx = (float)x + 0.5f;
        for (int v = max(-R, -y0); v <= min(R + ROWS - 1, H - 1 - y0); ++v) {
            // records of each pixel's run of the row, and of the widest
            const uint32_t *row = foff + (size_t)(y0 + v) * W;
            uint32_t beg[ROWS], end[ROWS], e0 = 0xFFFFFFFFu, e1 = 0;
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
                beg[k] = end[k] = 0;
                if (v - k >= -R && v - k <= R && y0 + k < H) {
                    const int hw = half_width(R, v - k);
                    beg[k] = __ldg(row + max(0, x - hw));
                    end[k] = __ldg(row + min(W - 1, x + hw) + 1);
                    if (!AFR_CHECK(beg[k] <= end[k] && end[k] <= dc.cap, dc.derr)) beg[k] = end[k] = 0;
                    if (beg[k] < end[k]) {
                        e0 = min(e0, beg[k]);
                        e1 = max(e1, end[k]);
                    }
                }
            }
            if (e0 >= e1) continue;
            FrameRec next = load_rec(frec + e0);
            for (uint32_t e = e0; e < e1; ++e) {
                const FrameRec q = next;
                next = load_rec(frec + e + 1);   // the frame arrays end in padding
#pragma unroll
                for (int k = 0; k < ROWS; ++k)
                    A[k].add(q.p, q.c, cx, (float)(y0 + k) + 0.5f, fc[k], e - beg[k] < end[k] - beg[k]);
            }
        }
    }
    if (PARAMS && ROWS > 1) {
        // An infinite or NaN colour times the weight 0 is NaN: where a pixel's sums
        // may hold one from outside its disc, they are made again without it. (A
        // branch for every record instead: 189 -> 200 us at 512x512x8, 100 -> 154 at
        // 352x288x8; the colours selected: 227 and 115.)
#pragma unroll
        for (int k = 0; k < ROWS; ++k)
            if (x < W && y0 + k < H && !(fmaf(A[k].sc[0], 0.f, fmaf(A[k].sc[1], 0.f, A[k].sc[2] * 0.f)) == 0.f)) {
                PixelSums<PARAMS> own;
                walk_own(W, H, R, x, y0 + k, fc[k], foff, frec, dc, own);
                A[k] = own;
            }
    }
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
        const int y = y0 + k;
        float gp[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (x < W && y < H) {
            const size_t p = (size_t)y * W + x;
            const float4 g = __ldg(gout + p);
            const PixelSums<PARAMS> &s = A[k];
            const float inv = 1.f / s.S;
            const bool any = s.S > 0.f;
            adj.k[p] = make_float4(fc[k].x, fc[k].y, fc[k].z, any ? g.x * inv : 0.f);
            adj.g[p] = any ? make_float2(g.y * inv, g.z * inv) : make_float2(0.f, 0.f);
            if (PARAMS && any) {
                const float2 sgm = __ldg(sigma + p);
                const float gch[3] = {g.x, g.y, g.z};
                const float s3 = sgm.x * sgm.x * sgm.x, t3 = sgm.y * sgm.y * sgm.y;
                float gs = 0.f, gt = 0.f;
                for (int ch = 0; ch < 3; ++ch) {
                    const float C = s.sc[ch] * inv;
                    gs = fmaf(gch[ch], (s.dsc[ch] - C * s.Ds) * inv / s3, gs);
                    gt = fmaf(gch[ch], (s.dtc[ch] - C * s.Dt) * inv / t3, gt);
                }
                // chain through the width mapping; the widths depend on theta only
                const Widths wd = widths(__ldg(grad + p), tile_volume(x, y, W, H, S_, ntx, window, tiles), eps, prm);
                if (fmaxf(wd.raw_s, kSigmaSMin) >= prm.clamp_s) gp[2] = gs;
                else if (wd.raw_s > kSigmaSMin) { gp[0] = gs * wd.es; gp[1] = gs; }
                if (fmaxf(wd.raw_t, kSigmaTMin) >= prm.clamp_t) gp[5] = gt;
                else if (wd.raw_t > kSigmaTMin) { gp[3] = gt * wd.et; gp[4] = gt; }
            }
        }
        if (PARAMS) {
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                float v = gp[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (threadIdx.x == 0) part[threadIdx.y * ROWS + k][i] = v;
            }
        }
    }
    if (PARAMS) {
        __syncthreads();
        constexpr int kParts = kBwdY * ROWS / kPartRows;
        const int t = threadIdx.y * kBwdX + threadIdx.x, j = t / 6, i = t % 6, py = blockIdx.y * kParts + j;
        if (j < kParts && py < (H + kPartRows - 1) / kPartRows) {
            float acc = 0.f;
            for (int w = 0; w < kPartRows; ++w) acc += part[j * kPartRows + w][i];
            bparam[((size_t)py * gridDim.x + blockIdx.x) * 6 + i] = acc;
        }
    }
}

// Gradient of each frame record's colour: sum over the pixels whose disc
// holds the record's bin of (dL/dC_p / S_p) * shifted weight. Bound: the bytes
// L1 delivers to registers (24 a pixel read, 128 a clock and SM), so a thread
// takes two neighbouring records, which mostly share a bin or lie in adjacent
// ones, and reads each pixel of their two discs once (512x512x8: 101 us with 32
// bytes a pixel and record, 61 us).
struct RecordAt {
    int qx, qy;
    float fx, fy, a2;   // position from the centre of bin (qx, qy), a^2
};

__device__ __forceinline__ RecordAt record_at(const FrameRec *__restrict__ frec, uint32_t e) {
    const float4 r = __ldg(&frec[e].p);
    const int qx = (int)floorf(r.x), qy = (int)floorf(r.y);
    return {qx, qy, r.x - ((float)qx + 0.5f), r.y - ((float)qy + 0.5f), r.z};
}

__device__ __forceinline__ float pixel_weight(float4 k, float dx, float dy2, float a2) {
    return ex2(fmaf(fmaf(dx, dx, dy2), k.x, fmaf(a2, k.y, k.z)));
}

__device__ __forceinline__ void add_pixel(float4 k, float2 g, float w, float3 &a) {
    a.x = fmaf(k.w, w, a.x);
    a.y = fmaf(g.x, w, a.y);
    a.z = fmaf(g.y, w, a.z);
}

// One record: RT >= 0 is R at compile time (every pixel at a constant offset)
// for discs inside the image; the others loop.
template <int RT>
__device__ float3 record_gradient(const RecordAt &r, int W, int H, int R, AdjointRead adj) {
    float3 a = make_float3(0.f, 0.f, 0.f);
    if (RT >= 0 && r.qx >= RT && r.qy >= RT && r.qx < W - RT && r.qy < H - RT) {
        size_t p = (size_t)(r.qy - RT) * W + r.qx;
#pragma unroll
        for (int dy = -RT; dy <= RT; ++dy, p += W) {
            const float ey = r.fy - (float)dy, dy2 = ey * ey;
#pragma unroll
            for (int dx = -RT; dx <= RT; ++dx) {
                if (dx * dx + dy * dy > RT * RT) continue;
                const float4 k = adj.k[p + dx];
                add_pixel(k, adj.g[p + dx], pixel_weight(k, r.fx - (float)dx, dy2, r.a2), a);
            }
        }
        return a;
    }
    for (int dy = max(-R, -r.qy); dy <= min(R, H - 1 - r.qy); ++dy) {
        const float ey = r.fy - (float)dy, dy2 = ey * ey;
        const int hw = half_width(R, dy);
        const size_t p = (size_t)(r.qy + dy) * W + r.qx;
        for (int dx = max(-hw, -r.qx); dx <= min(hw, W - 1 - r.qx); ++dx) {
            const float4 k = adj.k[p + dx];
            add_pixel(k, adj.g[p + dx], pixel_weight(k, r.fx - (float)dx, dy2, r.a2), a);
        }
    }
    return a;
}

template <int RT>
__global__ void __launch_bounds__(256, 4) k_bwd_record(int W, int H, int R, const uint32_t *__restrict__ foff,
                                                       const FrameRec *__restrict__ frec, AdjointRead adj,
                                                       float *__restrict__ gcol) {
    grid_order();
    const uint32_t n = __ldg(foff + (size_t)W * H);
    const uint32_t pairs = n / 2 + (n & 1);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < pairs; i += gridDim.x * blockDim.x) {
        const uint32_t e = 2 * i;
        const bool two = e + 1 < n;
        const RecordAt u = record_at(frec, e), v = record_at(frec, two ? e + 1 : e);
        const int s = v.qx - u.qx;
        float3 a = make_float3(0.f, 0.f, 0.f), b = a;
        if (RT >= 0 && v.qy == u.qy && (s == 0 || s == 1) && u.qx >= RT && u.qy >= RT && v.qx < W - RT &&
            u.qy < H - RT && u.qx + RT + 1 < W) {
            const float vx = v.fx + (float)s;   // from the centre of the first record's bin
            size_t p = (size_t)(u.qy - RT) * W + u.qx;
#pragma unroll
            for (int dy = -RT; dy <= RT; ++dy, p += W) {
                const float eu = u.fy - (float)dy, ev = v.fy - (float)dy, yu = eu * eu, yv = ev * ev;
                // the row's pixels of both discs: columns -hw .. hw of the first, s - hw .. s + hw of the second
#pragma unroll
                for (int dx = -RT; dx <= RT + 1; ++dx) {
                    const bool in = dx * dx + dy * dy <= RT * RT, in1 = (dx - 1) * (dx - 1) + dy * dy <= RT * RT;
                    if (!in && !in1) continue;
                    const float4 k = adj.k[p + dx];
                    const float2 g = adj.g[p + dx];
                    if (in) add_pixel(k, g, pixel_weight(k, u.fx - (float)dx, yu, u.a2), a);
                    // outside a record's disc a pixel adds nothing, infinite gradients included
                    const float w = pixel_weight(k, vx - (float)dx, yv, v.a2);
                    if ((in && in1) || s == (in ? 0 : 1)) add_pixel(k, g, w, b);
                }
            }
        } else {
            a = record_gradient<RT>(u, W, H, R, adj);
            if (two) b = record_gradient<RT>(v, W, H, R, adj);
        }
        float *o = gcol + 3 * (size_t)e;
        o[0] = a.x;
        o[1] = a.y;
        o[2] = a.z;
        if (two) {
            o[3] = b.x;
            o[4] = b.y;
            o[5] = b.z;
        }
    }
}

// The six parameter gradients summed over the blocks' partials: one warp per
// parameter, each lane a compensated (Kahan) FP32 sum over a strided share of
// the blocks, then the 32 lane sums (value and compensation) added in a fixed
// order by lane 0.
__global__ void k_bwd_params(Fresh<float> part, int nblocks, float *__restrict__ out) {
    grid_order();
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k >= 6) return;
    float s = 0.f, c = 0.f;
#pragma unroll 8
    for (int i = lane; i < nblocks; i += 32) {
        const float y = part[(size_t)i * 6 + k] - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __shared__ float ss[6][32], cs[6][32];
    ss[k][lane] = s;
    cs[k][lane] = c;
    __syncwarp();
    if (lane == 0) {
        float S = 0.f, C = 0.f;
        for (int l = 0; l < 32; ++l) {
            const float y = ss[k][l] - cs[k][l] - C;
            const float t = S + y;
            C = (t - S) - y;
            S = t;
        }
        out[k] = S;
    }
}

// Colours rounded to the storage type, then widened as the frame view holds them.
// Bound: HBM, twelve of the 32 bytes of every record, so each is read and written
// whole: 1280x720x8 83 us, where a plane of colours alone took 36. (A
// reconstruction, which follows and reads all 32, went from 562 to 346 us there.)
template <int CT>
__global__ void k_set_colors(const float *__restrict__ rgb, const uint32_t *__restrict__ foff, int P,
                             FrameRec *__restrict__ frec) {
    uint32_t n = __ldg(foff + P);
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        float v[3] = {rgb[3 * (size_t)e], rgb[3 * (size_t)e + 1], rgb[3 * (size_t)e + 2]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (CT == AFR_F16) v[k] = __half2float(__float2half_rn(v[k]));
            if (CT == AFR_BF16) v[k] = __bfloat162float(__float2bfloat16_rn(v[k]));
        }
        float *c = &frec[e].c.x;   // the sequence number beside it stays
        *reinterpret_cast<float2 *>(c) = make_float2(v[0], v[1]);
        c[2] = v[2];
    }
}

const dim3 kQuadBlock(256);

}  // namespace

cudaError_t launch_sigma(AfrContext *c, const AfrParams *prm, bool keep, bool adaptive, cudaStream_t s) {
    const dim3 block(kSigX, kSigY), grid((c->W + kSigX - 1) / kSigX, (c->H + kSigY - 1) / kSigY);
    if (adaptive) {
        const float *prev = c->cov_r[c->cov_cur];
        c->cov_cur = 1 - c->cov_cur;
        float *next = c->cov_r[c->cov_cur];
#define AFR_SIGMA(K)                                                                                                    \
    k_sigma_adaptive<K><<<grid, block, 0, s>>>(c->W, c->H, c->S, c->ntx, c->cfg.window, c->cfg.eps_grad, *prm, c->grad, \
                                               c->tiles, c->amin2, prev, next, 0.5f, 8.f, c->foff, c->cov_n, c->sigma,  \
                                               c->fconst)
        if (keep) AFR_SIGMA(true);
        else AFR_SIGMA(false);
#undef AFR_SIGMA
        return cudaGetLastError();
    }
#define AFR_SIGMA(K, R_)                                                                                             \
    k_sigma<K, R_><<<grid, block, 0, s>>>(c->W, c->H, c->R, c->S, c->ntx, c->cfg.window, c->cfg.eps_grad, *prm, c->grad, \
                                          c->tiles, c->amin2, c->sigma, c->fconst)
    if (keep) AFR_SIGMA(true, -1);
    else {
        switch (c->R) {   // the radii of the tuner and the default
            case 3: AFR_SIGMA(false, 3); break;
            case 4: AFR_SIGMA(false, 4); break;
            case 5: AFR_SIGMA(false, 5); break;
            default: AFR_SIGMA(false, -1); break;
        }
    }
#undef AFR_SIGMA
    return cudaGetLastError();
}

cudaError_t launch_coverage_init(AfrContext *c, cudaStream_t s) {
    k_coverage_init<<<grid_for(c->P, 256), 256, 0, s>>>(c->P, (float)c->R, c->cov_r[c->cov_cur], c->cov_n);
    return cudaGetLastError();
}

cudaError_t launch_filter(AfrContext *c, float t_now, bool adaptive, float4 *out, cudaStream_t s, bool next) {
    (void)t_now;
    const DebugCheck dc{(uint32_t)c->frame_cap, c->derr};
    const int tbx = c->tile_bx, tw = 2 * tbx;
    // Fewer blocks a warp until the CTAs fill the GPU (three a SM) twice over:
    // 128x128x4 13.8 us with four blocks a warp, 10.4 with one; split further,
    // the tile's set-up costs more than the fuller last wave gives (640x480x8
    // FP16 122 us whole, 126 halved, 140 quartered).
    int lsplit = 0, th = 64 / tbx;
    const long long want = 2ll * 3 * device_sms();
    while (lsplit < 2 && th > 2 && (long long)((c->W + tw - 1) / tw) * ((c->H + th - 1) / th) < want) {
        ++lsplit;
        th /= 2;
    }
    dim3 grid((c->W + tw - 1) / tw, (c->H + th - 1) / th);
#define AFR_FILTER(K_, V_)                                                                                            \
    do {                                                                                                              \
        if (next)                                                                                                     \
            launch_next(k_filter<K_, V_>, grid, kQuadBlock, 0, s, c->W, c->H, c->R, __builtin_ctz(tbx), lsplit,       \
                        c->fconst, c->foff, c->frec, out, dc);                                                        \
        else                                                                                                          \
            k_filter<K_, V_><<<grid, kQuadBlock, 0, s>>>(c->W, c->H, c->R, __builtin_ctz(tbx), lsplit, c->fconst,     \
                                                         c->foff, c->frec, out, dc);                                  \
    } while (0)
    // colours stored in 16 bits: compensated weight sums
    if (c->ct == AFR_F32 && adaptive) AFR_FILTER(false, true);
    else if (c->ct == AFR_F32) AFR_FILTER(false, false);
    else if (adaptive) AFR_FILTER(true, true);
    else AFR_FILTER(true, false);
#undef AFR_FILTER
    return cudaGetLastError();
}

cudaError_t launch_backward(AfrContext *c, const float4 *grad_rgb, float *grad_col, float *grad_prm,
                            cudaStream_t s) {
    const auto bands = [&](int rows) { return (c->H + kBwdY * rows - 1) / (kBwdY * rows); };
    const int cols = (c->W + kBwdX - 1) / kBwdX;
    const int rows = c->R <= 1 || (long long)cols * bands(kBwdRows) < 3ll * device_sms() / 2 ? 1 : kBwdRows;
    const dim3 block(kBwdX, kBwdY), grid(cols, bands(rows));
    const DebugCheck dc{(uint32_t)c->frame_cap, c->derr};
    const Adjoint adj{c->bgrad, reinterpret_cast<float2 *>(c->bgrad + c->P)};
    const AfrParams &prm = c->recon_params;
#define AFR_BWD(P_, N_)                                                                                          \
    k_bwd_pixel<P_, N_><<<grid, block, 0, s>>>(c->W, c->H, c->R, c->S, c->ntx, c->cfg.window, c->cfg.eps_grad, prm,   \
                                           c->grad, c->tiles, c->sigma, c->fconst, c->foff, c->frec, grad_rgb, adj, \
                                           c->bparam, dc)
    if (grad_prm && rows == 1) AFR_BWD(true, 1);
    else if (grad_prm) AFR_BWD(true, kBwdRows);
    else if (rows == 1) AFR_BWD(false, 1);
    else AFR_BWD(false, kBwdRows);
#undef AFR_BWD
#define AFR_REC(R_)                                                                                              \
    launch_next(k_bwd_record<R_>, dim3(grid_for((size_t)c->P * c->b / 2, 256)), dim3(256), 0, s, c->W, c->H, c->R, c->foff, \
                c->frec, AdjointRead{adj.k, adj.g}, grad_col)
    if (grad_col) {
        switch (c->R) {   // the radii of the tuner and the default
            case 3: AFR_REC(3); break;
            case 4: AFR_REC(4); break;
            case 5: AFR_REC(5); break;
            default: AFR_REC(-1); break;
        }
    }
#undef AFR_REC
    if (grad_prm) launch_next(k_bwd_params, dim3(1), dim3(6 * 32), 0, s, c->bparam, backward_blocks(c->W, c->H), grad_prm);
    return cudaGetLastError();
}

cudaError_t launch_set_frame_colors(AfrContext *c, const float *rgb, cudaStream_t s) {
    int g = grid_for((size_t)c->P * c->b, 256);
    switch (c->ct) {
        case AFR_F32: k_set_colors<AFR_F32><<<g, 256, 0, s>>>(rgb, c->foff, c->P, c->frec); break;
        case AFR_F16: k_set_colors<AFR_F16><<<g, 256, 0, s>>>(rgb, c->foff, c->P, c->frec); break;
        default: k_set_colors<AFR_BF16><<<g, 256, 0, s>>>(rgb, c->foff, c->P, c->frec); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_batch(int ct, const BatchCtx *cs, int nctx, uint32_t nchunks, uint32_t total, uint32_t *queue,
                         int grid, cudaStream_t s) {
    k_batch_sigma<<<grid_for((size_t)nchunks * 256, 256), 256, 0, s>>>(cs, nctx, nchunks);
    if (ct == AFR_F32) k_batch<false><<<grid, kQuadBlock, 0, s>>>(cs, nctx, total, queue);
    else k_batch<true><<<grid, kQuadBlock, 0, s>>>(cs, nctx, total, queue);
    return cudaGetLastError();
}

int backward_blocks(int W, int H) { return ((W + kBwdX - 1) / kBwdX) * ((H + kPartRows - 1) / kPartRows); }

}  // namespace afr
