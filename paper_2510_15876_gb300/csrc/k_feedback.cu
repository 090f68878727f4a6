// k_feedback.cu -- sections 4, 4.2 and 6.1: finalise the per-tile records
// from the partials of the gradient pass (each tile's record with its
// undersampling measure u = 1 - min(1, m * mean_empty / empty), the mean number
// of empty slots following from the samples the gradient pass counted), and the
// tile error E with the gain control of section 4.1. Counts are summed as
// integers and the rest runs in FP32: FP64 issues at 1/64 of the FP32 rate on
// this part, and every output is FP32.
#include "afr_internal.cuh"

namespace afr {
namespace {

constexpr int kFbThreads = 1024;
constexpr int kFinThreads = 256;

__device__ __forceinline__ uint32_t tile_area(int t, int W, int H, int S, int ntx) {
    const int tx = t % ntx, ty = t / ntx;
    return (uint32_t)(min(S, W - tx * S) * min(S, H - ty * S));
}

// Mean number of empty slots over the tiles: an exact integer, divided once.
__device__ __forceinline__ float mean_empty_slots(int W, int H, int b, int ntiles, const unsigned long long *total) {
    return (float)((unsigned long long)W * H * b - *total) / (float)ntiles;
}

__global__ void __launch_bounds__(kFinThreads) k_finalize(int W, int H, int S, int ntx, int ntiles, int b, float m,
                                                          const TilePartial *__restrict__ tiles,
                                                          const unsigned long long *__restrict__ total,
                                                          AfrTileStats *__restrict__ out) {
    const float mean_empty = mean_empty_slots(W, H, b, ntiles, total);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ntiles) {
        const TilePartial tp = tiles[t];
        const uint32_t empty = tile_area(t, W, H, S, ntx) * (uint32_t)b - tp.n;
        const float sw = (float)tp.sw, ne = (float)tp.nonempty;
        AfrTileStats o;
        o.n = tp.n;
        o.empty_slots = empty;
        o.mean_L = sw > 0.f ? (float)tp.mean : 0.f;
        o.var_L = sw > 0.f ? (float)tp.m2 / sw : 0.f;
        o.mean_Gx = tp.nonempty ? tp.sgx / ne : 0.f;
        o.mean_Gy = tp.nonempty ? tp.sgy / ne : 0.f;
        o.mean_Gt = tp.nonempty ? tp.sgt / ne : 0.f;
        const float r = empty ? m * mean_empty / (float)empty : 0.f;
        o.u = empty ? 1.f - fminf(r, 1.f) : 0.f;
        out[t] = o;
    }
}

// Sum of each of N values over the block's kFbThreads threads: warp sums by
// shuffles, then warp 0 sums the warps' partials and shares the totals.
template <typename T, int N>
__device__ __forceinline__ void block_sum(T (&v)[N], T (*sh)[kFbThreads / 32]) {
    static_assert(kFbThreads == 1024, "warp 0 sums one partial per lane");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        T x = v[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sh[i][warp] = x;
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            T x = sh[i][lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) sh[i][0] = x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = sh[i][0];
    __syncthreads();
}

// A tile's terms of the tile error that follow from its own record.
struct TileTerm {
    float v, u, o;   // luminance variance, undersampling measure, occluded share of the tile's slots
};

__device__ __forceinline__ TileTerm tile_term(const TilePartial &tp, uint32_t slots, float m_mean_empty,
                                              uint32_t occluded) {
    TileTerm t;
    const uint32_t empty = slots - tp.n;
    const float sw = (float)tp.sw;
    t.v = sw > 0.f ? (float)tp.m2 / sw : 0.f;
    // 1 - min(1, m mean_empty / empty), 0 without empty slots: one rounded division,
    // as in the tile record, so that a tile exactly at the limit gets 0 here too
    t.u = empty ? 1.f - fminf(m_mean_empty / (float)empty, 1.f) : 0.f;
    t.o = (float)occluded / (float)slots;
    return t;
}

// Sections 6.1 and 4.1: tile error shares and gain control, one block over
// the tile records. The sample ages were summed by the gradient pass, which
// reads the times anyway (a pass over the times of its own took 51 us at
// 1920x1080x16). Non-empty pixels and tiles with samples are summed as
// integers, exactly; the rest are tree sums in FP32.
__global__ void __launch_bounds__(kFbThreads) k_tile_error(int W, int H, int S, int ntx, int ntiles, int b, float m,
                                                           float kappa, float lambda, float importance, float eps,
                                                           const TilePartial *__restrict__ tiles,
                                                           const unsigned long long *__restrict__ total,
                                                           const uint32_t *__restrict__ occluded,
                                                           float *__restrict__ E, AfrGain *__restrict__ gain) {
    __shared__ unsigned long long shi[2][kFbThreads / 32];
    __shared__ float sh[6][kFbThreads / 32];
    const float m_mean_empty = m * mean_empty_slots(W, H, b, ntiles, total);
    unsigned long long cnt[2] = {0ull, 0ull};   // non-empty pixels, tiles with samples
    // sums: v, u, o, spatial gradient, temporal gradient, tile mean ages
    float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
        const TilePartial tp = tiles[t];
        const TileTerm tt = tile_term(tp, tile_area(t, W, H, S, ntx) * (uint32_t)b, m_mean_empty, occluded ? occluded[t] : 0u);
        cnt[0] += tp.nonempty;
        cnt[1] += tp.n ? 1u : 0u;
        acc[0] += tt.v;
        acc[1] += tt.u;
        acc[2] += tt.o;
        acc[3] += 0.5f * (tp.sgx + tp.sgy);
        acc[4] += tp.sgt;
        acc[5] += tp.n ? tp.age / (float)tp.n : 0.f;
    }
    block_sum(cnt, shi);
    block_sum(acc, sh);
    // E = s (kappa v / sum v + lambda u / sum u + (1 - kappa - lambda) o / sum o)
    const float wv = acc[0] > 0.f ? kappa / acc[0] : 0.f, wu = acc[1] > 0.f ? lambda / acc[1] : 0.f,
                wo = occluded && acc[2] > 0.f ? (1.f - kappa - lambda) / acc[2] : 0.f;
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
        const uint32_t A = tile_area(t, W, H, S, ntx);
        const TileTerm tt = tile_term(tiles[t], A * (uint32_t)b, m_mean_empty, occluded ? occluded[t] : 0u);
        E[t] = (float)A * (wv * tt.v + wu * tt.u + wo * tt.o);
    }
    if (threadIdx.x == 0 && gain) {
        const float nonempty = (float)cnt[0];
        const float dcds = cnt[0] ? acc[3] / nonempty : 0.f, dcdt = cnt[0] ? acc[4] / nonempty : 0.f;
        const float T = cnt[1] ? acc[5] / (float)cnt[1] : 0.f;
        const float Sw = importance * dcdt * T / (dcds > eps ? dcds : eps);
        const float P = (float)W * (float)H;
        float N = Sw > 0.f ? P / (Sw * Sw) : P;
        N = N < 1.f ? 1.f : (N > P ? P : N);
        AfrGain g;
        g.dC_ds = dcds;
        g.dC_dt = dcdt;
        g.mean_age = T;
        g.tile_width = Sw;
        g.tile_count = N;
        *gain = g;
    }
}

}  // namespace

cudaError_t launch_tile_error(AfrContext *c, float kappa, float lambda, float importance, const uint32_t *occluded,
                              float *E, AfrGain *gain, cudaStream_t s) {
    k_tile_error<<<1, kFbThreads, 0, s>>>(c->W, c->H, c->S, c->ntx, c->ntiles, c->b, c->cfg.undersample_m, kappa, lambda,
                                          importance, c->cfg.eps_grad, c->tiles, tile_total(c), occluded, E, gain);
    return cudaGetLastError();
}

cudaError_t launch_feedback(AfrContext *c, AfrTileStats *out, cudaStream_t s) {
    k_finalize<<<(c->ntiles + kFinThreads - 1) / kFinThreads, kFinThreads, 0, s>>>(
        c->W, c->H, c->S, c->ntx, c->ntiles, c->b, c->cfg.undersample_m, c->tiles, tile_total(c), out);
    return cudaGetLastError();
}

}  // namespace afr
