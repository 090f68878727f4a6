// k_reproject.cu -- section 6.2: move every buffered sample to the display
// time along its screen velocity and rebin it into the frame view (a CSR
// over destination pixels), ordered within each bin by sequence number.
//
//  count:  thread per queue slot; x' = x + m_x (t_now - t) with one rounding
//          per operation (__fmul_rn / __fadd_rn, so no contraction), drops
//          samples leaving the image and counts per destination bin (the
//          lanes of a warp grouped by bin with one match instruction).
//  scan:   bin offsets.
//  list:   each moved sample (its bin kept by the count pass, 4 bytes a
//          slot) writes its slot index and its sequence number, 8 bytes, into its
//          bin's list (unordered), at the ticket its bin's cursor returns (the
//          scan starts the cursors at the bin offsets).
//  place:  thread per frame record, in bin order: the slot of list entry e
//          is moved again, its rank in the bin is the number of sequence
//          numbers in the bin's list below its own (sequence numbers are
//          unique), and it writes the 32-byte frame record (x', y', a^2, its bin's
//          place, its colour in FP32, its sequence number) to the bin's offset +
//          rank. The lanes of a warp mostly share a bin, so the rank scans are
//          broadcast reads and the record writes whole sectors; the frame view,
//          and every sum over it, is deterministic without a reorder pass over
//          the records. Each bin's smallest a^2 (the filter's exponent shift) is
//          the minimum over the bin's warp segments, one atomic each. Samples of
//          the reconstructor's queue, which lie in arrival order, are placed
//          from that order instead (k_place_fifo), those of crowded bins by
//          sorting the bin (place_crowded).
//
// Bound: HBM (place), atomic latency (list). 1920x1080x16, FP32 colours: list
// 191 -> 148 us with one 8-byte entry for two 4-byte ones, place 533 -> 504 us
// with position and motion in one 16-byte field and 32-byte records; placing
// from the queues' slot order (no slot in the list, coalesced reads, records
// written out of order) measured 123 + 562 us, and 30 us more at 1024x1024x8.
// For the reconstructor's queue that order wins: 1024x1024, 4 samples a pixel,
// list and place 307 -> 191 us.
#include "afr_internal.cuh"

namespace afr {
namespace {

struct Moved {
    bool ok;
    uint32_t bin;
    float xp, yp, a2;
};

__device__ __forceinline__ Moved move_sample(float4 xm, float t, float t_now, int W, int H) {
    Moved r;
    float a = __fsub_rn(t_now, t);
    r.xp = __fadd_rn(xm.x, __fmul_rn(xm.z, a));
    r.yp = __fadd_rn(xm.y, __fmul_rn(xm.w, a));
    r.a2 = __fmul_rn(a, a);
    r.ok = r.xp >= 0.f && r.xp < (float)W && r.yp >= 0.f && r.yp < (float)H;
    r.bin = r.ok ? (uint32_t)(int)floorf(r.yp) * (uint32_t)W + (uint32_t)(int)floorf(r.xp) : kInvalid;
    return r;
}

// Section 6.2 with camera matrices: the stored hit point rendered by the
// current camera, plus the sample's own screen motion times its age; each
// matrix row summed left to right, one rounding per operation.
__device__ __forceinline__ float cam_row(const Camera &c, int r, float4 w) {
    float v = __fmul_rn(c.m[4 * r], w.x);
    v = __fadd_rn(v, __fmul_rn(c.m[4 * r + 1], w.y));
    v = __fadd_rn(v, __fmul_rn(c.m[4 * r + 2], w.z));
    return __fadd_rn(v, c.m[4 * r + 3]);
}

__device__ __forceinline__ Moved move_camera(float4 w, float4 xm, float t, float t_now, int W, int H,
                                             const Camera &cam) {
    Moved r;
    const float cx = cam_row(cam, 0, w), cy = cam_row(cam, 1, w), cw = cam_row(cam, 2, w);
    const float sx = __fmul_rn(__fadd_rn(__fmul_rn(__fdiv_rn(cx, cw), 0.5f), 0.5f), (float)W);
    const float sy = __fmul_rn(__fadd_rn(__fmul_rn(__fdiv_rn(cy, cw), 0.5f), 0.5f), (float)H);
    const float a = __fsub_rn(t_now, t);
    r.xp = __fadd_rn(sx, __fmul_rn(xm.z, a));
    r.yp = __fadd_rn(sy, __fmul_rn(xm.w, a));
    r.a2 = __fmul_rn(a, a);
    r.ok = cw > 0.f && r.xp >= 0.f && r.xp < (float)W && r.yp >= 0.f && r.yp < (float)H;
    r.bin = r.ok ? (uint32_t)(int)floorf(r.yp) * (uint32_t)W + (uint32_t)(int)floorf(r.xp) : kInvalid;
    return r;
}

// slot i -> (pixel, storage slot); b is a power of two in the common case
__device__ __forceinline__ void split_slot(uint32_t i, int b, int bshift, uint32_t &p, int &s) {
    if (bshift >= 0) {
        p = i >> bshift;
        s = (int)(i & (uint32_t)(b - 1));
    } else {
        p = i / (uint32_t)b;
        s = (int)(i - p * (uint32_t)b);
    }
}

__device__ __forceinline__ bool slot_live(uint32_t st, int s, int b) {
    int n = (int)(st & 0xFFFFu), h = (int)(st >> 16);
    int age = h - 1 - s;
    if (age < 0) age += b;
    return age < n;
}

// FIFO: the slots are the reconstructor queue's, live below min(*state, nslots)
// (state then points at its count of accepted samples). The slot's data is
// loaded together with its pixel's state (one round trip, not two).
template <bool FIFO, bool CAM>
__device__ __forceinline__ bool live_move(uint32_t i, uint32_t nlive, int b, int bshift, int W, int H, float t_now,
                                          const Camera &cam, const float4 *__restrict__ world,
                                          const uint32_t *__restrict__ state, const float4 *__restrict__ r_xm, const float *__restrict__ r_t, Moved &mv,
                                          bool &live) {
    uint32_t p = 0, st = 0;
    int s = 0;
    live = false;
    if (FIFO) {
        if (i >= nlive) return false;
    } else {
        split_slot(i, b, bshift, p, s);
        st = __ldg(state + p);
    }
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
    if (CAM) w = __ldg(world + i);
    const float4 xm = __ldg(r_xm + i);
    const float t = __ldg(r_t + i);
    if (!FIFO && !slot_live(st, s, b)) return false;
    live = true;
    mv = CAM ? move_camera(w, xm, t, t_now, W, H, cam) : move_sample(xm, t, t_now, W, H);
    return mv.ok;
}

// The reconstructor's queue of N slots holds the samples in the order of their
// arrival, which is that of their sequence numbers: slot of the oldest sample
// (total: samples it has taken), a slot's arrival rank, and the way back.
__device__ __forceinline__ uint32_t oldest_slot(uint32_t total, uint32_t N) { return total > N ? total % N : 0u; }
__device__ __forceinline__ uint32_t arrival_rank(uint32_t i, uint32_t oldest, uint32_t N) {
    return i >= oldest ? i - oldest : i + (N - oldest);
}
__device__ __forceinline__ uint32_t ranked_slot(uint32_t rank, uint32_t oldest, uint32_t N) {
    return rank < N - oldest ? rank + oldest : rank - (N - oldest);
}

// A warp takes kCountRows rows of 32 slots at a time, their loads issued
// together.
constexpr int kCountRows = 4;
template <bool FIFO, bool CAM>
__global__ void __launch_bounds__(256) k_count(uint32_t nslots, int b, int bshift, int W, int H, float t_now,
                                               Camera cam, const float4 *__restrict__ world,
                                               const uint32_t *__restrict__ state, const float4 *__restrict__ r_xm, const float *__restrict__ r_t,
                                               uint32_t *__restrict__ fcnt, uint32_t *__restrict__ sbin,
                                               unsigned long long *__restrict__ dcount) {
    grid_order();
    if (FIFO && blockIdx.x == 0 && threadIdx.x == 0) dcount[CNT_CROWDED] = 0ull;   // the scan sets it
    const uint32_t nlive = FIFO ? min(__ldg(state), nslots) : 0u;
    const int lane = threadIdx.x & 31;
    uint32_t dropped = 0;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i0 = warp * 32u * kCountRows; i0 < nslots; i0 += nwarps * 32u * kCountRows) {
        Moved mv[kCountRows];
        bool live[kCountRows];
#pragma unroll
        for (int r = 0; r < kCountRows; ++r) {
            const uint32_t i = i0 + (uint32_t)(r * 32 + lane);
            mv[r].ok = false;
            live[r] = false;
            if (i < nslots)
                live_move<FIFO, CAM>(i, nlive, b, bshift, W, H, t_now, cam, world, state, r_xm, r_t, mv[r],
                                     live[r]);
        }
#pragma unroll
        for (int r = 0; r < kCountRows; ++r) {
            const uint32_t i = i0 + (uint32_t)(r * 32 + lane);
            dropped += live[r] && !mv[r].ok;
            const uint32_t key = mv[r].ok ? mv[r].bin : kInvalid;
            if (i < nslots) sbin[i] = key;
            const unsigned peers = __match_any_sync(0xffffffffu, key);
            if (mv[r].ok && lane == __ffs(peers) - 1) atomicAdd(fcnt + mv[r].bin, (uint32_t)__popc(peers));
        }
    }
    const uint32_t d = __reduce_add_sync(0xffffffffu, dropped);
    if (lane == 0 && d) atomicAdd(dcount + CNT_DROPPING, (unsigned long long)d);
}

// The slots' bins from the count pass (kInvalid: dead or moved out). A warp
// takes kListRows rows of 32 slots at a time and issues every row's ticket
// atomic before it reads any back, so the atomics' latencies overlap.
// FIFO: the entry is the sample's arrival rank, which orders the bin as the
// sequence number does and names the slot as well.
constexpr int kListRows = 8;
template <bool FIFO>
__global__ void __launch_bounds__(256) k_list(uint32_t nslots, const uint32_t *__restrict__ sbin,
                                              const uint32_t *__restrict__ r_seq, const uint32_t *__restrict__ state,
                                              uint32_t *__restrict__ fcur, uint32_t *__restrict__ flist, DebugCheck dc) {
    grid_order();
    const uint32_t oldest = FIFO ? oldest_slot(__ldg(state), nslots) : 0u;
    const int lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i0 = warp * 32u * kListRows; i0 < nslots; i0 += nwarps * 32u * kListRows) {
        uint32_t bin[kListRows], sq[kListRows], first[kListRows];
        unsigned peers[kListRows];
#pragma unroll
        for (int r = 0; r < kListRows; ++r) {
            const uint32_t i = i0 + (uint32_t)(r * 32 + lane);
            bin[r] = kInvalid;
            sq[r] = 0;
            if (i < nslots) {
                bin[r] = __ldg(sbin + i);
                sq[r] = FIFO ? arrival_rank(i, oldest, nslots) : __ldg(r_seq + i);
            }
        }
#pragma unroll
        for (int r = 0; r < kListRows; ++r) {
            peers[r] = __match_any_sync(0xffffffffu, bin[r]);
            first[r] = 0;
            if (bin[r] != kInvalid && lane == __ffs(peers[r]) - 1)
                first[r] = atomicAdd(fcur + bin[r], (uint32_t)__popc(peers[r]));
        }
#pragma unroll
        for (int r = 0; r < kListRows; ++r) {
            const uint32_t i = i0 + (uint32_t)(r * 32 + lane);
            const uint32_t f = __shfl_sync(0xffffffffu, first[r], bin[r] != kInvalid ? __ffs(peers[r]) - 1 : lane);
            if (bin[r] == kInvalid) continue;
            const uint32_t at = f + __popc(peers[r] & ((1u << lane) - 1u));
            if (AFR_CHECK(at < dc.cap, dc.derr)) {
                if (FIFO) flist[at] = sq[r];
                else reinterpret_cast<uint2 *>(flist)[at] = make_uint2(i, sq[r]);
            }
        }
    }
}

// A record's place in a bin above kSortedBinMax records: fcur holds the bin's
// end (the list's cursor) and is counted down (arrival order); the bin is
// counted as unsorted.
__device__ __forceinline__ uint32_t unsorted_rank(uint32_t *fcur, uint32_t bin, uint32_t beg, unsigned long long *dcount) {
    const uint32_t rank = atomicSub(fcur + bin, 1u) - 1u - beg;
    if (rank == 0) atomicAdd(dcount + CNT_UNSORTED, 1ull);
    return rank;
}

// The frame records arrive in bin order, so the lanes of a warp that share a
// bin are one segment: its smallest a^2 goes to amin2 with one atomic (the
// filter's exponent shift; bit order = value order for a^2 >= 0).
template <int CT, bool CAM>
__global__ void __launch_bounds__(256) k_place_queues(int W, int H, float t_now, Camera cam, const float4 *__restrict__ world,
                                               const float4 *__restrict__ r_xm,
                                               const float *__restrict__ r_t, const void *__restrict__ r_col, uint32_t P,
                                               const uint32_t *__restrict__ foff, Fresh<uint2> flist,
                                               uint32_t *__restrict__ fcur, uint32_t *__restrict__ amin2,
                                               FrameRec *__restrict__ frec, unsigned long long *__restrict__ dcount,
                                               DebugCheck dc, uint32_t nsrc) {
    grid_order();
    using CS = ColorStore<CT>;
    uint32_t n = __ldg(foff + P);
    if (!AFR_CHECK(n <= dc.cap, dc.derr)) n = 0;
    const int lane = threadIdx.x & 31;
    const uint32_t stride = gridDim.x * blockDim.x;
    // warp-uniform trip count: every lane of a warp reaches the match below
    for (uint32_t e0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); e0 < n; e0 += stride) {
        const uint32_t e = e0 + (uint32_t)lane;
        uint2 en = make_uint2(0u, 0u);   // slot, sequence number
        bool ok = e < n;
        if (ok) {
            en = flist[e];
            ok = AFR_CHECK(en.x < nsrc, dc.derr);
        }
        const uint32_t i = en.x, sq = en.y;
        Moved mv;
        mv.ok = false;
        mv.bin = kInvalid;
        typename CS::T col;
        if (ok) {
            col = CS::raw(r_col, i);
            mv = CAM ? move_camera(__ldg(world + i), __ldg(r_xm + i), __ldg(r_t + i), t_now, W, H, cam)
                     : move_sample(__ldg(r_xm + i), __ldg(r_t + i), t_now, W, H);
        }
        const uint32_t key = mv.ok ? mv.bin : kInvalid;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        if (!mv.ok) continue;
        const uint32_t bits = __reduce_min_sync(peers, __float_as_uint(mv.a2));
        if (lane == __ffs(peers) - 1) atomicMin(amin2 + mv.bin, bits);
        const uint32_t beg = __ldg(foff + mv.bin), end = __ldg(foff + mv.bin + 1);
        uint32_t rank = 0;
        if (end - beg <= (uint32_t)kSortedBinMax) {
#pragma unroll 4
            for (uint32_t k = beg; k < end; ++k) rank += flist[k].y < sq;
        } else {
            rank = unsorted_rank(fcur, mv.bin, beg, dcount);
        }
        const uint32_t d = beg + rank;
        if (!AFR_CHECK(d < n, dc.derr)) continue;
        const float3 c = CS::widen(col);
        store_rec(frec + d, {make_float4(mv.xp, mv.yp, mv.a2, bin_place(mv.xp, mv.yp)),
                             make_float4(c.x, c.y, c.z, __uint_as_float(sq))});
    }
}

// The reconstructor's queue holds samples in arrival order, anywhere in the
// image: gathered in bin order, each field of a record cost a sector of its
// own. So a thread takes a slot, in queue order, and writes its record (one
// whole sector) where its place among the bin's arrival ranks puts it, four
// ranks a load. Every lane walks another list, so that only pays while the lists
// are short; longer ones are left to place_crowded.
constexpr uint32_t kCrowded = 64;

// Bins of kCrowded + 1 to kSortedBinMax records of the reconstructor's queue: the
// bin's arrival ranks are sorted in shared memory and its samples gathered in
// that order, by a warp up to kWarpBin records, else by a block. Neighbouring
// bins go to different blocks, for crowds are local.
// A reprojection of two million samples in 2,700 bins (some 800 each): 276 us;
// walking the lists 1147, gathering everything in bin order 413 to 447. 256x256
// with 32, 48, 64 and 96 samples a pixel: 158, 266, 393 and 597 us; gathering in
// bin order 158, 247, 349, 579, walking the lists 170, 304, 456, 650. Lines at 16,
// 24 and 32 records measured 184 to 201, 288, 392 and 613.
constexpr uint32_t kWarpBin = 512;
constexpr int kFifoWarps = 8;
static_assert(kFifoWarps * kWarpBin <= (uint32_t)kSortedBinMax, "a warp sorts in its share of the block's ranks");

struct CrowdSmem {
    uint32_t ranks[kSortedBinMax];
    uint32_t found[32 * kFifoWarps], n;
};

// Threads t, t + T, ... of T sort and place the bin whose list entries are beg .. beg + len - 1.
template <int CT, bool CAM, class Sync>
__device__ __forceinline__ void place_sorted(uint32_t *ranks, uint32_t t, uint32_t T, Sync sync, uint32_t beg, uint32_t len,
                                             uint32_t nslots, uint32_t oldest, int W, int H, float t_now,
                                             const Camera &cam, const float4 *__restrict__ world,
                                             const float4 *__restrict__ r_xm, const float *__restrict__ r_t,
                                             const uint32_t *__restrict__ r_seq, const void *__restrict__ r_col,
                                             const Fresh<uint32_t> &flist, FrameRec *__restrict__ frec, const DebugCheck &dc) {
    using CS = ColorStore<CT>;
    uint32_t n2 = 32;
    while (n2 < len) n2 *= 2;
    for (uint32_t k = t; k < n2; k += T) ranks[k] = k < len ? flist[beg + k] : kInvalid;
    for (uint32_t k = 2; k <= n2; k *= 2)
        for (uint32_t j = k / 2; j > 0; j /= 2) {   // bitonic, ascending
            sync();
            for (uint32_t c = t; c < n2 / 2; c += T) {
                const uint32_t i = 2 * c - (c & (j - 1));
                const uint32_t a = ranks[i], b = ranks[i + j];
                if ((a > b) == ((i & k) == 0)) {
                    ranks[i] = b;
                    ranks[i + j] = a;
                }
            }
        }
    sync();
    for (uint32_t r = t; r < len; r += T) {
        const uint32_t i = ranked_slot(ranks[r], oldest, nslots);
        if (!AFR_CHECK(i < nslots, dc.derr)) continue;
        const Moved mv = CAM ? move_camera(__ldg(world + i), __ldg(r_xm + i), __ldg(r_t + i), t_now, W, H, cam)
                             : move_sample(__ldg(r_xm + i), __ldg(r_t + i), t_now, W, H);
        const float3 c = CS::widen(CS::raw(r_col, i));
        store_rec(frec + beg + r, {make_float4(mv.xp, mv.yp, mv.a2, bin_place(mv.xp, mv.yp)),
                                   make_float4(c.x, c.y, c.z, __uint_as_float(__ldg(r_seq + i)))});
    }
    sync();   // the next bin overwrites the ranks
}

template <int CT, bool CAM>
__device__ __forceinline__ void place_crowded(CrowdSmem &sm, uint32_t nslots, uint32_t oldest, int W, int H, float t_now,
                                              const Camera &cam, const float4 *__restrict__ world,
                                              const float4 *__restrict__ r_xm, const float *__restrict__ r_t,
                                              const uint32_t *__restrict__ r_seq, const void *__restrict__ r_col,
                                              const uint32_t *__restrict__ foff, const Fresh<uint32_t> &flist,
                                              FrameRec *__restrict__ frec, const DebugCheck &dc) {
    const uint32_t P = (uint32_t)W * (uint32_t)H, G = gridDim.x, T = 32 * kFifoWarps, warp = threadIdx.x >> 5;
    for (uint32_t q0 = blockIdx.x; q0 < P; q0 += G * T) {   // bins q0, q0 + G, ...
        if (threadIdx.x == 0) sm.n = 0;
        __syncthreads();
        const unsigned long long q = q0 + (unsigned long long)threadIdx.x * G;
        if (q < P) {
            const uint32_t len = __ldg(foff + q + 1) - __ldg(foff + q);
            if (len > kCrowded && len <= (uint32_t)kSortedBinMax) sm.found[atomicAdd(&sm.n, 1u)] = (uint32_t)q;
        }
        __syncthreads();
        const uint32_t nf = sm.n;
        const auto place = [&](uint32_t *ranks, uint32_t t, uint32_t threads, auto sync, uint32_t f, bool block) {
            const uint32_t beg = __ldg(foff + sm.found[f]), end = __ldg(foff + sm.found[f] + 1), len = end - beg;
            if (block == (len <= kWarpBin) || !AFR_CHECK(end <= dc.cap, dc.derr)) return;   // uniform over the threads
            place_sorted<CT, CAM>(ranks, t, threads, sync, beg, len, nslots, oldest, W, H, t_now, cam, world, r_xm, r_t,
                                  r_seq, r_col, flist, frec, dc);
        };
        for (uint32_t f = warp; f < nf; f += kFifoWarps)
            place(sm.ranks + warp * kWarpBin, threadIdx.x & 31, 32, [] { __syncwarp(); }, f, false);
        __syncthreads();
        for (uint32_t f = 0; f < nf; ++f) place(sm.ranks, threadIdx.x, T, [] { __syncthreads(); }, f, true);
        __syncthreads();   // the next bins' count overwrites this one's
    }
}

template <int CT, bool CAM>
__global__ void __launch_bounds__(32 * kFifoWarps) k_place_fifo(uint32_t nslots, int W, int H, float t_now, Camera cam,
                                                    const float4 *__restrict__ world, const uint32_t *__restrict__ state,
                                                    const float4 *__restrict__ r_xm,
                                                    const float *__restrict__ r_t, const uint32_t *__restrict__ r_seq,
                                                    const void *__restrict__ r_col, const uint32_t *__restrict__ foff,
                                                    Fresh<uint32_t> flist, uint32_t *__restrict__ fcur,
                                                    uint32_t *__restrict__ amin2, FrameRec *__restrict__ frec,
                                                    unsigned long long *__restrict__ dcount, DebugCheck dc) {
    grid_order();
    using CS = ColorStore<CT>;
    const uint32_t nlive = min(__ldg(state), nslots), oldest = oldest_slot(__ldg(state), nslots);
    const int lane = threadIdx.x & 31;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < nlive; i0 += stride) {
        const uint32_t i = i0 + (uint32_t)lane;
        Moved mv;
        bool live;
        mv.ok = false;
        typename CS::T col;
        uint32_t sq = 0;
        if (i < nlive) {
            col = CS::raw(r_col, i);
            sq = __ldg(r_seq + i);
            live_move<true, CAM>(i, nlive, 1, 0, W, H, t_now, cam, world, state, r_xm, r_t, mv, live);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, mv.ok ? mv.bin : kInvalid);
        if (!mv.ok) continue;
        const uint32_t beg = __ldg(foff + mv.bin), end = __ldg(foff + mv.bin + 1);
        const uint32_t bits = __reduce_min_sync(peers, __float_as_uint(mv.a2));
        if (lane == __ffs(peers) - 1) atomicMin(amin2 + mv.bin, bits);
        if (!AFR_CHECK(beg < end && end <= dc.cap, dc.derr)) continue;
        uint32_t rank = 0;
        const uint32_t len = end - beg, mine = arrival_rank(i, oldest, nslots);
        if (len <= kCrowded) {
            for (uint32_t k = beg & ~3u; k < end; k += 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(&flist[k]);
                const uint32_t j = k - beg;   // entries outside the bin wrap past its length or lie beyond it
                rank += (uint32_t)((j < len) & (v.x < mine)) + (uint32_t)((j + 1u < len) & (v.y < mine)) +
                        (uint32_t)((j + 2u < len) & (v.z < mine)) + (uint32_t)((j + 3u < len) & (v.w < mine));
            }
        } else if (len <= (uint32_t)kSortedBinMax) {
            continue;
        } else {
            rank = unsorted_rank(fcur, mv.bin, beg, dcount);
        }
        const uint32_t d = beg + rank;
        if (!AFR_CHECK(d < end, dc.derr)) continue;
        const float3 c = CS::widen(col);
        store_rec(frec + d, {make_float4(mv.xp, mv.yp, mv.a2, bin_place(mv.xp, mv.yp)),
                             make_float4(c.x, c.y, c.z, __uint_as_float(sq))});
    }
    __shared__ CrowdSmem crowd;
    if (dcount[CNT_CROWDED])
        place_crowded<CT, CAM>(crowd, nslots, oldest, W, H, t_now, cam, world, r_xm, r_t, r_seq, r_col, foff, flist, frec, dc);
}

}  // namespace

cudaError_t launch_reproject(AfrContext *c, float t_now, const Camera *camp, cudaStream_t s) {
    cudaError_t e;
    // source: the per-pixel queues, or the reconstructor queue (section 5.2);
    // moved by screen motion, or rendered by a camera (hit points)
    const bool fifo = c->fifo_n > 0, cam = camp != nullptr;
    const Camera cm = cam ? *camp : Camera{};
    const size_t nsrc = fifo ? c->fifo_n : c->nslots;
    const uint32_t *state = fifo ? c->q_total : c->r_state;
    const float4 *xm = fifo ? c->q_xm : c->r_xm;
    const float *tt = fifo ? c->q_t : c->r_t;
    const uint32_t *sq = fifo ? c->q_seq : c->r_seq;
    const void *col = fifo ? c->q_col : c->r_col;
    const float4 *wp = fifo ? c->q_world : c->r_world;
    const int g = grid_for(nsrc, 256);
    const uint32_t ns = (uint32_t)nsrc;
    const int bshift = (c->b & (c->b - 1)) == 0 ? __builtin_ctz((unsigned)c->b) : -1;
    const DebugCheck dc{(uint32_t)c->frame_cap, c->derr};
#define AFR_COUNT(F_, C_)                                                                                    \
    k_count<F_, C_><<<g, 256, 0, s>>>(ns, c->b, bshift, c->W, c->H, t_now, cm, wp, state, xm, tt, c->fcnt, \
                                      c->sbin, c->dcount)
    if (fifo && cam) AFR_COUNT(true, true);
    else if (fifo) AFR_COUNT(true, false);
    else if (cam) AFR_COUNT(false, true);
    else AFR_COUNT(false, false);
#undef AFR_COUNT
    // the scan starts the list's append cursors at the bin offsets (a ticket is
    // the entry's place), clears the counts and the bins' smallest ages, and
    // makes the dropped count public
    ScanWith with;
    with.cursor = c->fcur;
    with.clear_in = true;
    with.fill = c->amin2;
    with.fill_value = 0x7f800000u;
    with.counter_from = c->dcount + CNT_DROPPING;
    with.counter_to = c->dcount + CNT_DROPPED;
    with.counter_zero = c->dcount + CNT_UNSORTED;
    if (fifo) {
        with.crowded = c->dcount + CNT_CROWDED;
        with.crowded_from = kCrowded;
    }
    if ((e = scan_exclusive(c->fcnt, c->foff, c->P, c->scan_tmp, s, with)) != cudaSuccess) return e;
    // Not by launch_next: its blocks then start unevenly and leave the lists out
    // of slot order, and placing, which gathers in list order, takes 1.1 ms
    // instead of 0.5 at 1920x1080x16 (3956 -> 4291 us for the step).
    if (fifo) k_list<true><<<g, 256, 0, s>>>(ns, c->sbin, sq, state, c->fcur, c->flist, dc);
    else k_list<false><<<g, 256, 0, s>>>(ns, c->sbin, sq, state, c->fcur, c->flist, dc);
#define AFR_QUEUES(CT_, C_)                                                                                         \
    launch_next(k_place_queues<CT_, C_>, dim3(g), dim3(256), 0, s, c->W, c->H, t_now, cm, wp, xm, tt, col, (uint32_t)c->P, c->foff,    \
                                              reinterpret_cast<const uint2 *>(c->flist), c->fcur, c->amin2, c->frec, \
                                              c->dcount, dc, ns)
#define AFR_FIFO(CT_, C_)                                                                                            \
    launch_next(k_place_fifo<CT_, C_>, dim3(g), dim3(256), 0, s, ns, c->W, c->H, t_now, cm, wp, state, xm, tt, sq, col, c->foff, c->flist, \
                                            c->fcur, c->amin2, c->frec, c->dcount, dc)
#define AFR_REPROJ(CT_)                       \
    do {                                      \
        if (fifo && cam) AFR_FIFO(CT_, true); \
        else if (fifo) AFR_FIFO(CT_, false);  \
        else if (cam) AFR_QUEUES(CT_, true);  \
        else AFR_QUEUES(CT_, false);          \
    } while (0)
    switch (c->ct) {
        case AFR_F32: AFR_REPROJ(AFR_F32); break;
        case AFR_F16: AFR_REPROJ(AFR_F16); break;
        default: AFR_REPROJ(AFR_BF16); break;
    }
#undef AFR_REPROJ
#undef AFR_QUEUES
#undef AFR_FIFO
    return cudaGetLastError();
}

}  // namespace afr
