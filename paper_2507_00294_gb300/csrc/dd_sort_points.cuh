// dd_sort_points.cuh -- spatial order of a list of evaluation points for the FP32-mixed tile.
//
// The tile kernel picks one series degree per (warp, visit, snapshot) from the box of the warp's
// 128 points.  Points scattered in the caller's order give every warp a box as large as the
// region, and with it the high degrees or the two-E1 form for visits that most of its points see
// on degree 2.  sort_points_block orders up to kSortPts points of a list along a Morton curve of
// their own bounding box (16 bits; ties keep the caller's order, so the result is deterministic)
// with a bitonic sort, and deals them out so that each warp of a 512-point tile (128 threads x 4
// points, thread t holding the points t + 128 k) holds 128 consecutive ones (in a list's last, partial
// tile, up to four runs of 32); the reduce writes the field back through the permutation.  A warp
// holds 64 keys in registers, so that only the steps across warps (15 of 66) go through shared
// memory and barriers.  It reads the float-float points (an FP64 pass over 4096 points takes one
// SM 10 us).  2048 points per CTA: with 4096 the sort took 28 us of the 50 it saved (one SM's
// shuffles).  33 snapshots of a 2457-visit random scan on 10,007 random points: 284 us in the
// caller's order, 260 us in this one
// (sort 16 us, field kernel 258 to 209 us); a batch of 256 scans on 997 random points each 774
// and 667 us.
//
// A block of points that the caller already gave in compact runs stays as it is: where the boxes of
// the 128 points that each warp of a tile would hold (four runs of 32) have a mean squared diagonal
// of at most the block's own area.  (Sorted runs have an eighth of it.  A row-major list of 128 x 128
// points, half of it: sorted, the tile took as long and the call 3 % longer, 540 us against 525;
// lists in random order, or sorted by one coordinate only, have 2 to 5 times it and gain by the sort.)
#pragma once
#include <cstdint>

#include "dd_field_impl.cuh"

namespace ddk {

constexpr int kSortPts = 2048, kSortThreads = 1024, kSortTile = 512;
constexpr int kSortPer = kSortPts / kSortThreads, kSortWarp = 32 * kSortPer;     // keys per thread, per warp
static_assert(kSortPer == 2 && kSortPts % kSortTile == 0, "two keys per thread, whole tiles");

struct SortSmem {
    uint32_t key[kSortPts];
    float lo[kSortThreads / 32][2], hi[kSortThreads / 32][2];
    float4 box[kSortPts / 32];               // of the runs of 32 points: x from, to, y from, to
};

__device__ __forceinline__ uint32_t spread8(uint32_t v) {
    v = (v | (v << 4)) & 0x0F0Fu;
    v = (v | (v << 2)) & 0x3333u;
    return (v | (v << 1)) & 0x5555u;
}

// Points c0 .. c0 + cnt - 1 (cnt <= kSortPts, c0 a multiple of kSortPts) of the list of n points
// `in`: F[slot] and perm[slot] receive the points and their indices.
__device__ __forceinline__ void sort_points_block(SortSmem &sm, int64_t n, int64_t c0, int cnt,
                                                  const float4 *__restrict__ in, float4 *__restrict__ F,
                                                  int *__restrict__ perm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // this thread's points (and later its keys): kSortWarp warp + 32 e + lane
    float x[kSortPer], y[kSortPer];
    float xl = 3e38f, xh = -3e38f, yl = 3e38f, yh = -3e38f;
#pragma unroll
    for (int e = 0; e < kSortPer; ++e) {
        const int i = kSortWarp * warp + 32 * e + lane;
        x[e] = y[e] = 0.0f;
        float ax = 3e38f, bx = -3e38f, ay = 3e38f, by = -3e38f;
        if (i < cnt) {
            const float4 p = in[c0 + i];
            ax = bx = x[e] = p.x;
            ay = by = y[e] = p.z;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ax = fminf(ax, __shfl_xor_sync(0xffffffffu, ax, o));
            bx = fmaxf(bx, __shfl_xor_sync(0xffffffffu, bx, o));
            ay = fminf(ay, __shfl_xor_sync(0xffffffffu, ay, o));
            by = fmaxf(by, __shfl_xor_sync(0xffffffffu, by, o));
        }
        if (lane == 0) sm.box[kSortPer * warp + e] = make_float4(ax, bx, ay, by);
        xl = fminf(xl, ax); xh = fmaxf(xh, bx);
        yl = fminf(yl, ay); yh = fmaxf(yh, by);
    }
    if (lane == 0) {
        sm.lo[warp][0] = xl; sm.lo[warp][1] = yl;
        sm.hi[warp][0] = xh; sm.hi[warp][1] = yh;
    }
    __syncthreads();
    xl = sm.lo[lane][0]; yl = sm.lo[lane][1];
    xh = sm.hi[lane][0]; yh = sm.hi[lane][1];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        xl = fminf(xl, __shfl_xor_sync(0xffffffffu, xl, o));
        xh = fmaxf(xh, __shfl_xor_sync(0xffffffffu, xh, o));
        yl = fminf(yl, __shfl_xor_sync(0xffffffffu, yl, o));
        yh = fmaxf(yh, __shfl_xor_sync(0xffffffffu, yh, o));
    }
    // the caller's order: warp w of tile T would hold the runs 16 T + w + 4 j (lane = 4 T + w)
    float d2 = 0.0f;
    const int n_warps = 4 * ((cnt + kSortTile - 1) / kSortTile);
    if (lane < n_warps) {
        float4 u = make_float4(3e38f, -3e38f, 3e38f, -3e38f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 q = sm.box[16 * (lane >> 2) + (lane & 3) + 4 * j];
            u = make_float4(fminf(u.x, q.x), fmaxf(u.y, q.y), fminf(u.z, q.z), fmaxf(u.w, q.w));
        }
        if (u.y >= u.x) d2 = (u.y - u.x) * (u.y - u.x) + (u.w - u.z) * (u.w - u.z);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    if (d2 <= (float)n_warps * ((xh - xl) * (yh - yl))) {        // (not where a coordinate is not finite)
#pragma unroll
        for (int e = 0; e < kSortPer; ++e) {
            const int64_t i = c0 + kSortWarp * warp + 32 * e + lane;
            if (i >= c0 + cnt) continue;
            F[i] = in[i];
            perm[i] = (int)i;
        }
        return;
    }
    const float side = fmaxf(xh - xl, yh - yl), inv = side > 0.0f ? 255.999f / side : 0.0f;
    uint32_t v[kSortPer];
#pragma unroll
    for (int e = 0; e < kSortPer; ++e) {
        const int i = kSortWarp * warp + 32 * e + lane;
        // (a coordinate that is not finite takes an arbitrary cell)
        const uint32_t a = min((uint32_t)fmaxf((x[e] - xl) * inv, 0.0f), 255u);
        const uint32_t b = min((uint32_t)fmaxf((y[e] - yl) * inv, 0.0f), 255u);
        v[e] = i < cnt ? ((spread8(a) | (spread8(b) << 1)) << 12) | (uint32_t)i : 0xFFFFFFFFu;
    }
    int size = kSortWarp;
    while (size < cnt) size <<= 1;
    const bool busy = kSortWarp * warp < size;   // the warps past it hold padding only
    for (int k = 2; k <= size; k <<= 1) {
        for (int j = k >> 1; j >= kSortWarp; j >>= 1) {
            __syncthreads();                 // the last step's reads
#pragma unroll
            for (int e = 0; e < kSortPer; ++e) sm.key[kSortWarp * warp + 32 * e + lane] = v[e];
            __syncthreads();
#pragma unroll
            for (int e = 0; e < kSortPer; ++e) {
                const int i = kSortWarp * warp + 32 * e + lane;
                const uint32_t o = sm.key[i ^ j];
                v[e] = ((i & j) == 0) == ((i & k) == 0) ? min(v[e], o) : max(v[e], o);
            }
        }
        for (int j = min(k >> 1, kSortWarp / 2); j > 0 && busy; j >>= 1) {
            uint32_t o[kSortPer];
#pragma unroll
            for (int e = 0; e < kSortPer; ++e)
                o[e] = j == 32 ? v[e ^ 1] : __shfl_xor_sync(0xffffffffu, v[e], j);
#pragma unroll
            for (int e = 0; e < kSortPer; ++e) {
                const int i = kSortWarp * warp + 32 * e + lane;
                v[e] = ((i & j) == 0) == ((i & k) == 0) ? min(v[e], o[e]) : max(v[e], o[e]);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < kSortPer; ++e) {
        const int s = kSortWarp * warp + 32 * e + lane;
        if (s >= cnt) continue;
        const int64_t i = c0 + (v[e] & (kSortPts - 1)), q = c0 + s, tile = q / kSortTile;
        const int r = (int)(q - tile * kSortTile);
        const int64_t slot = (tile + 1) * kSortTile <= n
                                 ? tile * kSortTile + 128 * ((r >> 5) & 3) + 32 * (r >> 7) + (r & 31) : q;
        F[slot] = in[i];
        perm[slot] = (int)i;
    }
}

}  // namespace ddk
