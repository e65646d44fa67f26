// dd_dose_rows.cuh -- dwell-start dose of whole raster and serpentine scans with a uniform
// dwell, from the scan's own symmetry.
//
// Visit j = iy nx + m (row iy, m-th visit of its row) sees the visit that is q-th of the row
// s rows before its own at lag k = s nx + m - q and at the offset (dx, s), where
//   raster:      dx = m - q;
//   serpentine:  dx = m - q for even s and m - (nx - 1 - q) for odd s (rows alternate in
//                direction, and a pair seen from an odd row is the mirror image of the pair
//                seen from an even one).
// So the pair term depends on (s, m, q) and not on iy, and with
//   R(s, m) = sum over q of the term of (s, m, q)      (q < m only for s = 0)
// the dose is the running sum out[iy nx + m] = pref sum_{s <= iy} R(s, m): nx^2 ny pair terms
// instead of n^2 / 2 with n = nx ny (128 times fewer for 256 x 256).
//
// On a raster the term depends on d = m - q alone at a given s, so that R(s, m) is the sum of the
// window d = m - nx + 1 .. m of 2 nx - 1 terms: 2 n pair terms in all.  The window splits at
// d = 0 into a running sum of the terms d = 0 .. m and one, taken from the far end, of the
// negative d: only sums of positive terms.  dose_raster_kernel: one CTA per s and 256 terms of each
// of the two sums, one half of its threads for each, one lag record and one term per thread, then
// a block scan (compensated in FP32).  It is bound by the latency of a record's serial chain and
// one term.  Device time of a call: 256 x 256 FP32 22 us, against 2.72 ms for the direct sum's
// 2.1e9 terms; 64 x 64 FP64 25 us, against 787 us.  A scan of one row is a raster in either order.
//
// On a serpentine the odd s have no such window; dose_rows_kernel forms R from all nx^2 terms of
// each s, in pieces of qc visits of the source row: one CTA per (s, piece, 32 targets m), lane =
// target, the piece's visits dealt out to the eight warps.  A warp's lanes read consecutive lag
// records, which come through shared memory (a lane stride of 80 bytes: no bank conflicts among
// the eight lanes of a 16-byte phase).  Costliest rows (small s) first.  It is bound by
// instruction issue and the barriers of its stages (FP32: 53 us for 256 x 256, 71 us a call) or
// the FP64 pipe.
//
// dose_rows_scan_kernel adds the pieces and takes the running sum over the rows: a CTA holds 8
// targets and deals the rows out to 32 groups of 8 lanes, each of which sums its rows, then adds
// the sum of the rows before them.  FP32 pieces are summed in compensated FP32 (an FP64 sum of
// them over 32 targets per CTA took 49 us for 256 x 256: each SM adds 1.6 FP64 numbers per
// clock); it is bound by the latency of its loads.
#pragma once
#include <cstdint>

#include "dd_coef.cuh"
#include "dd_field_impl.cuh"

namespace ddk {

constexpr int kDoseRowsWarps = 8;
constexpr int kDoseRowsStage = 64;           // source visits per staging of lag records

template <typename Cfg>
__global__ void __launch_bounds__(32 * kDoseRowsWarps)
dose_rows_kernel(int64_t nx, int64_t n_mt, int64_t n_q, int64_t qc,
                 const typename Cfg::Rec *__restrict__ lagrec, typename Cfg::Real *__restrict__ partial) {
    using Rec = typename Cfg::Rec;
    using Real = typename Cfg::Real;
    constexpr int RV = sizeof(Rec) / 16, ST = kDoseRowsStage, NT = 32 * kDoseRowsWarps;
    __shared__ __align__(16) Rec s_rec[32 + ST];
    __shared__ Real s_sum[kDoseRowsWarps][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t mt = blockIdx.x % n_mt, rest = blockIdx.x / n_mt;
    const int64_t c = rest % n_q, s = rest / n_q;
    const int64_t m0 = mt * 32, m = m0 + lane;
    const bool flip = (s & 1) != 0;          // dx = m - (nx - 1 - q)
    const Real sy = (Real)s, sy2 = sy * sy;
    // the pieces of row s = 0 hold the visits before the target only
    const int64_t q_end = min(min((c + 1) * qc, nx), s == 0 ? m0 + 31 : nx);
    BlockSum<Real> tot;
    for (int64_t q0 = c * qc; q0 < q_end; q0 += ST) {
        const int cnt = (int)min((int64_t)ST, q_end - q0);
        // records of the lags k_lo .. k_hi, at most 31 + cnt of them (a negative lag belongs to
        // pairs that do not exist)
        const int64_t k_lo = s * nx + m0 - (q0 + cnt - 1);
        const int64_t k_hi = s * nx + min(m0 + 32, nx) - 1 - q0;
        __syncthreads();
        {
            const float4 *row = reinterpret_cast<const float4 *>(lagrec);
            float4 *dst = reinterpret_cast<float4 *>(&s_rec[0]);
            const int lim = (int)(k_hi - k_lo + 1) * RV;
            for (int v = tid; v < lim; v += NT)
                dst[v] = k_lo * RV + v >= 0 ? row[k_lo * RV + v] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        Real acc = 0;
        const int dx0 = (int)(flip ? m - (nx - 1 - q0) : m - q0);
        // the visits of this stage that come before the target: q < m on its own row
        const int n_ok = m >= nx ? 0 : s > 0 ? cnt : (int)max((int64_t)0, min((int64_t)cnt, m - q0));
        for (int u = warp; u < cnt; u += kDoseRowsWarps) {
            const bool ok = u < n_ok;
            const Rec &R = s_rec[ok ? lane + cnt - 1 - u : 0];
            const Real dx = (Real)(flip ? dx0 + u : dx0 - u);
            const Real r2 = dx * dx + sy2;
            if constexpr (std::is_same<Real, float>::value) {
                // one series degree per warp, as in dose_lags_f32: degree 2 by one vote, else
                // the largest class of the lanes' own; a pair whose own a is 87 or more (its
                // term below 2e-38) is left out there
                const float dq = R.dq(), h = r2 * dq;
                if (__all_sync(0xffffffffu, !ok || (h <= kL2H && dq >= kMinDqX))) {
                    if (ok) acc += log_term<2>(r2, R);
                    continue;
                }
                const uint32_t own = ok ? series_class(h, r2 * R.q1(), dq) : kCodeSkip;
                const uint32_t cls = __reduce_max_sync(0xffffffffu, own);
                if (cls == kCodeSkip) continue;
                float t;
                if (cls <= kCodeD4) t = log_term<4>(r2, R);
                else if (cls == kCodeD8) t = log_term<8>(r2, R);
                else if (cls == kCodeD12) t = log_term<12>(r2, R);
                else t = own == kCodeSkip ? 0.0f : pair_term(r2, R);
                if (own != kCodeSkip) acc += t;
            } else {
                if (ok) acc += pair_term(r2, R);
            }
        }
        tot.add(acc);
    }
    s_sum[warp][lane] = tot.result();
    __syncthreads();
    if (warp == 0 && m < nx) {
        BlockSum<Real> sum;
#pragma unroll
        for (int w = 0; w < kDoseRowsWarps; ++w) sum.add(s_sum[w][lane]);
        partial[(s * n_q + c) * nx + m] = sum.result();
    }
}

// One pair term on the cheapest series that holds it (each lane has a record of its own).
__device__ __forceinline__ float lone_pair_term(float r2, const RecF32 &R) {
    const uint32_t cls = series_class(r2 * R.dq(), r2 * R.q1(), R.dq());
    return cls == kCodeSkip ? 0.0f : cls == kCodeD2 ? log_term<2>(r2, R) : cls == kCodeD4 ? log_term<4>(r2, R)
         : pair_term(r2, R);
}
__device__ __forceinline__ double lone_pair_term(double r2, const RecF64 &R) { return pair_term(r2, R); }

// Terms d = 0 .. of row offset s (side 0) and -1, -2 .. (side 1; none at s = 0) in chunks of half =
// blockDim.x / 2 threads, one CTA for both sides of a chunk: partial[2 s nx + m] = sum of the chunk's
// terms up to d = m, partial[(2 s + 1) nx + m] = sum of its terms down to d = m - nx + 1.  A row of one
// chunk (nx <= 256) is then complete; dose_raster_base_kernel sums the chunks before each one.  (One
// CTA walking a row's chunks with a carry took 3 us for each: 58 us for 4096 x 1 FP32, the direct sum
// 44, this 21; 8192 x 1: 105, 66, 23; 65,536 x 1: 774, 1465, 57.)
constexpr int kDoseRasterHalf = 256;         // largest half of a CTA
template <typename Cfg, bool kChunks>
__global__ void __launch_bounds__(2 * kDoseRasterHalf)
dose_raster_kernel(int nx, int n_chunks, double s_dim, double kappa, typename Cfg::Real *__restrict__ partial) {
    using Rec = typename Cfg::Rec;
    using Real = typename Cfg::Real;
    __shared__ BlockSum<Real> s_warp[2 * kDoseRasterHalf / 32];
    const int half = blockDim.x / 2, side = threadIdx.x >= half, t = threadIdx.x - side * half;
    const int lane = threadIdx.x & 31, warp0 = side * half / 32, warp = t / 32;
    const int64_t s = kChunks ? blockIdx.x / n_chunks : blockIdx.x;
    Real *const row = partial + (2 * s + side) * (int64_t)nx;
    // one pass (as a loop it compiles to a shorter FP64 chain: 18.9 us against 20.3 for 20 x 20)
    const int first = kChunks ? (int)(blockIdx.x % n_chunks) * half : 0, end = kChunks ? first + 1 : nx;
    for (int i0 = first; i0 < end; i0 += half) {
        const int i = i0 + t, d = side ? -1 - i : i;
        const int64_t k = s * nx + d;        // lag
        BlockSum<Real> v;
        if (i < nx - side && k > 0) {
            double q1, dq, r, ell;
            pair_geometry<RecTraits<Rec>::kFP64Ell>((double)k, 1.0, s_dim, kappa, q1, dq, r, ell);
            Rec R;
            RecTraits<Rec>::fill(R, q1, dq, r, ell);
            const Real dx = (Real)d, dy = (Real)s, r2 = dx * dx + dy * dy;
            v.add(lone_pair_term(r2, R));
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const BlockSum<Real> u = v.shfl_up(o);
            if (lane >= o) v.add(u);
        }
        if (lane == 31) s_warp[warp0 + warp] = v;
        __syncthreads();
        BlockSum<Real> base;
        for (int w = 0; w < warp; ++w) base.add(s_warp[warp0 + w]);
        v.add(base);
        if (i < nx) row[!side ? i : i < nx - 1 ? nx - 2 - i : nx - 1] = side && i == nx - 1 ? (Real)0 : v.result();
        __syncthreads();
    }
}

// Chunk of column m on a side, and the column that holds the chunk's whole sum (side 1 runs from m =
// nx - 2 down; its m = nx - 1, no terms, belongs to chunk 0).
__device__ __forceinline__ int dose_chunk(int m, int nx, int side) {
    return (side ? max(nx - 2 - m, 0) : m) / kDoseRasterHalf;
}
__device__ __forceinline__ int dose_chunk_end(int c, int nx, int side) {
    const int i = (c + 1) * kDoseRasterHalf - 1;
    return side ? nx - 2 - i : i;
}
// base[(2 s + side) n_chunks + c] = sum of the chunks before c.
template <typename Part>
__global__ void __launch_bounds__(128)
dose_raster_base_kernel(const Part *__restrict__ partial, int nx, int n_chunks, int64_t n, Part *__restrict__ base) {
    const int64_t g = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (g >= n) return;
    const int64_t k = g / n_chunks;
    const int c = (int)(g % n_chunks), side = (int)(k & 1);
    BlockSum<Part> sum;
#pragma unroll 8
    for (int e = 0; e < c; ++e) sum.add(partial[k * nx + dose_chunk_end(e, nx, side)]);
    base[g] = sum.result();
}

// out[iy nx + m - j0] = pref * sum over rows s <= iy and pieces of partial (and, on a raster of several
// chunks, of the chunks before m's: base), for the targets j0 <= iy nx + m < j1.
constexpr int kDoseScanCols = 8, kDoseScanGroups = 32;
template <typename Part, bool kBase>
__global__ void __launch_bounds__(kDoseScanCols * kDoseScanGroups)
dose_rows_scan_kernel(const Part *__restrict__ partial, const Part *__restrict__ base, int n_chunks, int64_t nx,
                      int64_t n_rows, int64_t n_q, int64_t j0, int64_t j1, double pref, double *__restrict__ out) {
    __shared__ BlockSum<Part> s_sum[kDoseScanGroups][kDoseScanCols];
    const int col = threadIdx.x % kDoseScanCols, g = threadIdx.x / kDoseScanCols;
    const int64_t m = (int64_t)blockIdx.x * kDoseScanCols + col;
    const bool live = m < nx;
    const int64_t ra = n_rows * g / kDoseScanGroups, rb = n_rows * (g + 1) / kDoseScanGroups;
    const int c0 = kBase && live ? dose_chunk((int)m, (int)nx, 0) : 0, c1 = kBase && live ? dose_chunk((int)m, (int)nx, 1) : 0;
    BlockSum<Part> sum;
    if (live) {
        const Part *p = partial + ra * n_q * nx + m;
#pragma unroll 8
        for (int64_t k = 0; k < (rb - ra) * n_q; ++k) sum.add(p[k * nx]);
        if (kBase) {
            const Part *b = base + ra * 2 * n_chunks;
#pragma unroll 4
            for (int64_t r = 0; r < rb - ra; ++r) {
                sum.add(b[2 * r * n_chunks + c0]);
                sum.add(b[(2 * r + 1) * n_chunks + c1]);
            }
        }
    }
    s_sum[g][col] = sum;
    __syncthreads();
    if (!live) return;
    BlockSum<Part> run;
    for (int k = 0; k < g; ++k) run.add(s_sum[k][col]);
    for (int64_t r = ra; r < rb; ++r) {
        const Part *p = partial + r * n_q * nx + m;
#pragma unroll 4
        for (int64_t k = 0; k < n_q; ++k) run.add(p[k * nx]);
        if (kBase) {
            run.add(base[2 * r * n_chunks + c0]);
            run.add(base[(2 * r + 1) * n_chunks + c1]);
        }
        const int64_t j = r * nx + m;
        if (j >= j0 && j < j1) out[j - j0] = pref * run.value();
    }
}

}  // namespace ddk
