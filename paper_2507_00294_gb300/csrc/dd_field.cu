// dd_field.cu -- cumulative damage field psi(r, t) of Eq. 5 on the GPU.
//
//   psi(r,t) = Q0/(4 pi D) sum_{i : t_i < t} [E1(rho_i^2 / w1) - E1(rho_i^2 / w0)]
//   w1 = 2s + 4 kappa (t - t_i),  w0 = 2s (beam on, Eq. 1) or 2s + 4 kappa (t - t_i - tau_i)
//   (beam off, Eq. 2), in units of the pitch and the reference dwell (dd_internal.h).
//
// Pipeline of one dd_field_at_times call (all on the caller's stream):
//   1. points SI -> pitch units (prep_points_kernel; with the lag table of step 2 in one
//      launch, prep_points_lag_kernel, when the snapshots lie on the dwell lattice);
//   2. per (snapshot, visit) FP64 coefficients: q1 = 1/w1, dq = 1/w0 - 1/w1 and the
//      moment coefficients c_0..c_M of dd_e1.cuh (coef_kernel);
//   3. work items (point tile, snapshot chunk, visit block), sorted by cost, one CTA
//      each (field_kernel): the block's visits are staged in shared memory in visit
//      order, every thread keeps PPT points x TCH snapshots in registers, and each
//      snapshot only sums the visits that have started (causal prefix n_active(t));
//   4. deterministic reduce of the per-block partial sums in block order, times
//      Q0/(4 pi D), into out[snapshot][point] (reduce_kernel).
#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstring>
#include <limits>
#include <numeric>
#include <vector>

#include "dd_coef.cuh"
#include "dd_e1.cuh"
#include "dd_field_grid.cuh"
#include "dd_field_impl.cuh"
#include "dd_grid.h"
#include "dd_internal.h"
#include "dd_sort_points.cuh"

namespace ddk {

// A rectilinear grid of evaluation points: point k = r W + c at (x0 + c dx, y0 + r dy)
// (SI); W = 0 for an explicit point list.
struct GridDesc {
    double x0 = 0, y0 = 0, dx = 0, dy = 0;
    int64_t W = 0, H = 0;
};

// Points in pitch units: FP64 X, Y, and float-float (x_hi, x_lo, y_hi, y_lo) for the FP32
// tile, so that the FP32 kernels form coordinate differences without FP64 arithmetic.
// A grid point is formed in SI as x0 + c dx (one product, one sum, no fused multiply-add:
// the values a caller's point list of the same grid holds).
__device__ __forceinline__ void prep_point(int64_t k, const double *__restrict__ xy, const GridDesc &g, int64_t n,
                                           double inv_p, double *__restrict__ X, double *__restrict__ Y,
                                           float4 *__restrict__ F) {
    if (k >= n) return;
    double xs, ys;
    if (g.W > 0) {
        const int64_t r = k / g.W, c = k - r * g.W;
        xs = __dadd_rn(__dmul_rn((double)c, g.dx), g.x0);
        ys = __dadd_rn(__dmul_rn((double)r, g.dy), g.y0);
    } else {
        xs = xy[2 * k];
        ys = xy[2 * k + 1];
    }
    const double x = xs * inv_p, y = ys * inv_p;
    X[k] = x;
    Y[k] = y;
    const float xh = (float)x, yh = (float)y;
    F[k] = make_float4(xh, (float)(x - (double)xh), yh, (float)(y - (double)yh));
}
__global__ void prep_points_kernel(const double *__restrict__ xy, GridDesc g, int64_t n, double inv_p,
                                   double *__restrict__ X, double *__restrict__ Y, float4 *__restrict__ F) {
    prep_point((int64_t)blockIdx.x * blockDim.x + threadIdx.x, xy, g, n, inv_p, X, Y, F);
}

// A point list in spatial order (dd_sort_points.cuh).
__global__ void __launch_bounds__(kSortThreads)
sort_points_kernel(const float4 *__restrict__ in, int64_t n, float4 *__restrict__ F, int *__restrict__ perm) {
    __shared__ SortSmem sm;
    const int64_t c0 = (int64_t)blockIdx.x * kSortPts;
    sort_points_block(sm, n, c0, (int)min((int64_t)kSortPts, n - c0), in, F, perm);
}

// The reversed lag table (blocks [0, nb_lag), one record per thread: a long serial chain,
// so these blocks go first) and the points in pitch units (the blocks after) in one
// launch: the field's two preparation steps cost one launch instead of two.
template <typename Rec>
__global__ void prep_points_lag_kernel(int nb_lag, int64_t M, double s, double kappa, Rec *__restrict__ rev,
                                       const double *__restrict__ xy, GridDesc g, int64_t n, double inv_p,
                                       double *__restrict__ X, double *__restrict__ Y, float4 *__restrict__ F) {
    if ((int)blockIdx.x < nb_lag)
        rev_lag_record<Rec>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, M, s, kappa, rev);
    else
        prep_point((int64_t)(blockIdx.x - nb_lag) * blockDim.x + threadIdx.x, xy, g, n, inv_p, X, Y, F);
}

// out[row[j]][p] = pref * sum_{k < nblk[j]} partial[(k * n_tg + j) * pstride + p], the visit
// blocks of snapshot j in that order (deterministic); four points per thread, so that each
// load moves 16 bytes or more.  perm (NULL: none): slot p holds the caller's point perm[p].
template <typename Part>
__global__ void reduce_kernel(const Part *__restrict__ partial, const int *__restrict__ nblk_of_snap,
                              const int *__restrict__ row, int n_tg, int64_t n_pts, int64_t pstride, double pref,
                              const int *__restrict__ perm, double *__restrict__ out) {
    const int j = blockIdx.y;
    const int64_t p0 = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (p0 >= n_pts) return;
    const int nb = nblk_of_snap[j];
    BlockSum<Part> acc[4];
#pragma unroll 4
    for (int k = 0; k < nb; ++k) {
        Part v[4];
        load4_cg(partial + ((int64_t)k * n_tg + j) * pstride + p0, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q].add(v[q]);
    }
    if (perm) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (p0 + q < n_pts) out[(int64_t)row[j] * n_pts + perm[p0 + q]] = pref * acc[q].result();
        return;
    }
    double *o = out + (int64_t)row[j] * n_pts + p0;
    if (p0 + 3 < n_pts && (reinterpret_cast<uintptr_t>(o) & 15) == 0) {
        // 32 contiguous bytes per thread: whole lines per warp
        reinterpret_cast<double2 *>(o)[0] = make_double2(pref * acc[0].result(), pref * acc[1].result());
        reinterpret_cast<double2 *>(o)[1] = make_double2(pref * acc[2].result(), pref * acc[3].result());
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (p0 + q < n_pts) o[q] = pref * acc[q].result();
    }
}

}  // namespace ddk

// ============================================================== host dispatcher
namespace {

using ddk::RecF32;
using ddk::RecF64;

struct Carve {
    char *base;
    size_t off = 0;
    explicit Carve(void *b) : base((char *)b) {}
    template <typename T>
    T *take(size_t count) {
        off = (off + 255) & ~size_t(255);
        T *p = (T *)(base + off);
        off += count * sizeof(T);
        return p;
    }
};

// Host-side tables, uploaded through pinned staging blocks; freed (and the blocks given
// back) once an event recorded after the uploads has completed.
struct HostTables {
    std::vector<std::vector<int2>> items;
    std::vector<std::vector<int>> ints;
    std::vector<std::vector<double>> reals;
    std::vector<std::vector<int64_t>> offs;
    std::vector<std::vector<char>> images; // per group: the tables as laid out on the device
    dd::CallStaging staging;               // pinned copies the uploads were made from
    static void release(void *p) { delete static_cast<HostTables *>(p); }
};

// Sizes of the workspace a call needs (the same function drives the carve).
template <typename Cfg>
size_t workspace_bytes(int64_t n_pts, int64_t n_src, int group, int sb, bool out_host, bool pts_host,
                       int n_t, int64_t n_rec, bool sorted) {
    using Rec = typename Cfg::Rec;
    const int nblk_max = (int)((n_src + sb - 1) / sb);
    const int n_chunks = (group + Cfg::kTCH - 1) / Cfg::kTCH;
    size_t b = 0;
    auto add = [&](size_t bytes) { b = ((b + 255) & ~size_t(255)) + bytes; };
    if (pts_host) add(2 * (size_t)n_pts * sizeof(double));
    if (out_host) add((size_t)n_t * n_pts * sizeof(double));
    add(2 * (size_t)n_pts * sizeof(double));                  // X, Y in pitch units
    add((size_t)n_pts * sizeof(float4));                      // the same as float-float
    if (sorted) {                                             // in spatial order, and the caller's indices
        add((size_t)n_pts * sizeof(float4));
        add((size_t)n_pts * sizeof(int));
    }
    add((size_t)group * sizeof(double));                      // snapshot times
    add((size_t)group * sizeof(int) * 3);                     // nact, row, nblk per snapshot
    add((size_t)group * sizeof(int64_t));                     // record row offset per snapshot
    add((size_t)n_chunks * nblk_max * sizeof(int2));          // (chunk, block) descriptors
    add((size_t)n_rec * sizeof(Rec));                         // coefficient records
    add((size_t)nblk_max * group * ((n_pts + 3) / 4 * 4) * sizeof(typename Cfg::Real));   // partial sums
    return b + 256;
}

// Shared-memory carveout of the tile kernels (Cfg::kCarveout, percent of the L1/shared
// array), set once per device: the FP32-mixed tile's 8 CTAs of 13 KB fit in 132 KB and
// the rest stays L1 for the minority classes' record reads (about 1 % faster than the
// whole array as shared memory); the FP64 tile takes the whole array.
// The grid tile (dd_field_grid.cuh): 128 columns x GridCfg::kPPT = 4 rows (a tile of 8 rows
// per thread, 80 registers and 6 CTAs per SM, measured 8 % slower).  Its row tables sit
// beside the general tile's 12 KB: 8 CTAs of 17.3 KB (with the per-CTA reserve) need a 66 %
// carveout.
using GridCfg = ddk::CfgMixed;
constexpr int kGridCarveout = 66;

template <typename Cfg, bool kGrid>
struct TileKernel {
    static constexpr auto fn() { return ddk::field_kernel<Cfg>; }
    static constexpr int carveout = Cfg::kCarveout;
};
template <>
struct TileKernel<ddk::CfgMixed, true> {
    static constexpr auto fn() { return ddk::field_grid_kernel<GridCfg>; }
    static constexpr int carveout = kGridCarveout;
};

template <typename Cfg, bool kGrid = false>
cudaError_t prefer_shared() {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess || dev >= 64) return err;
    if (done.load() & (uint64_t(1) << dev)) return cudaSuccess;
    err = cudaFuncSetAttribute(TileKernel<Cfg, kGrid>::fn(), cudaFuncAttributePreferredSharedMemoryCarveout,
                               TileKernel<Cfg, kGrid>::carveout);
    if (err == cudaSuccess) done.fetch_or(uint64_t(1) << dev);
    return err;
}

// CTAs of the tile kernel resident on the whole device at once (0 if unknown).
template <typename Cfg, bool kGrid = false>
int64_t resident_ctas() {
    static std::atomic<int64_t> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return 0;
    int64_t v = cached[dev].load();
    if (v > 0) return v;
    if (prefer_shared<Cfg, kGrid>() != cudaSuccess) cudaGetLastError();   // occupancy at the carveout used
    int per_sm = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, TileKernel<Cfg, kGrid>::fn(), Cfg::kThreads, 0) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    v = (int64_t)per_sm * sms;
    cached[dev].store(v);
    return v;
}

// ---- the prefixes that dd_field_grid_split reports
//
// A visit is on the degree-2 (degree-4) series at every point of the grid when
// h = rho^2 dq <= kL2H (kL4H) for rho^2 up to R2, the largest squared distance between the
// grid's box and the box of the visits.  With c = 4 kappa tau_max, dq = 1/w0 - 1/w1 <=
// c / ((w1 - c) w1) for every visit of the scan (dq grows with the dwell at a fixed
// w1 = 2s + 4 kappa (t - T_i)), so every visit with w1 at or above the root w1* of
// (w1 - c) w1 = c R2 / h_limit (and its dwell over) qualifies: the prefix of the visits that
// started by t_j - dT*, dT* = (w1* - 2s) / (4 kappa), found by bisection of the start times.
// (The degree-4 band only while its records' coefficients of rho^8 stay in the FP32 normal
// range, dq >= kMinDqX.)  All of them are among the visits that the contraction of dd_grid.cu
// takes, whose bands reach h = 218.
constexpr int64_t kSplitMinSide = 64;

struct TcPlan {
    bool on = false;
    std::vector<int> K2;         // per snapshot (time order): the degree-2 visits [0, K2)
    std::vector<int> K;          // and the degree-4 band [K2, K)
};

// Age (in dwells) from which every visit of the scan is on the series of the given h limit
// at every point within R2, or a negative value if none is.
double tc_min_age(const dd_scan *scan, double R2, double h_limit, double *w1s_out) {
    const double dq_max = h_limit * (1.0 - 1e-4) / R2;
    const double c = 4.0 * scan->kappa * scan->tau_max;
    if (!(c > 0.0) || !(dq_max > 0.0) || !std::isfinite(dq_max)) return -1.0;
    double w1s = 0.5 * (c + std::sqrt(c * c + 4.0 * c / dq_max));
    w1s = std::max(w1s, (2.0 * scan->s + c) * (1.0 + 1e-9));        // the dwell is over
    if (w1s_out) *w1s_out = w1s;
    return (w1s - 2.0 * scan->s) / (4.0 * scan->kappa) * (1.0 + 1e-9);
}

TcPlan plan_tc(const dd_scan *scan, const ddk::GridDesc &grid, const std::vector<double> &tdim,
               const std::vector<int> &nact) {
    TcPlan tp;
    const int n_t = (int)tdim.size();
    tp.K2.assign(n_t, 0);
    tp.K.assign(n_t, 0);
    if (grid.W < kSplitMinSide || grid.H < kSplitMinSide || scan->n == 0) return tp;
    const double ip = 1.0 / scan->pitch;
    const double xa = grid.x0 * ip, xb = (grid.x0 + (double)(grid.W - 1) * grid.dx) * ip;
    const double ya = grid.y0 * ip, yb = (grid.y0 + (double)(grid.H - 1) * grid.dy) * ip;
    const double ex = std::max(std::max(xa, xb) - scan->x_lo, scan->x_hi - std::min(xa, xb));
    const double ey = std::max(std::max(ya, yb) - scan->y_lo, scan->y_hi - std::min(ya, yb));
    // margins for the points' own rounding and the records' rounding to FP32
    const double R2 = (ex * ex + ey * ey) * (1.0 + 1e-6) + 1e-6;
    double w1s2 = 0.0;
    const double age2 = tc_min_age(scan, R2, (double)ddk::kL2H, &w1s2);
    if (age2 < 0.0) return tp;
    double age4 = tc_min_age(scan, R2, (double)ddk::kL4H, nullptr);
    // the degree-4 band's smallest dq: its oldest visit (w1 up to w1s2) with the shortest dwell
    const double cmin = 4.0 * scan->kappa * scan->tau_min;
    if (age4 < 0.0 || !(w1s2 > cmin) || cmin / ((w1s2 - cmin) * w1s2) < 2.0 * (double)ddk::kMinDqX) age4 = age2;
    int64_t any = 0;
    for (int k = 0; k < n_t; ++k) {
        const int64_t k2 = std::upper_bound(scan->T.begin(), scan->T.end(), tdim[k] - age2) - scan->T.begin();
        const int64_t k4 = std::upper_bound(scan->T.begin(), scan->T.end(), tdim[k] - std::min(age4, age2)) - scan->T.begin();
        tp.K2[k] = (int)std::min<int64_t>(k2, nact[k]);
        tp.K[k] = (int)std::max<int64_t>(tp.K2[k], std::min<int64_t>(k4, nact[k]));
        any += tp.K[k];
    }
    if (any == 0) return tp;
    tp.on = true;
    return tp;
}

// The contraction's second launch runs on a side stream of the calling thread, forked from the
// caller's stream after the coefficients and joined back before the final kernel, so that its
// CTAs start as the first launch's leave their SMs.  One stream and two events per
// (thread, device), created on first use (reusing an event is safe: a wait takes the state
// of the event's latest record when it is issued).
struct SideStream {
    cudaStream_t s = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
};
cudaError_t side_stream(SideStream **out) {
    thread_local SideStream per_dev[64];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev >= 64) return cudaErrorInvalidDevice;
    SideStream &ss = per_dev[dev];
    if (!ss.s) {
        int lo = 0, hi = 0;
        if ((err = cudaDeviceGetStreamPriorityRange(&lo, &hi)) != cudaSuccess) return err;
        if ((err = cudaStreamCreateWithPriority(&ss.s, cudaStreamNonBlocking, lo)) != cudaSuccess)
            return err;
        if ((err = cudaEventCreateWithFlags(&ss.fork, cudaEventDisableTiming)) != cudaSuccess) return err;
        if ((err = cudaEventCreateWithFlags(&ss.join, cudaEventDisableTiming)) != cudaSuccess) return err;
    }
    *out = &ss;
    return cudaSuccess;
}

// Snapshots in time order: order[k] = index into times of the k-th earliest, tdim[k] its time
// in dwells and nact[k] = #{i : T_i < t} (the visits started by then).  Returns true for
// snapshots on the dwell lattice of a uniform scan (t = integer number of dwells, to within
// 2 ulp of the quotient -- the rounding t/dwell itself already carries; tdim is then rounded
// to those integers and M is the last): the record of (snapshot, visit) then depends on the
// lag only, so one reversed lag table of M + 1 records serves every snapshot.
bool snapshot_dims(const dd_scan *scan, const std::vector<double> &times, std::vector<int> &order,
                   std::vector<double> &tdim, std::vector<int> &nact, int64_t &M) {
    const int n_t = (int)times.size();
    const int64_t n_src = scan->n;
    order.resize(n_t);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return times[a] < times[b]; });
    tdim.resize(n_t);
    nact.resize(n_t);
    for (int k = 0; k < n_t; ++k) tdim[k] = times[order[k]] / scan->dwell;
    bool lattice = scan->uniform;
    M = 0;
    for (int k = 0; k < n_t && lattice; ++k) {
        const double r = std::nearbyint(tdim[k]);
        if (std::fabs(tdim[k] - r) > 2.0 * std::numeric_limits<double>::epsilon() * std::fabs(r)) lattice = false;
        else if (r > (double)M) M = (int64_t)r;
    }
    if (M < 1 || M > 4 * n_src + 64) lattice = false;
    if (lattice)
        for (int k = 0; k < n_t; ++k) tdim[k] = std::nearbyint(tdim[k]);
    for (int k = 0; k < n_t; ++k)
        nact[k] = (int)(std::lower_bound(scan->T.begin(), scan->T.end(), tdim[k]) - scan->T.begin());
    return lattice;
}

// pts_xy_m == NULL: the points are the grid `grid` (row-major, n_pts = W H), formed on
// the device; the FP32-mixed path then runs the grid tile kernel.
template <typename Cfg>
dd_status run_field(const dd_scan *scan, const double *pts_xy_m, int64_t n_pts, const ddk::GridDesc &grid,
                    const std::vector<double> &times, double *out, cudaStream_t stream) {
    using Rec = typename Cfg::Rec;
    constexpr bool kMixed = std::is_same<typename Cfg::Real, float>::value;
    const bool on_grid = grid.W > 0;
    const bool grid_tiles = kMixed && on_grid;
    const int64_t n_src = scan->n;
    const int n_t = (int)times.size();
    const dd::MemKind pts_kind = on_grid ? dd::MemKind::Device : dd::memory_kind(pts_xy_m);
    const dd::MemKind out_kind = dd::memory_kind(out);
    const bool pts_host = pts_kind != dd::MemKind::Device;
    const bool out_host = out_kind != dd::MemKind::Device;
    // host buffers go through a workspace copy (a pinned output written in place by the
    // reduce measured slower than the copy engine's transfer)
    const bool pts_copy = pts_host, out_copy = out_host;

    std::vector<int> order, nact;
    std::vector<double> tdim;
    int64_t M = 0;
    const bool lattice = snapshot_dims(scan, times, order, tdim, nact, M);
    // visit block size and snapshot groups bound the partial and record buffers
    const int tile = Cfg::kThreads * Cfg::kPPT;
    // grid tiles: 128 columns x 4 rows (kThreads x kPPT); otherwise 512 consecutive points
    const int64_t n_tc = grid_tiles ? (grid.W + Cfg::kThreads - 1) / Cfg::kThreads : 0;
    const int64_t n_tiles = grid_tiles ? n_tc * ((grid.H + GridCfg::kPPT - 1) / GridCfg::kPPT)
                                       : (n_pts + tile - 1) / tile;
    int sb = Cfg::kSB;
    int group = n_t;
    const size_t budget = size_t(1) << 30;
    while (group > Cfg::kTCH &&
           (size_t)(lattice ? 0 : group * n_src) * sizeof(Rec) + (size_t)((n_src + sb - 1) / sb) * group * ((n_pts + 3) / 4 * 4) * sizeof(typename Cfg::Real) > budget)
        group = std::max(Cfg::kTCH, group / 2);
    // larger blocks only while the FP32 stage sums stay short (<= 32 stages)
    while ((size_t)((n_src + sb - 1) / sb) * group * ((n_pts + 3) / 4 * 4) * sizeof(typename Cfg::Real) > budget && sb < 32 * Cfg::kSTILE) sb *= 2;
    // smaller blocks (down to 128 visits, 64 for grid tiles) while one launch has fewer than
    // 4 waves of resident CTAs, so that the last wave's stragglers cost little
    {
        constexpr int kWaves = 4;
        const int64_t waves4 = kWaves * (grid_tiles ? resident_ctas<Cfg, true>() : resident_ctas<Cfg>());
        const int n_groups = (n_t + group - 1) / group;
        auto items_per_launch = [&](int b) {
            int64_t blocks = 0;
            for (int j0 = 0; j0 < n_t; j0 += Cfg::kTCH) {
                int cmax = 0;
                for (int j = j0; j < std::min(n_t, j0 + Cfg::kTCH); ++j) cmax = std::max(cmax, nact[j]);
                blocks += (cmax + b - 1) / b;
            }
            return blocks * n_tiles / std::max(1, n_groups);
        };
        const int sb_min = grid_tiles ? 64 : 128;
        auto fits = [&](int b) {
            return (size_t)((n_src + b - 1) / b) * group * ((n_pts + 3) / 4 * 4) * sizeof(typename Cfg::Real) <= budget;
        };
        while (sb > sb_min && waves4 > 0 && items_per_launch(sb) < waves4 && fits(sb / 2)) sb /= 2;
        // and down to one stage while the launch leaves a quarter of the resident CTAs' places
        // empty: the call then takes as long as one CTA's visits.  128 or 64 visits against
        // this, in us: FP64, 593 points, 4 snapshots of 308 visits 2288, 665; mixed, 1290 points, 5 of
        // 816: 76, 55; 2000 points, 40 of 2458: 205, 144; 32 x 32 points, 16 of 576: 81, 56.
        // Above the line it depends: 1000 of 1216 places, 10,007 points 168, 182, 2000 points 228, 196.
        while (sb > Cfg::kSTILE && 16 * items_per_launch(sb) < 3 * waves4 && fits(sb / 2)) sb /= 2;
    }
    const int nblk_max = (int)((n_src + sb - 1) / sb);
    const int n_chunks_max = (group + Cfg::kTCH - 1) / Cfg::kTCH;
    // a point list in spatial order (FP32-mixed; FP64 keeps the caller's order, whose degrees
    // are those of the same points as a grid).  Measured at 4.0e8 pairs: 49 us less in the tile,
    // 16 us of sorting, 8 us of its launch and the scattered reduce; so from 2e8 pairs on
    int64_t pairs = 0;
    for (int a : nact) pairs += a;
    const bool sorted = kMixed && !on_grid && n_pts >= 256 && n_pts < (int64_t(1) << 31) - ddk::kSortPts &&
                        (double)pairs * (double)n_pts >= 2e8;
    const int64_t n_rec = lattice ? M + 1 : (int64_t)group * n_src;
    const size_t ws_bytes = workspace_bytes<Cfg>(n_pts, n_src, group, sb, out_copy, pts_copy, n_t, n_rec, sorted);
    dd_status st = DD_OK;
    const double *src = dd::device_sources(scan, stream, &st);
    if (!src) return st;
    const dd::ScanUse use{scan, stream};
    const float4 *srcF = dd::device_sources_ff(scan, stream, &st);
    void *ws = nullptr;
    cudaError_t err = dd::fault_injected("alloc") ? cudaErrorMemoryAllocation
                                                  : dd::workspace_alloc(&ws, ws_bytes, stream);
    if (err != cudaSuccess) {
        cudaGetLastError();
        return dd::fail(err == cudaErrorMemoryAllocation ? DD_ENOMEM : DD_ECUDA,
                        std::string("field workspace allocation: ") + cudaGetErrorString(err));
    }
    Carve cv(ws);
    const double *pts_dev = pts_xy_m;
    if (pts_copy) {
        double *p = cv.take<double>(2 * (size_t)n_pts);
        DD_CUDA_TRY(cudaMemcpyAsync(p, pts_xy_m, 2 * (size_t)n_pts * sizeof(double), cudaMemcpyHostToDevice, stream));
        pts_dev = p;
    }
    double *out_dev = out_copy ? cv.take<double>((size_t)n_t * n_pts) : out;
    double *X = cv.take<double>(2 * (size_t)n_pts);
    double *Y = X + n_pts;
    float4 *PF = cv.take<float4>((size_t)n_pts);
    float4 *const PF0 = PF;
    int *d_perm = nullptr;
    if (sorted) {
        PF = cv.take<float4>((size_t)n_pts);
        d_perm = cv.take<int>((size_t)n_pts);
    }
    double *d_t = cv.take<double>(group);
    int *d_nact = cv.take<int>(3 * (size_t)group);
    int *d_row = d_nact + group;
    int *d_nblk = d_row + group;
    int64_t *d_roff = cv.take<int64_t>(group);
    int2 *d_desc = cv.take<int2>((size_t)n_chunks_max * nblk_max);
    Rec *d_rec = cv.take<Rec>((size_t)n_rec);
    using Part = typename Cfg::Real;
    const int64_t pstride = (n_pts + 3) / 4 * 4;            // 16-byte aligned partial rows
    Part *d_part = cv.take<Part>((size_t)nblk_max * group * pstride);

    if (!lattice) {
        DD_PROFILED("prep_points", stream,
                    (ddk::prep_points_kernel<<<(unsigned)((n_pts + 255) / 256), 256, 0, stream>>>(pts_dev, grid, n_pts, 1.0 / scan->pitch, X, Y, PF0)));
        DD_CUDA_TRY(cudaGetLastError());
    }

    const double *srcX = src, *srcY = src + n_src, *srcT = src + 2 * n_src, *srcTAU = src + 3 * n_src;
    // host staging for the per-group tables, released by a host callback once the
    // stream has consumed them (the copies below may read pageable memory late)
    HostTables *keep = new HostTables();
    if (lattice) {
        // the lag table and the points in one launch of 32-thread blocks
        const int nb_lag = (int)((M + 1 + 31) / 32);
        const int64_t nb_pts = (n_pts + 31) / 32;
        DD_PROFILED(Cfg::kCoefName, stream,
                    (ddk::prep_points_lag_kernel<Rec><<<(unsigned)(nb_lag + nb_pts), 32, 0, stream>>>(
                        nb_lag, M, scan->s, scan->kappa, d_rec, pts_dev, grid, n_pts, 1.0 / scan->pitch, X, Y, PF0)));
        DD_CUDA_TRY(cudaGetLastError());
    }
    if (sorted) {
        DD_PROFILED("sort_points", stream,
                    (ddk::sort_points_kernel<<<(unsigned)((n_pts + ddk::kSortPts - 1) / ddk::kSortPts), ddk::kSortThreads, 0, stream>>>(
                        PF0, n_pts, PF, d_perm)));
        DD_CUDA_TRY(cudaGetLastError());
    }
    for (int g0 = 0; g0 < n_t; g0 += group) {
        const int ng = std::min(group, n_t - g0);
        const int n_chunks = (ng + Cfg::kTCH - 1) / Cfg::kTCH;
        std::vector<int> tabs(3 * (size_t)ng);
        std::vector<double> tg(ng);
        std::vector<int64_t> roff(ng);
        int max_nact = 0;
        for (int j = 0; j < ng; ++j) {
            tg[j] = tdim[g0 + j];
            tabs[j] = nact[g0 + j];
            tabs[ng + j] = order[g0 + j];
            max_nact = std::max(max_nact, nact[g0 + j]);
            // lattice: snapshot t reads lag t - i at rev[M - t + i]; otherwise row j of the
            // per-(snapshot, visit) records
            roff[j] = lattice ? (tdim[g0 + j] > 0 ? M - (int64_t)tdim[g0 + j] : M) : (int64_t)j * n_src;
        }
        // work items: (tile, chunk, block) for every block below the chunk's largest
        // n_active, longest first.  Every tile of a (chunk, block) costs the
        // same, so the (chunk, block) descriptors are sorted (stable: ties keep chunk, block
        // order) and the kernel expands each into its tiles in tile order.
        std::vector<std::pair<int64_t, int2>> blocks;
        for (int c = 0; c < n_chunks; ++c) {
            const int j0 = c * Cfg::kTCH, j1 = std::min(ng, j0 + Cfg::kTCH);
            int cmax = 0;
            for (int j = j0; j < j1; ++j) cmax = std::max(cmax, nact[g0 + j]);
            const int nb = (cmax + sb - 1) / sb;
            for (int j = j0; j < j1; ++j) tabs[2 * ng + j] = nb;
            for (int k = 0; k < nb; ++k) {
                int64_t cost = 0;
                for (int j = j0; j < j1; ++j) cost += std::max(0, std::min(nact[g0 + j], (k + 1) * sb) - k * sb);
                blocks.push_back({cost, make_int2(c, k)});
            }
        }
        std::stable_sort(blocks.begin(), blocks.end(),
                         [](const std::pair<int64_t, int2> &a, const std::pair<int64_t, int2> &b) { return a.first > b.first; });
        std::vector<int2> it(blocks.size());
        for (size_t q = 0; q < blocks.size(); ++q) it[q] = blocks[q].second;

        // the group's tables in one copy: a host image of the device span d_t .. the end of
        // the descriptors
        {
            char *const d0 = reinterpret_cast<char *>(d_t);
            const size_t span = reinterpret_cast<char *>(d_desc + it.size()) - d0;
            std::vector<char> img(span);
            std::memcpy(img.data(), tg.data(), ng * sizeof(double));
            std::memcpy(img.data() + (reinterpret_cast<char *>(d_nact) - d0), tabs.data(), 3 * (size_t)ng * sizeof(int));
            std::memcpy(img.data() + (reinterpret_cast<char *>(d_roff) - d0), roff.data(), ng * sizeof(int64_t));
            std::memcpy(img.data() + (reinterpret_cast<char *>(d_desc) - d0), it.data(), it.size() * sizeof(int2));
            DD_CUDA_TRY(keep->staging.upload(d0, img.data(), span, stream));
            keep->images.push_back(std::move(img));
        }
        if (max_nact > 0 && !lattice) {
            dim3 cg((unsigned)((max_nact + 127) / 128), (unsigned)ng);
            DD_PROFILED(Cfg::kCoefName, stream,
                        (ddk::coef_kernel<Rec><<<cg, 128, 0, stream>>>(srcT, srcTAU, d_t, d_nact, scan->s, scan->kappa, d_rec, n_src)));
            DD_CUDA_TRY(cudaGetLastError());
        }
        if (!it.empty()) {
            if (grid_tiles) DD_CUDA_TRY((prefer_shared<Cfg, true>()));
            else DD_CUDA_TRY(prefer_shared<Cfg>());
            // one CTA per item, in launches of at most 2^31 - 1 CTAs (the grid's x limit)
            const int64_t n_items = (int64_t)it.size() * n_tiles, kMaxGrid = (int64_t(1) << 31) - 1;
            for (int64_t item0 = 0; item0 < n_items; item0 += kMaxGrid) {
                const unsigned nctas = (unsigned)std::min(kMaxGrid, n_items - item0);
                if constexpr (kMixed) {
                    if (grid_tiles) {
                        DD_PROFILED("field_grid_mixed", stream,
                                    (ddk::field_grid_kernel<GridCfg><<<nctas, Cfg::kThreads, 0, stream>>>(
                                        grid.W, grid.H, n_tc, d_rec, d_roff, d_nact, d_desc,
                                        n_tiles, item0, ng, sb, d_part, pstride, srcF, PF)));
                        DD_CUDA_TRY(cudaGetLastError());
                        continue;
                    }
                }
                DD_PROFILED(Cfg::kFieldName, stream,
                            (ddk::field_kernel<Cfg><<<nctas, Cfg::kThreads, 0, stream>>>(
                                srcX, srcY, X, Y, n_pts, d_rec, d_roff, d_nact, d_desc, n_tiles, item0, ng, sb, d_part,
                                pstride, srcF, PF)));
                DD_CUDA_TRY(cudaGetLastError());
            }
        }
        dim3 rg((unsigned)((n_pts + 1023) / 1024), (unsigned)ng);
        DD_PROFILED("field_reduce", stream,
                    (ddk::reduce_kernel<Part><<<rg, 256, 0, stream>>>(
                        d_part, d_nblk, d_row, ng, n_pts, pstride, scan->pref, d_perm, out_dev)));
        DD_CUDA_TRY(cudaGetLastError());
        keep->items.push_back(std::move(it));
        keep->ints.push_back(std::move(tabs));
        keep->reals.push_back(std::move(tg));
        keep->offs.push_back(std::move(roff));
    }
    if (out_copy)
        DD_CUDA_TRY(cudaMemcpyAsync(out, out_dev, (size_t)n_t * n_pts * sizeof(double), cudaMemcpyDeviceToHost, stream));
    DD_CUDA_TRY(dd::workspace_release(ws, stream));
    DD_CUDA_TRY(dd::defer_release(stream, keep, HostTables::release));
    if (dd::host_sync_needed(stream, {pts_kind, out_kind})) DD_CUDA_TRY(cudaStreamSynchronize(stream));
    return DD_OK;
}

// FP32-mixed grids of at least this many columns, rows and points take the contraction
// (dd_grid.cu); smaller ones leave most of its tiles empty.
constexpr int64_t kQuadMinSide = 32, kQuadMinPts = 4096;

// ... unless the contraction would leave most of the pairs to the CUDA cores, more than this many
// visits per snapshot (grids far wider than the diffusion of a visit): its kernel for those takes 1.2
// to 1.5 times as long per pair as the grid tile, which shares a factor among snapshots.  4096 visits
// in a line, D = 1e-16, 8 snapshots on 512 x 64 points: 339 us by it, 238 by the tile; 65,536 visits, D =
// 6e-16, 128 x 64 points: 2172, 1932.
constexpr double kQuadRecentVisits = 256.0;

// Narrow grids (below 64 columns, half of the CUDA-core grid tile's 128, whose lanes mostly idle
// there) take the final kernel of dd_grid.cu with every visit left to it, a CTA per 32 columns x 16 rows
// and snapshot: where there are many snapshots of few visits.  The grid tile splits a snapshot's visits
// over CTAs, which is faster for few snapshots, and it pays for idle lanes in each group of four.
// Tile against walk in us, 16 x 16, 32 x 32 and 48 x 48 points: 144 visits, 32 snapshots 63, 44; 64, 52; 58, 44; 256
// visits, 16 58, 68; 58, 58; 56, 60; 32 62, 60 (all three); 400 visits, 64 72, 83; 79, 83; 84, 89; 128 83, 85; 102, 85;
// 124, 101; 1024 visits, 64 79, 93; 117, 95; 134, 126; 128 124, 97; 168, 117; 187, 179; 1600 visits of 48 x 48 points,
// 256 snapshots 379, 414.
bool narrow_grid(const ddk::GridDesc &g, int64_t n_t, int64_t n_visits) {
    return g.W < 64 && g.H < dd::kGridMaxSide && n_visits <= 1024 && n_t >= (n_visits <= 256 ? 32 : 128);
}

// Snapshots (indices k0 .. k1 - 1 in time order) of a whole raster on the dwell lattice that share
// their sums by a shift of scan rows (dd_grid_quad.cuh), grouped by phase, where that leaves at most
// half of the pairs and takes at most twice the partial rows; the rest is returned in `rest`.  rows:
// grid rows per pitch.  The grid covers the scan, so that every visit passes the same grid points
// closely in each snapshot: a tile of the tall grid then holds no terms that are large only where
// this snapshot does not look (the contraction's factors are relative to the tile's largest).
struct ShiftGroups {
    std::vector<std::vector<int>> groups;
    std::vector<int> rest;
    int rows = 0;
    int64_t H_ext = 0;
};
ShiftGroups shift_groups(const dd_scan *scan, const ddk::GridDesc &grid, const std::vector<double> &tdim, bool lattice,
                         int k0, int k1) {
    ShiftGroups out;
    out.H_ext = grid.H;
    const double per = grid.dy > 0.0 ? std::nearbyint(scan->pitch / grid.dy) : 0.0;
    const double xe = grid.x0 + (double)(grid.W - 1) * grid.dx, tol = 1e-9 * scan->pitch;
    const bool covers = std::min(grid.x0, xe) <= tol && std::max(grid.x0, xe) >= (scan->nx - 1) * scan->pitch - tol &&
                        grid.y0 <= tol && grid.y0 + (double)(grid.H - 1) * grid.dy >= (scan->ny - 1) * scan->pitch - tol;
    // (a row further down then lies where the scan's next row shifts it, to 1e-12 pitch over the
    // largest scan)
    const bool fits = lattice && covers && scan->order == DD_RASTER && scan->n == (int64_t)scan->nx * scan->ny &&
                      per >= 1.0 && per <= 64.0 && std::fabs(per * grid.dy - scan->pitch) * scan->ny <= 1e-12 * scan->pitch;
    std::vector<std::pair<int64_t, int>> by_phase;       // (phase, index), whole dwells inside the scan
    for (int k = k0; k < k1; ++k) {
        if (fits && tdim[k] >= 1.0 && tdim[k] <= (double)scan->n) by_phase.push_back({(int64_t)tdim[k] % scan->nx, k});
        else out.rest.push_back(k);
    }
    std::sort(by_phase.begin(), by_phase.end());
    for (size_t a = 0; a < by_phase.size();) {
        size_t b = a;
        std::vector<int> g;
        double direct = 0.0, shifted = 0.0, rows_shifted = 0.0;       // pairs / W, partial rows
        for (; b < by_phase.size() && by_phase[b].first == by_phase[a].first; ++b) {
            const int k = by_phase[b].second;
            // (a snapshot given twice is its own sum)
            if (!g.empty() && tdim[k] == tdim[g.back()]) out.rest.push_back(k);
            else g.push_back(k);
        }
        const int64_t last = (int64_t)tdim[g.back()], h_ext = grid.H + (int64_t)per * ((last - (int64_t)tdim[g[0]]) / scan->nx);
        double before = 0.0;
        for (int k : g) {
            const double H = (double)(grid.H + (int64_t)per * ((last - (int64_t)tdim[k]) / scan->nx));
            direct += tdim[k] * (double)grid.H;
            shifted += (tdim[k] - before) * H;
            rows_shifted += H;
            before = tdim[k];
        }
        if (shifted <= 0.5 * direct && rows_shifted <= 2.0 * (double)(g.size() * grid.H) && h_ext < dd::kGridMaxSide) {
            out.rows = (int)per;
            out.H_ext = std::max(out.H_ext, h_ext);
            out.groups.push_back(std::move(g));
        } else {
            out.rest.insert(out.rest.end(), g.begin(), g.end());
        }
        a = b;
    }
    return out;
}

dd_status run_grid_mixed(const dd_scan *scan, const ddk::GridDesc &grid, const std::vector<double> &times, bool contract,
                         double *out, cudaStream_t stream) {
    const int n_t = (int)times.size();
    const int64_t n_pts = grid.W * grid.H;
    const dd::MemKind out_kind = dd::memory_kind(out);
    const bool out_copy = out_kind != dd::MemKind::Device;
    std::vector<int> order, nact;
    std::vector<double> tdim;
    int64_t M = 0;
    const bool lattice = snapshot_dims(scan, times, order, tdim, nact, M);
    const dd::GridBox box{grid.x0, grid.y0, grid.dx, grid.dy, grid.W, grid.H};
    double all = 0.0;
    for (int n : nact) all += (double)n;
    std::vector<int> recents;                    // left to the CUDA cores, where there can be many
    if (contract && all > kQuadRecentVisits * n_t) {
        const double age = dd::GridEngine::banded_age(scan, box);
        double recent = 0.0;
        recents.resize((size_t)n_t);
        for (int k = 0; k < n_t; ++k) {
            recents[k] = lattice ? (int)std::min((double)nact[k], std::ceil(age))
                                 : nact[k] - (int)std::min<int64_t>(nact[k], std::upper_bound(scan->T.begin(), scan->T.end(), tdim[k] - age) - scan->T.begin());
            recent += recents[k];
        }
        if (recent > kQuadRecentVisits * n_t && recent > 0.5 * all && shift_groups(scan, grid, tdim, lattice, 0, n_t).groups.empty())
            return run_field<ddk::CfgMixed>(scan, nullptr, n_pts, grid, times, out, stream);
    }
    // snapshots of a pass: their tables (off the lattice; on it one serves them all), about four
    // partial rows each and those of many recent visits, so that the workspace stays in the
    // allocator's 1 GiB class
    constexpr int64_t kPassBytes = 960 * (int64_t(1) << 20);
    const bool few = lattice || all * (double)dd::GridEngine::kMostVisitBytes < 0.5 * (double)kPassBytes;
    auto pass_bytes = [&](int k) {
        return (16 + (recents.empty() ? 0 : recents[k] / 512 * 4)) * n_pts + (few ? 0 : dd::GridEngine::table_device_bytes(scan, box, tdim[k], nact[k], contract));
    };
    dd_status st = DD_OK;
    const double *src = dd::device_sources(scan, stream, &st);
    if (!src) return st;
    const dd::ScanUse use{scan, stream};
    const float4 *srcF = dd::device_sources_ff(scan, stream, &st);
    double *out_dev = out;
    void *out_ws = nullptr;
    auto no_memory = [](cudaError_t err) {
        cudaGetLastError();
        return dd::fail(err == cudaErrorMemoryAllocation ? DD_ENOMEM : DD_ECUDA,
                        std::string("field workspace allocation: ") + cudaGetErrorString(err));
    };
    if (out_copy) {
        const cudaError_t err = dd::workspace_alloc(&out_ws, (size_t)n_t * n_pts * sizeof(double), stream);
        if (err != cudaSuccess) return no_memory(err);
        out_dev = static_cast<double *>(out_ws);
    }
    auto *keep = new HostTables();
    for (int g0 = 0, ng = 0; g0 < n_t; g0 += ng) {
        int64_t bytes = few && !lattice ? kPassBytes / 2 : 0;
        for (ng = 0; g0 + ng < n_t && ng < 4096; ++ng) {
            bytes += pass_bytes(g0 + ng);
            if (ng > 0 && bytes > kPassBytes) break;
        }
        dd::GridEngine eng;
        const ShiftGroups sg = shift_groups(scan, grid, tdim, lattice && contract, g0, g0 + ng);
        // (a row of a group's tall grid counts only where some snapshot sees it, at a distance
        // that the grid itself has)
        const int lag = lattice ? eng.add_lag_table(scan, box, M, contract) : -1;
        if (!sg.groups.empty()) {
            dd::GridBox tall = box;
            tall.H = sg.H_ext;
            const int gt = eng.add_grid(scan, tall);
            for (const std::vector<int> &g : sg.groups) {
                std::vector<std::pair<int64_t, int64_t>> snaps;
                for (int k : g) snaps.push_back({(int64_t)tdim[k], (int64_t)order[k] * n_pts});
                eng.add_shift_group(scan, srcF, gt, lag, M, grid.H, sg.rows, snaps);
            }
        }
        const int gi = sg.rest.empty() ? -1 : eng.add_grid(scan, box);
        for (int j : sg.rest) {
            // on the lattice, snapshot t sees visit v at lag t - v: table visit M - t + v
            const int table = lattice ? lag : eng.add_table(scan, box, src, tdim[j], nact[j], contract);
            const int shift = lattice ? (int)(tdim[j] > 0 ? M - (int64_t)tdim[j] : M) : 0;
            eng.add_job(scan, srcF, gi, table, nact[j], shift, (int64_t)order[j] * n_pts);
        }
        DD_CUDA_TRY(eng.finish());
        void *ws = nullptr;
        const cudaError_t err = dd::fault_injected("alloc") ? cudaErrorMemoryAllocation
                                                            : dd::workspace_alloc(&ws, eng.workspace_bytes(), stream);
        if (err != cudaSuccess) {
            dd::defer_release(stream, keep, HostTables::release);   // earlier groups may be in flight
            if (out_ws) dd::workspace_release(out_ws, stream);
            return no_memory(err);
        }
        eng.bind(ws);
        const size_t n_tab = eng.table_bytes();
        char *tables = static_cast<char *>(keep->staging.stage(n_tab));
        if (!tables) {                           // no pinned memory: a pageable image
            keep->images.emplace_back(n_tab);
            tables = keep->images.back().data();
        }
        eng.write_tables(tables);
        DD_CUDA_TRY(cudaMemcpyAsync(ws, tables, n_tab, cudaMemcpyHostToDevice, stream));
        SideStream *side = nullptr;
        DD_CUDA_TRY(side_stream(&side));
        // DD_FAULT=field_tc_wait (tests): no MMA is issued, so the completion waits run out and
        // the kernel reports it (dd_field_check)
        DD_CUDA_TRY(eng.enqueue(out_dev, stream, side->s, side->fork, side->join, dd::fault_injected("field_tc_wait"), true));
        DD_CUDA_TRY(dd::workspace_release(ws, stream));
    }
    if (out_copy) {
        DD_CUDA_TRY(cudaMemcpyAsync(out, out_dev, (size_t)n_t * n_pts * sizeof(double), cudaMemcpyDeviceToHost, stream));
        DD_CUDA_TRY(dd::workspace_release(out_ws, stream));
    }
    DD_CUDA_TRY(dd::defer_release(stream, keep, HostTables::release));
    if (dd::host_sync_needed(stream, {out_kind})) DD_CUDA_TRY(cudaStreamSynchronize(stream));
    return DD_OK;
}

}  // namespace

extern "C" dd_status dd_field_at_times(const dd_scan *scan, const double *pts_xy_m, int64_t n_pts,
                                       const double *times_s, int64_t n_t, dd_precision prec,
                                       double *out, void *cuda_stream) try {
    dd::clear_error();
    if (!scan) return dd::fail(DD_EINVAL, "dd_field_at_times: NULL scan");
    if (n_pts < 0 || n_t < 0) return dd::fail(DD_EINVAL, "dd_field_at_times: negative size");
    if (prec != DD_FP64 && prec != DD_MIXED) return dd::fail(DD_EINVAL, "dd_field_at_times: unknown precision");
    if (n_pts == 0 || n_t == 0) return DD_OK;
    if (!pts_xy_m || !times_s || !out) return dd::fail(DD_EINVAL, "dd_field_at_times: NULL buffer");
    if (n_t > (int64_t(1) << 24) || n_pts > (int64_t(1) << 31))
        return dd::fail(DD_EINVAL, "dd_field_at_times: too many points or snapshots");
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    std::vector<double> times((size_t)n_t);
    if (dd::is_device_pointer(times_s)) {
        DD_CUDA_TRY(cudaMemcpyAsync(times.data(), times_s, n_t * sizeof(double), cudaMemcpyDeviceToHost, stream));
        DD_CUDA_TRY(cudaStreamSynchronize(stream));
    } else {
        std::memcpy(times.data(), times_s, n_t * sizeof(double));
    }
    for (double t : times)
        if (!std::isfinite(t)) return dd::fail(DD_EINVAL, "dd_field_at_times: non-finite time");
    const ddk::GridDesc list;                                     // an explicit point list
    if (prec == DD_MIXED) return run_field<ddk::CfgMixed>(scan, pts_xy_m, n_pts, list, times, out, stream);
    return run_field<ddk::CfgF64>(scan, pts_xy_m, n_pts, list, times, out, stream);
} catch (...) {
    return dd::fail_exception("dd_field_at_times");
}

extern "C" dd_status dd_field_on_grid(const dd_scan *scan, double x0_m, double y0_m, double dx_m, double dy_m,
                                      int64_t n_cols, int64_t n_rows, const double *times_s, int64_t n_t,
                                      dd_precision prec, double *out, void *cuda_stream) try {
    dd::clear_error();
    if (!scan) return dd::fail(DD_EINVAL, "dd_field_on_grid: NULL scan");
    if (n_cols < 0 || n_rows < 0 || n_t < 0) return dd::fail(DD_EINVAL, "dd_field_on_grid: negative size");
    if (prec != DD_FP64 && prec != DD_MIXED) return dd::fail(DD_EINVAL, "dd_field_on_grid: unknown precision");
    if (!std::isfinite(x0_m) || !std::isfinite(y0_m) || !std::isfinite(dx_m) || !std::isfinite(dy_m))
        return dd::fail(DD_EINVAL, "dd_field_on_grid: grid origin and spacing must be finite");
    if (n_cols == 0 || n_rows == 0 || n_t == 0) return DD_OK;
    if (!times_s || !out) return dd::fail(DD_EINVAL, "dd_field_on_grid: NULL buffer");
    if (n_t > (int64_t(1) << 24) || n_cols > (int64_t(1) << 31) || n_rows > (int64_t(1) << 31) ||
        n_cols * n_rows > (int64_t(1) << 31))
        return dd::fail(DD_EINVAL, "dd_field_on_grid: too many points or snapshots");
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    std::vector<double> times((size_t)n_t);
    if (dd::is_device_pointer(times_s)) {
        DD_CUDA_TRY(cudaMemcpyAsync(times.data(), times_s, n_t * sizeof(double), cudaMemcpyDeviceToHost, stream));
        DD_CUDA_TRY(cudaStreamSynchronize(stream));
    } else {
        std::memcpy(times.data(), times_s, n_t * sizeof(double));
    }
    for (double t : times)
        if (!std::isfinite(t)) return dd::fail(DD_EINVAL, "dd_field_on_grid: non-finite time");
    ddk::GridDesc g;
    g.x0 = x0_m; g.y0 = y0_m; g.dx = dx_m; g.dy = dy_m; g.W = n_cols; g.H = n_rows;
    const int64_t n_pts = n_cols * n_rows;
    if (prec == DD_MIXED && std::min(n_cols, n_rows) >= kQuadMinSide && n_pts >= kQuadMinPts && std::max(n_cols, n_rows) < dd::kGridMaxSide)
        return run_grid_mixed(scan, g, times, true, out, stream);
    if (prec == DD_MIXED && narrow_grid(g, n_t, scan->n)) return run_grid_mixed(scan, g, times, false, out, stream);
    if (prec == DD_MIXED) return run_field<ddk::CfgMixed>(scan, nullptr, n_pts, g, times, out, stream);
    return run_field<ddk::CfgF64>(scan, nullptr, n_pts, g, times, out, stream);
} catch (...) {
    return dd::fail_exception("dd_field_on_grid");
}

extern "C" dd_status dd_field_check(void) {
    dd::clear_error();
    DD_CUDA_TRY(cudaDeviceSynchronize());
    bool timed_out = false;
    DD_CUDA_TRY(dd::grid_engine_timed_out(&timed_out));
    if (!timed_out) return DD_OK;
    return dd::fail(DD_ETIMEOUT, "dd_field_check: a tensor-core contraction of the grid field gave up waiting for its MMAs");
}

extern "C" dd_status dd_field_grid_split(const dd_scan *scan, double x0_m, double y0_m, double dx_m, double dy_m,
                                         int64_t n_cols, int64_t n_rows, const double *times_s, int64_t n_t,
                                         int64_t *prefix, int64_t *prefix_deg2) try {
    dd::clear_error();
    if (!scan) return dd::fail(DD_EINVAL, "dd_field_grid_split: NULL scan");
    if (n_cols < 0 || n_rows < 0 || n_t < 0) return dd::fail(DD_EINVAL, "dd_field_grid_split: negative size");
    if (!std::isfinite(x0_m) || !std::isfinite(y0_m) || !std::isfinite(dx_m) || !std::isfinite(dy_m))
        return dd::fail(DD_EINVAL, "dd_field_grid_split: grid origin and spacing must be finite");
    if (n_t == 0) return DD_OK;
    if (!times_s || !prefix) return dd::fail(DD_EINVAL, "dd_field_grid_split: NULL buffer");
    if (dd::is_device_pointer(times_s) || dd::is_device_pointer(prefix) || (prefix_deg2 && dd::is_device_pointer(prefix_deg2)))
        return dd::fail(DD_EINVAL, "dd_field_grid_split: times and prefix are host arrays");
    std::vector<double> times(times_s, times_s + n_t);
    for (double t : times)
        if (!std::isfinite(t)) return dd::fail(DD_EINVAL, "dd_field_grid_split: non-finite time");
    std::vector<int> order, nact;
    std::vector<double> tdim;
    int64_t M = 0;
    snapshot_dims(scan, times, order, tdim, nact, M);
    ddk::GridDesc g;
    g.x0 = x0_m; g.y0 = y0_m; g.dx = dx_m; g.dy = dy_m; g.W = n_cols; g.H = n_rows;
    const TcPlan tp = n_cols > 0 && n_rows > 0 ? plan_tc(scan, g, tdim, nact) : TcPlan();
    for (int k = 0; k < (int)n_t; ++k) {
        prefix[order[k]] = tp.on ? tp.K[k] : 0;
        if (prefix_deg2) prefix_deg2[order[k]] = tp.on ? tp.K2[k] : 0;
    }
    return DD_OK;
} catch (...) {
    return dd::fail_exception("dd_field_grid_split");
}
