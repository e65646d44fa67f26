// dd_grid.cu -- the FP32-mixed field on grids of points: visits in bands of Gauss-Legendre nodes
// on the tensor cores, the last few on the CUDA cores (dd_grid_quad.cuh), for one scan's
// snapshots (dd_field_on_grid) or a batch of scans (dd_batch_create_grid).
//
// Launches: prep (axes, rows of k, records of the recent visits), the contraction, and the final
// kernel (recent visits, partial rows, prefactor).
#include "dd_grid.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <utility>

#include "dd_grid_quad.cuh"

namespace {

using ddk::kGqBands;
using ddk::kGqNodes;

// Largest distances along x and y between the grid's box and the visits' box (pitch units).
void box_reach(const dd_scan *scan, const dd::GridBox &g, double &ex, double &ey) {
    const double ip = 1.0 / scan->pitch;
    const double xa = g.x0 * ip, xb = (g.x0 + (double)(g.W - 1) * g.dx) * ip;
    const double ya = g.y0 * ip, yb = (g.y0 + (double)(g.H - 1) * g.dy) * ip;
    ex = std::max(std::max(xa, xb) - scan->x_lo, scan->x_hi - std::min(xa, xb));
    ey = std::max(std::max(ya, yb) - scan->y_lo, scan->y_hi - std::min(ya, yb));
}

// The largest squared distance between them.
double reach2(const dd_scan *scan, const dd::GridBox &g) {
    double ex, ey;
    box_reach(scan, g, ex, ey);
    // margins for the points' own rounding
    return (ex * ex + ey * ey) * (1.0 + 1e-6) + 1e-6;
}

// Ages (in dwells) from which every visit of the scan takes each band at every point of the
// grid (+inf: none): h = rho^2 dq <= kGqH for rho^2 up to R2, the largest squared distance
// between the grid's box and the visits' box, r = w1/w0 - 1 <= kGqR, and the dwell over.  With
// c = 4 kappa tau_max, dq <= c / ((w1 - c) w1) and r <= c / (w1 - c) for every visit (both grow
// with the dwell at a fixed w1 = 2s + 4 kappa (t - T_i)).  Without the contraction: none.
void band_ages(const dd_scan *scan, const dd::GridBox &g, bool contract, double (&age)[kGqBands]) {
    if (!contract) {
        for (double &a : age) a = INFINITY;
        return;
    }
    const double R2 = reach2(scan, g);
    const double c = 4.0 * scan->kappa * scan->tau_max;
    double prev = INFINITY;
    for (int b = 0; b < kGqBands; ++b) {
        const double dq = ddk::kGqH[b] * (1.0 - 1e-4) / R2;
        double w1 = 0.5 * (c + std::sqrt(c * c + 4.0 * c / dq));
        w1 = std::max({w1, c + c / ddk::kGqR[b], 2.0 * scan->s + c}) * (1.0 + 1e-9);
        const double a = (w1 - 2.0 * scan->s) / (4.0 * scan->kappa) * (1.0 + 1e-9);
        prev = age[b] = std::isfinite(a) && a > 0.0 ? std::min(prev, a) : INFINITY;
    }
}

// Longest time (in dwells) from one visit's start to the next's.
double longest_step(const dd_scan *scan) {
    const double diagonal = scan->pitch * std::hypot((double)scan->nx, (double)scan->ny);
    return scan->tau_max + (scan->flyback + scan->blank + scan->blank_per_m * diagonal) / scan->dwell;
}

// Age (in dwells) from which FP16 pieces (dd_grid_quad.cuh: full precision down to 2^-24 of a piece's
// largest factor) hold a visit's factors at every point of the grid: q D^2, q <= log2(e) / w0, with D the
// largest distance along x or y between the grid's box and the visits', plus the spread of a piece's
// weights within 24.  That is 4 for a rule's, and what dwells of several lengths and the ages of a
// piece's visits (384 at most) make of L = ln(w1/w0).  At most 18 for q D^2; +inf: none.
double fp16_age(const dd_scan *scan, const dd::GridBox &g) {
    double ex, ey;
    box_reach(scan, g, ex, ey);
    const double D = std::max(ex, ey);
    auto age = [&](double range) {
        const double w0 = 1.44269504088896340736 * (D * D) * (1.0 + 1e-6) / range;
        return std::max((w0 - 2.0 * scan->s) / (4.0 * scan->kappa) + scan->tau_max, scan->tau_max);
    };
    const double ages = std::log2(1.0 + (double)ddk::kGqPieceK * longest_step(scan) / age(18.0));
    const double range = std::min(18.0, 20.0 - ages - std::log2(scan->tau_max / scan->tau_min));
    if (!(range >= 6.0)) return INFINITY;
    const double a = age(range);                     // (an older visit's ages spread less)
    return std::isfinite(a) ? a : INFINITY;
}

// Whether FP16 pieces hold the field of a table's visits [i0, i1), at ages age(i), to its full precision
// at every point within R2, so that all of them can take those pieces.  What a piece drops is at most
// 3 2^-50 of its largest weight per row of k.  With weights a few times one another in a piece, and the
// L = ln(w1/w0) of visits one after the other adding up to at most S = ln(w(oldest) / w(youngest)),
// that is 32 2^-50 (S + 1) in all (more with dead times between visits, by the ages that they put into
// the youngest piece), and FP32's rounding is 2^-24 of the field.  The field is at least what the older
// half of the visits leave at the largest distance.
template <typename Age>
bool fp16_everywhere(const dd_scan *scan, double R2, int i0, int i1, int banded, const Age &age) {
    const int half = (i1 - i0) / 2;
    if (half < 1 || banded <= i0) return false;
    auto w1 = [&](int i) { return 2.0 * scan->s + 4.0 * scan->kappa * age(i); };
    const double c = 4.0 * scan->kappa, w_half = w1(i0 + half - 1) - c * scan->tau_max;
    if (!(R2 < 16.0 * w_half)) return false;         // (e^-16 is below the bound)
    const double S = std::log(w1(i0) / (w1(banded - 1) - c * scan->tau_max));
    const double dead = (double)ddk::kGqPieceK * (longest_step(scan) - scan->tau_max) / age(banded - 1);
    const double least = half * std::log1p(c * scan->tau_min / w1(i0)) * std::exp(-R2 / w_half);
    return least >= 0x1p-21 * (S + 1.0) * (1.0 + dead);
}

// The snapshot's first visit past each band.
void band_starts(const dd_scan *scan, const double (&age)[kGqBands], double tdim, int nact, int (&vb)[kGqBands + 1]) {
    vb[0] = 0;
    for (int b = 0; b < kGqBands; ++b) {
        const int64_t k = std::isinf(age[b]) ? 0 : std::upper_bound(scan->T.begin(), scan->T.end(), tdim - age[b]) - scan->T.begin();
        vb[b + 1] = std::max(vb[b], (int)std::min<int64_t>(k, nact));
    }
}

// Rows of k of the table visits before i.
int64_t rows_before(const int (&vb)[kGqBands + 1], int64_t i) {
    int64_t k = 0;
    for (int b = 0; b < kGqBands && vb[kGqBands] > 0; ++b)
        k += std::max<int64_t>(0, std::min<int64_t>(i, vb[b + 1]) - vb[b]) * kGqNodes[b];
    return k;
}

int sm_count() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return 1;
    int v = cached[dev].load();
    if (v > 0) return v;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1) {
        cudaGetLastError();
        return 1;
    }
    cached[dev].store(v);
    return v;
}

cudaError_t prepare_kernel() {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess || dev >= 64) return err;
    if (done.load() & (uint64_t(1) << dev)) return cudaSuccess;
    err = cudaFuncSetAttribute(ddk::grid_quad_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ddk::kGqSmemBytes);
    if (err == cudaSuccess)
        err = cudaFuncSetAttribute(ddk::grid_quad_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ddk::kGqSmemBytes);
    if (err == cudaSuccess) done.fetch_or(uint64_t(1) << dev);
    return err;
}

}  // namespace

namespace dd {

struct GridEngine::Tables {
    std::vector<ddk::GqGrid> grids;
    std::vector<ddk::GqTable> tabs;
    std::vector<ddk::GqJob> jobs;
    std::vector<ddk::GqRun> runs;                        // CTA by CTA, launch by launch
    std::vector<int> cta_off;                            // first run of each CTA, per launch n_cta + 1
    std::vector<int64_t> ax_offs, vis_offs, rec_offs;
    std::vector<int64_t> part_tiles, out_tiles;          // tiles of the jobs that write partial rows, the field
    std::vector<double> tab_R2;                          // per table: largest squared distance to the grid
    struct Span { int64_t k0, k1, split; };              // rows of k of a job; from split on: BF16 pieces
    std::vector<Span> spans;
    std::vector<ddk::GqGroup> groups;                    // raster snapshots summed by segments of lags
    std::vector<ddk::GqSegment> segs;
    std::vector<int> seg_job;
    int64_t n_shift_blocks = 0;
    int n_cta[2] = {0, 0};
    int64_t n_ax = 0, n_vis = 0, n_rows = 0, n_rec = 0, n_part = 0;
    // device
    char *base = nullptr;
    ddk::GqRow *rows = nullptr;
    ddk::RecF32 *rec = nullptr;
    float2 *ax = nullptr;
    float *part = nullptr;

    struct Layout { size_t grids, tabs, jobs, runs, cta, axo, viso, reco, parto, outo, groups, segs, end; };
    Layout layout() const {
        Layout l;
        size_t b = 0;
        auto add = [&](size_t n) { const size_t o = b; b = (b + n + 255) & ~size_t(255); return o; };
        l.grids = add(grids.size() * sizeof(ddk::GqGrid));
        l.tabs = add(tabs.size() * sizeof(ddk::GqTable));
        l.jobs = add(jobs.size() * sizeof(ddk::GqJob));
        l.runs = add(runs.size() * sizeof(ddk::GqRun));
        l.cta = add(cta_off.size() * sizeof(int));
        l.axo = add(ax_offs.size() * sizeof(int64_t));
        l.viso = add(vis_offs.size() * sizeof(int64_t));
        l.reco = add(rec_offs.size() * sizeof(int64_t));
        l.parto = add(part_tiles.size() * sizeof(int64_t));
        l.outo = add(out_tiles.size() * sizeof(int64_t));
        l.groups = add(groups.size() * sizeof(ddk::GqGroup));
        l.segs = add(segs.size() * sizeof(ddk::GqSegment));
        l.end = b;
        return l;
    }
};

GridEngine::GridEngine() : t(new Tables()) {}
GridEngine::~GridEngine() { delete t; }

int GridEngine::add_grid(const dd_scan *scan, const GridBox &g) {
    t->grids.push_back({g.x0, g.y0, g.dx, g.dy, 1.0 / scan->pitch, t->n_ax, (int)g.W, (int)g.H});
    t->ax_offs.push_back(t->n_ax);
    t->n_ax += g.W + g.H;
    return (int)t->grids.size() - 1;
}

int GridEngine::add_table(const dd_scan *scan, const GridBox &g, const double *src, double tdim, int nact, bool contract) {
    double age[kGqBands];
    band_ages(scan, g, contract, age);
    ddk::GqTable tb{src + 2 * scan->n, src + 3 * scan->n, scan->s, scan->kappa, tdim, t->n_vis, t->n_rows, t->n_rec, nact, 0, {}};
    band_starts(scan, age, tdim, nact, tb.vb);
    const double a16 = fp16_age(scan, g);
    if (!std::isinf(a16))
        tb.n_fp16 = (int)std::min<int64_t>(tb.vb[kGqBands], std::upper_bound(scan->T.begin(), scan->T.end(), tdim - a16) - scan->T.begin());
    t->tabs.push_back(tb);
    t->tab_R2.push_back(reach2(scan, g));
    t->vis_offs.push_back(t->n_vis);
    t->rec_offs.push_back(t->n_rec);
    t->n_vis += nact;
    t->n_rows += rows_before(tb.vb, nact);
    t->n_rec += nact - tb.vb[kGqBands];
    return (int)t->tabs.size() - 1;
}

int GridEngine::add_lag_table(const dd_scan *scan, const GridBox &g, int64_t M, bool contract) {
    double age[kGqBands];
    band_ages(scan, g, contract, age);
    ddk::GqTable tb{nullptr, nullptr, scan->s, scan->kappa, 0.0, t->n_vis, t->n_rows, t->n_rec, (int)M, 0, {}};
    tb.vb[0] = 0;
    for (int b = 0; b < kGqBands; ++b) {
        const double last = std::floor((double)M - age[b]);             // lag M - i >= age
        tb.vb[b + 1] = last >= 0.0 ? std::max(tb.vb[b], (int)std::min((double)M, last + 1.0)) : tb.vb[b];
    }
    const double oldest = std::floor((double)M - fp16_age(scan, g));
    if (oldest >= 0.0) tb.n_fp16 = (int)std::min((double)tb.vb[kGqBands], oldest + 1.0);
    t->tabs.push_back(tb);
    t->tab_R2.push_back(reach2(scan, g));
    t->vis_offs.push_back(t->n_vis);
    t->rec_offs.push_back(t->n_rec);
    t->n_vis += M;
    t->n_rows += rows_before(tb.vb, M);
    t->n_rec += M - tb.vb[kGqBands];
    return (int)t->tabs.size() - 1;
}

void GridEngine::add_job(const dd_scan *scan, const float4 *srcF, int grid, int table, int nact, int shift,
                         int64_t out_off) {
    add_span(scan, srcF, grid, table, shift, shift + nact, shift, t->grids[grid].H, out_off);
}

// Table visits [i0, i1) on the first H rows of the grid.
void GridEngine::add_span(const dd_scan *scan, const float4 *srcF, int grid, int table, int i0, int i1, int shift, int H,
                          int64_t out_off) {
    const ddk::GqGrid &g = t->grids[grid];
    const ddk::GqTable &tb = t->tabs[table];
    ddk::GqJob j{};
    j.srcF = srcF;
    j.ax_off = g.ax_off;
    j.W = g.W;
    j.H = H;
    j.n_tc = (g.W + ddk::kGqTile - 1) / ddk::kGqTile;
    j.tw = ((g.W + j.n_tc - 1) / j.n_tc + 15) / 16 * 16;               // even widths: less padding
    j.shift = shift;
    const int kc = std::min(std::max(tb.vb[kGqBands], i0), i1);
    j.r0 = kc - shift;
    j.r1 = i1 - shift;
    j.rec0 = tb.rec_off + (kc - tb.vb[kGqBands]);
    j.t_stride = ((int64_t)g.W * H + 3) / 4 * 4;
    j.out_off = out_off;
    j.pref = scan->pref;
    t->jobs.push_back(j);
    // (a segment's field holds the younger segments, too)
    const bool fp16 = kc > std::max(tb.n_fp16, i0) && fp16_everywhere(scan, t->tab_R2[table], i0, out_off < 0 ? tb.n_vis : i1, kc, [&](int i) {
        return tb.T ? tb.tdim - scan->T[(size_t)i] : (double)(tb.n_vis - i);
    });
    const int mid = fp16 ? kc : std::min(std::max(tb.n_fp16, i0), kc);
    t->spans.push_back({tb.k_off + rows_before(tb.vb, i0), tb.k_off + rows_before(tb.vb, kc), tb.k_off + rows_before(tb.vb, mid)});
}

void GridEngine::add_shift_group(const dd_scan *scan, const float4 *srcF, int grid, int table, int64_t M, int64_t H,
                                 int rows_per_scan_row, const std::vector<std::pair<int64_t, int64_t>> &snaps) {
    const int64_t last = snaps.back().first, shift = M - last;
    const int W = t->grids[grid].W, H_ext = (int)(H + rows_per_scan_row * ((last - snaps[0].first) / scan->nx));
    const int64_t tiles = (int64_t)((W + 31) / 32) * ((H_ext + 3) / 4);
    t->groups.push_back({t->n_shift_blocks, (int)t->segs.size(), (int)snaps.size(), W, (int)H, H_ext, 0, scan->pref});
    t->n_shift_blocks += tiles;
    int64_t before = 0;
    for (const auto &s : snaps) {
        const int rows = rows_per_scan_row * (int)((last - s.first) / scan->nx);
        t->seg_job.push_back((int)t->jobs.size());
        t->segs.push_back({0, 0, s.second, 0, rows, (int)H + rows, 0});
        add_span(scan, srcF, grid, table, (int)(M - s.first), (int)(M - before), (int)shift, (int)H + rows, -1);
        before = s.first;
    }
}

double GridEngine::banded_age(const dd_scan *scan, const GridBox &g) {
    double age[kGqBands];
    band_ages(scan, g, true, age);
    return age[kGqBands - 1];
}

int64_t GridEngine::table_device_bytes(const dd_scan *scan, const GridBox &g, double tdim, int nact, bool contract) {
    double age[kGqBands];
    int vb[kGqBands + 1];
    band_ages(scan, g, contract, age);
    band_starts(scan, age, tdim, nact, vb);
    return rows_before(vb, nact) * (int64_t)sizeof(ddk::GqRow) + (nact - vb[kGqBands]) * (int64_t)sizeof(ddk::RecF32);
}

// Tiles of a job's recent visits (a segment with none has none).
static int64_t fin_tiles(const ddk::GqJob &j) {
    return j.out_off < 0 && j.r1 <= j.r0 ? 0 : (int64_t)((j.W + 31) / 32) * ((j.H + ddk::kGqFinRows - 1) / ddk::kGqFinRows);
}

// Places of a job's partial rows; its recent visits in P parts, the earlier ones as jobs of their own
// that write partial rows after the contraction's.
void GridEngine::place_rows(size_t k, int P) {
    ddk::GqJob &j = t->jobs[k];
    const int r0 = j.r0, n = j.r1 - r0, nq = j.nq;
    j.t_off = t->n_part;
    j.row = j.nq = nq + P - 1;
    t->n_part += (int64_t)(j.row + (j.out_off < 0 && n > 0 ? 1 : 0)) * j.t_stride;
    if (P < 2) return;
    auto at = [&](int e) { return r0 + (int)((int64_t)n * e / P); };
    const int64_t rec0 = j.rec0;
    j.r0 = at(P - 1);
    j.rec0 += j.r0 - r0;
    ddk::GqJob part = j;
    part.out_off = -1;
    for (int e = 0; e + 1 < P; ++e) {
        part.row = nq + e;
        part.r0 = at(e);
        part.r1 = at(e + 1);
        part.rec0 = rec0 + (part.r0 - r0);
        t->jobs.push_back(part);
    }
}

cudaError_t GridEngine::finish() {
    const int sms = sm_count();
    // Cost of a run: its rows of k times the factors formed per row (32 positions at a time),
    // plus about 130 rows' worth of factors for its start, drain and output (500 left 64 short segments
    // in 110 runs of 152 SMs: 8 us longer).
    auto row_cost = [](const ddk::GqJob &j, int tile) {
        const int nc = std::min(j.tw, j.W - (tile % j.n_tc) * j.tw);
        const int nr = std::min(ddk::kGqTile, j.H - (tile / j.n_tc) * ddk::kGqTile);
        return (int64_t)((nc + 31) / 32 + (nr + 31) / 32 + 1);
    };
    constexpr int64_t kRunCost = 1200;
    for (int launch = 0; launch < 2; ++launch) {
        auto span = [&](size_t j, int64_t &k0, int64_t &k1) {
            const Tables::Span &s = t->spans[j];
            k0 = launch == 0 ? s.split : s.k0;
            k1 = launch == 0 ? s.k1 : s.split;
        };
        int64_t total = 0;
        for (size_t j = 0; j < t->jobs.size(); ++j) {
            int64_t k0, k1;
            span(j, k0, k1);
            const ddk::GqJob &J = t->jobs[j];
            const int n_tiles = J.n_tc * ((J.H + ddk::kGqTile - 1) / ddk::kGqTile);
            for (int q = 0; q < n_tiles && k1 > k0; ++q) total += (k1 - k0) * row_cost(J, q);
        }
        if (total == 0) continue;
        // about two runs per CTA, so that dealing them out longest first evens the CTAs' shares
        const int64_t per = std::max<int64_t>(total / (2 * sms), 2 * kRunCost);
        std::vector<ddk::GqRun> list;
        std::vector<std::pair<int64_t, int>> order;      // (- cost, run)
        list.reserve((size_t)(4 * sms) + t->jobs.size());
        order.reserve(list.capacity());
        for (size_t j = 0; j < t->jobs.size(); ++j) {
            int64_t k0, k1;
            span(j, k0, k1);
            if (k1 <= k0) continue;
            ddk::GqJob &J = t->jobs[j];
            const int n_tiles = J.n_tc * ((J.H + ddk::kGqTile - 1) / ddk::kGqTile);
            // every tile of the job in the same number of pieces (whole partial rows)
            const int64_t cost = (k1 - k0) * row_cost(J, 0), steps = (k1 - k0 + 15) / 16;
            const int64_t P = std::min(std::max({int64_t(1), (cost + per / 2) / per, (steps + ddk::kGqRunSteps - 1) / ddk::kGqRunSteps}), steps);
            for (int64_t p = 0; p < P; ++p) {
                const int64_t a = k0 + steps * p / P * 16, b = std::min(k1, k0 + steps * (p + 1) / P * 16);
                for (int q = 0; q < n_tiles; ++q) {
                    order.push_back({-((b - a) * row_cost(J, q) + kRunCost), (int)list.size()});
                    list.push_back(ddk::GqRun{a, (int)(b - a), (int)j, q, J.nq + (int)p});
                }
            }
            J.nq += (int)P;
        }
        std::sort(order.begin(), order.end());
        // dealt out longest first, back and forth over the CTAs: run k goes to CTA k % n on even
        // rounds and n - 1 - k % n on odd ones
        const int n = (int)std::min<int64_t>(sms, (int64_t)list.size()), full = (int)list.size() / n, rest = (int)list.size() % n;
        const int base = (int)t->runs.size();
        auto extra = [&](int c) { return (full & 1 ? n - 1 - c : c) < rest ? 1 : 0; };   // a run of the last round
        t->n_cta[launch] = n;
        for (int c = 0, off = base; c <= n; ++c) {
            t->cta_off.push_back(off);
            if (c < n) off += full + extra(c);
        }
        const int *const off = t->cta_off.data() + t->cta_off.size() - (size_t)(n + 1);
        t->runs.resize((size_t)base + list.size());
        for (size_t k = 0; k < list.size(); ++k) {
            const int round = (int)k / n, pos = (int)k % n, c = (round & 1) ? n - 1 - pos : pos;
            t->runs[(size_t)(off[c] + round)] = list[(size_t)order[k].second];
        }
    }
    // places of the partial rows and the tiles of the recent visits, every job's in one part
    const size_t n_jobs = t->jobs.size();
    int64_t n_part = 0, n_out = 0;
    auto tile_tables = [&] {
        n_part = n_out = 0;
        t->part_tiles.resize(t->jobs.size() + 1);
        t->out_tiles.resize(t->jobs.size() + 1);
        for (size_t k = 0; k <= t->jobs.size(); ++k) {
            t->part_tiles[k] = n_part;
            t->out_tiles[k] = n_out;
            if (k < t->jobs.size()) (t->jobs[k].out_off < 0 ? n_part : n_out) += fin_tiles(t->jobs[k]);
        }
    };
    int longest = 0;
    for (ddk::GqJob &j : t->jobs) {
        const int n = j.r1 - j.r0;
        j.t_off = t->n_part;
        j.row = j.nq;
        t->n_part += (int64_t)(j.nq + (j.out_off < 0 && n > 0 ? 1 : 0)) * j.t_stride;
        longest = std::max(longest, n);
    }
    tile_tables();
    // more than kGqFinSplit recent visits are split while the tiles leave places for CTAs (two waves),
    // more than kGqFinMost always
    if (longest > ddk::kGqFinSplit) {
        const int64_t most = std::max<int64_t>(1, 2 * ddk::kGqFinResident * (int64_t)sms / (n_part + n_out));
        t->n_part = 0;
        for (size_t k = 0; k < n_jobs; ++k) {
            const int n = t->jobs[k].r1 - t->jobs[k].r0;
            const int64_t parts = n > ddk::kGqFinSplit ? (n + ddk::kGqFinVisits - 1) / ddk::kGqFinVisits : 1;
            place_rows(k, (int)std::max<int64_t>((n + ddk::kGqFinMost - 1) / ddk::kGqFinMost, std::max<int64_t>(1, std::min(most, parts))));
        }
        tile_tables();
    }
    if (n_part == 0) t->part_tiles.clear();
    if (n_out == 0) t->out_tiles.clear();
    for (size_t k = 0; k < t->segs.size(); ++k) {
        const ddk::GqJob &j = t->jobs[(size_t)t->seg_job[k]];
        t->segs[k].t_off = j.t_off;
        t->segs[k].t_stride = j.t_stride;
        t->segs[k].n_part = j.row + (j.r1 > j.r0 ? 1 : 0);
    }
    return t->runs.empty() ? cudaSuccess : prepare_kernel();
}

size_t GridEngine::table_bytes() const { return t->layout().end; }

size_t GridEngine::workspace_bytes() const {
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    return up(table_bytes()) + up((size_t)t->n_rows * sizeof(ddk::GqRow)) + up((size_t)t->n_rec * sizeof(ddk::RecF32)) +
           up((size_t)t->n_ax * sizeof(float2)) + up((size_t)t->n_part * sizeof(float)) + 256;
}

void GridEngine::write_tables(char *dst) const {
    const Tables::Layout l = t->layout();
    auto put = [&](size_t off, const auto &v) {
        if (!v.empty()) std::memcpy(dst + off, v.data(), v.size() * sizeof(v[0]));
    };
    put(l.grids, t->grids);
    put(l.tabs, t->tabs);
    put(l.jobs, t->jobs);
    put(l.runs, t->runs);
    put(l.cta, t->cta_off);
    put(l.axo, t->ax_offs);
    put(l.viso, t->vis_offs);
    put(l.reco, t->rec_offs);
    put(l.parto, t->part_tiles);
    put(l.outo, t->out_tiles);
    put(l.groups, t->groups);
    put(l.segs, t->segs);
}

void GridEngine::bind(void *workspace) {
    char *p = static_cast<char *>(workspace);
    auto take = [&](size_t b) { char *q = p; p += (b + 255) & ~size_t(255); return q; };
    t->base = take(table_bytes());
    t->rows = reinterpret_cast<ddk::GqRow *>(take((size_t)t->n_rows * sizeof(ddk::GqRow)));
    t->rec = reinterpret_cast<ddk::RecF32 *>(take((size_t)t->n_rec * sizeof(ddk::RecF32)));
    t->ax = reinterpret_cast<float2 *>(take((size_t)t->n_ax * sizeof(float2)));
    t->part = reinterpret_cast<float *>(take((size_t)t->n_part * sizeof(float)));
}

int64_t GridEngine::n_tiles() const {
    return (t->part_tiles.empty() ? 0 : t->part_tiles.back()) + (t->out_tiles.empty() ? 0 : t->out_tiles.back());
}
int64_t GridEngine::n_runs() const { return (int64_t)t->runs.size(); }

cudaError_t GridEngine::enqueue(double *out, cudaStream_t stream, cudaStream_t side, cudaEvent_t fork,
                                cudaEvent_t join, bool withhold, bool profile) {
    if (t->jobs.empty()) return cudaSuccess;
    const Tables::Layout l = t->layout();
    const ddk::GqJob *jobs = reinterpret_cast<const ddk::GqJob *>(t->base + l.jobs);
    const ddk::GqRun *runs = reinterpret_cast<const ddk::GqRun *>(t->base + l.runs);
    const int *cta = reinterpret_cast<const int *>(t->base + l.cta);
    cudaError_t err;
    auto scoped = [&](const char *name, cudaStream_t s, auto &&launch) {
        if (profile) {
            dd::ProfScope ps(name, s);
            launch();
        } else {
            launch();
        }
        return cudaGetLastError();
    };
    const int64_t n_prep = ddk::gq_warps(t->n_rec) + ddk::gq_warps(t->n_vis) + t->n_ax;
    auto offs = [&](size_t o) { return reinterpret_cast<const int64_t *>(t->base + o); };
    const ddk::GqPrep prep{reinterpret_cast<const ddk::GqTable *>(t->base + l.tabs), offs(l.reco), offs(l.viso), offs(l.axo),
                           reinterpret_cast<const ddk::GqGrid *>(t->base + l.grids), t->n_rec, t->n_vis, t->n_ax,
                           (int)t->tabs.size(), (int)t->grids.size(), t->rows, t->rec, t->ax};
    if ((err = scoped("coef_mixed", stream, [&] {
             ddk::grid_quad_prep_kernel<<<(unsigned)((n_prep + 63) / 64), 64, 0, stream>>>(prep);
         })) != cudaSuccess)
        return err;
    // launch 0: the BF16 pieces, the longer runs; launch 1: the FP16 pieces
    auto contraction = [&](int k, cudaStream_t s) -> cudaError_t {
        if (t->n_cta[k] == 0) return cudaSuccess;
        const char *name = k == 0 || t->n_cta[0] == 0 ? "field_grid_tc" : "field_grid_tc4";
        const int *off = cta + (k == 0 || t->n_cta[0] == 0 ? 0 : t->n_cta[0] + 1);
        auto *const kernel = k == 0 ? ddk::grid_quad_kernel<true> : ddk::grid_quad_kernel<false>;
        return scoped(name, s, [&] {
            kernel<<<(unsigned)t->n_cta[k], ddk::kGqThreads, ddk::kGqSmemBytes, s>>>(
                jobs, runs, off, t->rows, t->ax, t->part, withhold ? 1 : 0);
        });
    };
    auto recent = [&](const std::vector<int64_t> &tiles, size_t o, cudaStream_t s) -> cudaError_t {
        if (tiles.empty()) return cudaSuccess;
        return scoped("field_grid_mixed", s, [&] {
            ddk::grid_quad_final_kernel<<<(unsigned)tiles.back(), ddk::kGqFinThreads, 0, s>>>(
                jobs, offs(o), (int)t->jobs.size(), t->rec, t->ax, t->part, out);
        });
    };
    // beside the first contraction launch: the second, and the recent visits that go to partial
    // rows (all on one stream: 86 us instead of 72 on 64 shared row snapshots)
    const bool both = side != nullptr && t->n_cta[0] > 0 && (t->n_cta[1] > 0 || !t->part_tiles.empty());
    cudaStream_t second = both ? side : stream;
    if (both) {
        if ((err = cudaEventRecord(fork, stream)) != cudaSuccess) return err;
        if ((err = cudaStreamWaitEvent(side, fork, 0)) != cudaSuccess) return err;
    }
    if ((err = contraction(0, stream)) != cudaSuccess) return err;
    if ((err = recent(t->part_tiles, l.parto, second)) != cudaSuccess) return err;
    if ((err = contraction(1, second)) != cudaSuccess) return err;
    if (both) {
        if ((err = cudaEventRecord(join, side)) != cudaSuccess) return err;
        if ((err = cudaStreamWaitEvent(stream, join, 0)) != cudaSuccess) return err;
    }
    if ((err = recent(t->out_tiles, l.outo, stream)) != cudaSuccess) return err;
    if (t->groups.empty()) return cudaSuccess;
    return scoped("field_reduce", stream, [&] {
        ddk::grid_quad_shift_kernel<<<(unsigned)t->n_shift_blocks, 128, 0, stream>>>(
            reinterpret_cast<const ddk::GqGroup *>(t->base + l.groups), (int)t->groups.size(),
            reinterpret_cast<const ddk::GqSegment *>(t->base + l.segs), t->part, out);
    });
}

cudaError_t grid_engine_timed_out(bool *timed_out) {
    int flag = 0;
    cudaError_t err = cudaMemcpyFromSymbol(&flag, ddk::g_grid_quad_timeout, sizeof(int));
    *timed_out = err == cudaSuccess && flag != 0;
    if (!*timed_out) return err;
    const int zero = 0;
    return cudaMemcpyToSymbol(ddk::g_grid_quad_timeout, &zero, sizeof(int));
}

}  // namespace dd
