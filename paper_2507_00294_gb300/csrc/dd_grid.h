// dd_grid.h -- host side of the FP32-mixed field on grids of points (dd_grid.cu): the tables,
// workspace layout and launches of a set of jobs, one job = one snapshot of one scan on one grid.
// Used per call by dd_field_on_grid and per plan by the grid batches.
#pragma once
#include <cstdint>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "dd_internal.h"

namespace ddk {
struct GqGrid;
struct GqTable;
struct GqJob;
struct GqRun;
struct GqRow;
}  // namespace ddk

namespace dd {

// A grid of evaluation points [m].
struct GridBox {
    double x0 = 0, y0 = 0, dx = 0, dy = 0;
    int64_t W = 0, H = 0;
};

// Sides below this: the engine's column, row and tile numbers are 32-bit.
constexpr int64_t kGridMaxSide = int64_t(1) << 30;

class GridEngine {
  public:
    GridEngine();
    ~GridEngine();
    GridEngine(const GridEngine &) = delete;
    GridEngine &operator=(const GridEngine &) = delete;

    // Axes of a grid (W, H < kGridMaxSide) in the scan's pitch units; returns its index.
    int add_grid(const dd_scan *scan, const GridBox &g);
    // Coefficients of the visits [0, nact) of a scan at tdim (dwells), or of the lags M .. 1 of a
    // uniform scan; src: the scan's device block; contract: false leaves every visit to the
    // CUDA cores.  Returns the table's index.
    int add_table(const dd_scan *scan, const GridBox &g, const double *src, double tdim, int nact, bool contract);
    int add_lag_table(const dd_scan *scan, const GridBox &g, int64_t M, bool contract);
    // The scan's snapshot with nact started visits, table visit = visit + shift; its field goes to
    // out + out_off (W H values).
    void add_job(const dd_scan *scan, const float4 *srcF, int grid, int table, int nact, int shift, int64_t out_off);
    // Snapshots M_0 < M_1 < .. (dwells; each with its offset in out) of one phase of a raster, on
    // the first H rows of a grid that reaches the tall grid of the group (dd_grid_quad.cuh);
    // table: the lags M .. 1; rows_per_scan_row: grid rows per pitch.
    void add_shift_group(const dd_scan *scan, const float4 *srcF, int grid, int table, int64_t M, int64_t H,
                         int rows_per_scan_row, const std::vector<std::pair<int64_t, int64_t>> &snaps);
    // Age (in dwells) from which every visit of a scan is in the contraction's bands on a grid.
    static double banded_age(const dd_scan *scan, const GridBox &g);
    // Device bytes that add_table takes, and the most a visit can.
    static int64_t table_device_bytes(const dd_scan *scan, const GridBox &g, double tdim, int nact, bool contract);
    static constexpr int64_t kMostVisitBytes = 512;      // 32 nodes
    // Splits the contraction into runs for the device's SMs, in two launches: the rows of k in BF16
    // pieces, and those in FP16 pieces.
    cudaError_t finish();

    size_t table_bytes() const;          // host tables, uploaded to the workspace's first bytes
    size_t workspace_bytes() const;
    void write_tables(char *dst) const;
    void bind(void *workspace);
    // Launches on `stream`; the second contraction launch goes to `side` (may be NULL), forked and
    // joined by the two events.  withhold: testing hook of the bounded waits.
    cudaError_t enqueue(double *out, cudaStream_t stream, cudaStream_t side, cudaEvent_t fork, cudaEvent_t join,
                        bool withhold, bool profile);
    int64_t n_tiles() const;             // tiles of the recent visits' kernel
    int64_t n_runs() const;

  private:
    void add_span(const dd_scan *scan, const float4 *srcF, int grid, int table, int i0, int i1, int shift, int H,
                  int64_t out_off);
    void place_rows(size_t job, int parts);
    struct Tables;
    Tables *t;
};

// Whether a contraction gave up waiting since the last call (clears the flag).
cudaError_t grid_engine_timed_out(bool *timed_out);

}  // namespace dd
