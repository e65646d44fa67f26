// dd_grid_quad.cuh -- the FP32-mixed field on a rectilinear grid of points as a contraction on
// the 5th-generation tensor cores.
//
// A visit's pair term is E1(rho^2/w1) - E1(rho^2/w0) = int_0^L exp(-(rho^2/w1) e^y) dy with
// L = ln(w1/w0) (substitute u = (rho^2/w1) e^y in E1's integral).  Gauss-Legendre with n nodes
// u_j, weights c_j on [0, 1] makes it a sum of n Gaussians,
//   term = sum_j w_j 2^(-q_j rho^2),  q_j = log2(e) e^(L u_j) / w1,  w_j = L c_j,
// each of which splits into a column and a row factor, 2^(-q_j dx^2) 2^(-q_j dy^2).  So the
// field of the visits is a matrix product over (visit, node): F(r, c) = sum_k Y_k(r) X_k(c).
// The nodes needed for 1e-7 of the term depend on h = rho^2 (1/w0 - 1/w1) and on r = w1/w0 - 1
// (kGqH, kGqR, checked against 300-point quadrature): one node for the oldest visits, 2 and 3
// for most, 12 for h up to 28.5, 32 up to 218.  With R2 the largest squared distance between the grid's box
// and the visits' box, every visit older than some age takes a given n, so the visits of a
// snapshot fall into bands of rising n; only the last few visits (h past 218 somewhere on the
// grid, r > 1, or still under the beam) stay with the CUDA cores.
//
// (A form with one exponential per visit, X Y + A B + .., covers h <= 0.04 with two products
// and h <= 0.33 with four, in pieces of 7 and 12 MMAs per 16 visits; here 16 rows of k take 3
// MMAs, two nodes reach h = 0.143 and three 0.76.)
//
// Factors are formed in FP32 and split into 16-bit pieces, in one of two forms.
//   BF16: F = h + m + l, each the round-to-nearest of what is left (2^-24 of F, FP32's exponent
//     range); six products, X_h Y_h, X_h Y_m, X_m Y_h, X_m Y_m, X_h Y_l, X_l Y_h.
//   FP16: F 2^14 = h + l 2^-11 (2^-23 of F down to F = 2^-26, then an absolute 2^-49; -l is what is
//     stored); three products, X_h Y_h, X_h Y_l, X_l Y_h (X_l Y_l, 2^-22 at most and of either sign,
//     is left out).
// FP16 takes the visits old enough that no factor reaches below 2^-18 anywhere on the grid (fp16_age of
// dd_grid.cu), and every visit where the field itself stays so close to its largest term that what FP16
// drops is below FP32's rounding (fp16_everywhere); BF16 the rest, so that the field keeps FP32's
// relative accuracy where it is many orders below its peak: with FP16 pieces alone it was off by 3e-5 at
// 1e-8 to 1e-12 of the peak and lost below that (64 x 64 visits, D = 1e-15 .. 6e-14); now 4e-7 to
// 1.3e-5 down to 1e-32 of it, as the exponents' own rounding.  All in BF16 pieces: 200 us instead of
// 156 for 256 x 256 points x 65,536 visits x 2 snapshots, 1313 instead of 1150 for 512 uneven scans
// (all in FP16: 171, 1000).  One kernel that chose per piece: 196, 1307.
// The leading products accumulate in one FP32 tensor-memory accumulator and the rest in a second.
// The factors are taken relative to the tile: p = floor(q dxmin^2) moves from Y's exponent to X's
// (dxmin: the visit's distance from the tile's columns), so that X's largest value is about 1, and
// the piece's largest Y is scaled to 1 .. 2.
//
// The tensor core's FP32 accumulation drops low bits of every product against the running sum:
// with the leading products of 512 rows of k in one accumulator the field came out 2e-6 low.  So
// the leading accumulator takes one stage of 64 rows of k (four MMAs), and four warps add the
// stages up in FP32 registers while the next one forms in a second accumulator set; the other
// products, 2^-8 or 2^-11 as large, accumulate over a piece of up to 384 rows.  What four MMAs
// still lose of the field on average, 1.0e-7 to 1.7e-7 in FP16 pieces and 0.3e-7 to 1.5e-7 in BF16,
// is put back by a factor (gq_unbias); one to three MMAs lose under 0.5e-7.
//
// One CTA per SM walks its list of runs (a run: one tile of one snapshot, a range of k), piece by
// piece.  Three warps fetch a piece's rows of k and visits and turn them into coefficients
// relative to the tile, one or two pieces ahead; 16 producer warps form 64 k x (rows +
// columns) factors per stage -- warp = 8 rows of k of the row or the column side, lane = four
// positions, so that coefficients come from shared memory once for 128 factors; one warp
// issues the MMAs; and four draining warps (128 accumulators each lane:
// registers moved from the other warps by setmaxnreg) write each run's sums as one FP32 row.
// All of them meet at mbarriers only.
//
// Measured (GB300, a call with its other kernels, before: two contractions of 7 and 12 MMAs per 16
// visits beside a CUDA-core tile kernel for the last visits): 256 x 256 points x 65,536 visits
// x 2 snapshots 306 -> 156 us (3,000 clocks per stage of FP16 pieces and SM, the producers'
// instruction latency; 3,900 in BF16); 512 uneven scans on their probe grids 1683 -> 1150 us; 64 row
// snapshots of a 64 x 64 raster on 128 x 128 points 223 -> 80 us (with shared sums, below).  Error
// against 64 bits (2-norm) 3.2e-7, 1.0e-6 and 2.1e-7 -> 0.3e-7, 1.5e-7 and 0.6e-7.
#pragma once
#include <cstdint>

#include "dd_coef.cuh"
#include "dd_field_impl.cuh"
#include "dd_umma.cuh"

namespace ddk {

// Bands, oldest first: nodes, largest h and largest r = w1/w0 - 1 at which they hold 1e-7.
constexpr int kGqBands = 13;
constexpr int kGqNodes[kGqBands] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32};
constexpr double kGqH[kGqBands] = {1.5e-3, 0.143, 0.76, 1.93, 3.59, 5.77, 11.5, 19.2, 28.5, 52.0, 83.0, 121.0, 218.0};
constexpr double kGqR[kGqBands] = {1e-3, 0.1, 0.5, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 1.0};

// Gauss-Legendre nodes on [0, 1] and weights, band after band.
constexpr int kGqRuleSize = 143;
struct GqRule {
    float u[kGqRuleSize], c[kGqRuleSize];
    int first[kGqBands], nodes[kGqBands];
};
static __device__ __constant__ GqRule kGqRule = {
    {5.000000000e-01f, 2.113248654e-01f, 7.886751346e-01f, 1.127016654e-01f, 5.000000000e-01f, 8.872983346e-01f,
     6.943184420e-02f, 3.300094782e-01f, 6.699905218e-01f, 9.305681558e-01f, 4.691007703e-02f, 2.307653449e-01f,
     5.000000000e-01f, 7.692346551e-01f, 9.530899230e-01f, 3.376524290e-02f, 1.693953068e-01f, 3.806904070e-01f,
     6.193095930e-01f, 8.306046932e-01f, 9.662347571e-01f, 1.985507175e-02f, 1.016667613e-01f, 2.372337950e-01f,
     4.082826788e-01f, 5.917173212e-01f, 7.627662050e-01f, 8.983332387e-01f, 9.801449282e-01f, 1.304673574e-02f,
     6.746831666e-02f, 1.602952159e-01f, 2.833023029e-01f, 4.255628305e-01f, 5.744371695e-01f, 7.166976971e-01f,
     8.397047841e-01f, 9.325316833e-01f, 9.869532643e-01f, 9.219682877e-03f, 4.794137181e-02f, 1.150486629e-01f,
     2.063410229e-01f, 3.160842505e-01f, 4.373832957e-01f, 5.626167043e-01f, 6.839157495e-01f, 7.936589771e-01f,
     8.849513371e-01f, 9.520586282e-01f, 9.907803171e-01f, 5.299532504e-03f, 2.771248846e-02f, 6.718439881e-02f,
     1.222977958e-01f, 1.910618778e-01f, 2.709916112e-01f, 3.591982246e-01f, 4.524937451e-01f, 5.475062549e-01f,
     6.408017754e-01f, 7.290083888e-01f, 8.089381222e-01f, 8.777022042e-01f, 9.328156012e-01f, 9.722875115e-01f,
     9.947004675e-01f, 3.435700407e-03f, 1.801403636e-02f, 4.388278587e-02f, 8.044151409e-02f, 1.268340468e-01f,
     1.819731596e-01f, 2.445664990e-01f, 3.131469556e-01f, 3.861070744e-01f, 4.617367394e-01f, 5.382632606e-01f,
     6.138929256e-01f, 6.868530444e-01f, 7.554335010e-01f, 8.180268404e-01f, 8.731659532e-01f, 9.195584859e-01f,
     9.561172141e-01f, 9.819859636e-01f, 9.965642996e-01f, 2.406390001e-03f, 1.263572201e-02f, 3.086272400e-02f,
     5.679223650e-02f, 8.999900701e-02f, 1.299379042e-01f, 1.759531740e-01f, 2.272892643e-01f, 2.831032462e-01f,
     3.424786602e-01f, 4.044405663e-01f, 4.679715536e-01f, 5.320284464e-01f, 5.955594337e-01f, 6.575213398e-01f,
     7.168967538e-01f, 7.727107357e-01f, 8.240468260e-01f, 8.700620958e-01f, 9.100009930e-01f, 9.432077635e-01f,
     9.691372760e-01f, 9.873642780e-01f, 9.975936100e-01f, 1.368069075e-03f, 7.194244227e-03f, 1.761887221e-02f,
     3.254696203e-02f, 5.183942212e-02f, 7.531619313e-02f, 1.027581020e-01f, 1.339089406e-01f, 1.684778665e-01f,
     2.061421214e-01f, 2.465500455e-01f, 2.893243619e-01f, 3.340656989e-01f, 3.803563189e-01f, 4.277640192e-01f,
     4.758461672e-01f, 5.241538328e-01f, 5.722359808e-01f, 6.196436811e-01f, 6.659343011e-01f, 7.106756381e-01f,
     7.534499545e-01f, 7.938578786e-01f, 8.315221335e-01f, 8.660910594e-01f, 8.972418980e-01f, 9.246838069e-01f,
     9.481605779e-01f, 9.674530380e-01f, 9.823811278e-01f, 9.928057558e-01f, 9.986319309e-01f},
    {1.000000000e+00f, 5.000000000e-01f, 5.000000000e-01f, 2.777777778e-01f, 4.444444444e-01f, 2.777777778e-01f,
     1.739274226e-01f, 3.260725774e-01f, 3.260725774e-01f, 1.739274226e-01f, 1.184634425e-01f, 2.393143352e-01f,
     2.844444444e-01f, 2.393143352e-01f, 1.184634425e-01f, 8.566224619e-02f, 1.803807865e-01f, 2.339569673e-01f,
     2.339569673e-01f, 1.803807865e-01f, 8.566224619e-02f, 5.061426815e-02f, 1.111905172e-01f, 1.568533229e-01f,
     1.813418917e-01f, 1.813418917e-01f, 1.568533229e-01f, 1.111905172e-01f, 5.061426815e-02f, 3.333567215e-02f,
     7.472567458e-02f, 1.095431813e-01f, 1.346333597e-01f, 1.477621124e-01f, 1.477621124e-01f, 1.346333597e-01f,
     1.095431813e-01f, 7.472567458e-02f, 3.333567215e-02f, 2.358766819e-02f, 5.346966300e-02f, 8.003916427e-02f,
     1.015837134e-01f, 1.167462683e-01f, 1.245735229e-01f, 1.245735229e-01f, 1.167462683e-01f, 1.015837134e-01f,
     8.003916427e-02f, 5.346966300e-02f, 2.358766819e-02f, 1.357622971e-02f, 3.112676197e-02f, 4.757925584e-02f,
     6.231448563e-02f, 7.479799441e-02f, 8.457825970e-02f, 9.130170752e-02f, 9.472530523e-02f, 9.472530523e-02f,
     9.130170752e-02f, 8.457825970e-02f, 7.479799441e-02f, 6.231448563e-02f, 4.757925584e-02f, 3.112676197e-02f,
     1.357622971e-02f, 8.807003570e-03f, 2.030071490e-02f, 3.133602417e-02f, 4.163837079e-02f, 5.096505991e-02f,
     5.909726598e-02f, 6.584431922e-02f, 7.104805466e-02f, 7.458649324e-02f, 7.637669357e-02f, 7.637669357e-02f,
     7.458649324e-02f, 7.104805466e-02f, 6.584431922e-02f, 5.909726598e-02f, 5.096505991e-02f, 4.163837079e-02f,
     3.133602417e-02f, 2.030071490e-02f, 8.807003570e-03f, 6.170614900e-03f, 1.426569431e-02f, 2.213871941e-02f,
     2.964929246e-02f, 3.667324071e-02f, 4.309508077e-02f, 4.880932605e-02f, 5.372213506e-02f, 5.775283403e-02f,
     6.083523646e-02f, 6.291872817e-02f, 6.396909767e-02f, 6.396909767e-02f, 6.291872817e-02f, 6.083523646e-02f,
     5.775283403e-02f, 5.372213506e-02f, 4.880932605e-02f, 4.309508077e-02f, 3.667324071e-02f, 2.964929246e-02f,
     2.213871941e-02f, 1.426569431e-02f, 6.170614900e-03f, 3.509305005e-03f, 8.137197365e-03f, 1.269603265e-02f,
     1.713693146e-02f, 2.141794901e-02f, 2.549902963e-02f, 2.934204674e-02f, 3.291111139e-02f, 3.617289705e-02f,
     3.909694789e-02f, 4.165596211e-02f, 4.382604650e-02f, 4.558693935e-02f, 4.692219954e-02f, 4.781936004e-02f,
     4.827004426e-02f, 4.827004426e-02f, 4.781936004e-02f, 4.692219954e-02f, 4.558693935e-02f, 4.382604650e-02f,
     4.165596211e-02f, 3.909694789e-02f, 3.617289705e-02f, 3.291111139e-02f, 2.934204674e-02f, 2.549902963e-02f,
     2.141794901e-02f, 1.713693146e-02f, 1.269603265e-02f, 8.137197365e-03f, 3.509305005e-03f},
    {0, 1, 3, 6, 10, 15, 21, 29, 39, 51, 67, 87, 111},
    {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32}};

// One row of k: exponent factor q, log2 of the weight as an integer and a fraction in [0, 1),
// and the visit's index in its table.
struct GqRow {
    float q, wfrac, wint;
    int vis;
};

// Where rows of k and records come from: the visits [0, n_vis) of a scan at one time (T, TAU),
// or the lags n_vis .. 1 of a uniform scan (T == NULL: visit i has age n_vis - i, dwell 1).
// Visits [vb[b], vb[b + 1]) take band b, from row k_off on; those from vb[kGqBands] on get
// records (RecF32) from rec_off on.
struct GqTable {
    const double *T, *TAU;
    double s, kappa, tdim;
    int64_t vis_off, k_off, rec_off;
    int n_vis, n_fp16;              // visits, and how many of them, the oldest, take FP16 pieces
    int vb[kGqBands + 1];
};
// A grid of points: columns x0 + c dx, rows y0 + r dy [m] (one product, one sum), as float-float
// pairs in pitch units at ax + ax_off (W columns, then H rows).
struct GqGrid {
    double x0, y0, dx, dy, inv_pitch;
    int64_t ax_off;
    int W, H;
};

// One snapshot of one scan on one grid.
struct GqJob {
    const float4 *srcF;             // the scan's visits, float-float pairs in pitch units
    int64_t ax_off;                 // axes of the grid
    int W, H;
    int tw, n_tc;                   // contraction tiles: tw columns (a multiple of 16) x 128 rows
    int shift;                      // visit of a table visit i: i - shift
    int r0, r1;                     // recent visits [r0, r1): the CUDA cores' part
    int nq;                         // partial rows to sum up (the contraction's, then others' recent visits)
    int row;                        // out_off < 0: the partial row that takes this job's recent visits
    int64_t rec0;                   // record of visit r0
    int64_t t_off, t_stride;        // first partial row, row stride (floats)
    int64_t out_off;                // < 0: a segment of lags (below), summed by its group, or a part of
                                    // another job's recent visits
    double pref;
};

// On a raster with a uniform dwell, the visit at lag l of snapshot M lies at the same offset from
// the beam for every M of one phase M mod nx: a field at two such snapshots differs by a shift
// of whole rows of the scan and by the lags past the smaller one.  So a group of snapshots M_0 <
// M_1 < .. of one phase is summed in the frame of its last, on a grid that reaches (M_last - M_0)
// / nx rows of the scan further down: segment s, the lags (M_(s-1), M_s], on the rows that
// snapshots from s on look at, and out_s(r) = sum of the segments up to s at row r + shift_s.
// (64 row snapshots of 64 x 64 visits on 128 x 128 points: 1.0e8 pairs instead of 2.2e9, 127 us
// before and 78 us with it; the launches are a few pieces long, so their latency bounds it.)
struct GqSegment {
    int64_t t_off, t_stride, out_off;
    int n_part, shift, H, pad;      // partial rows; shift of its snapshot and its own height in grid rows
};
struct GqGroup {
    int64_t block0;                 // first block of the group
    int seg0, n_seg, W, H, H_ext, pad;
    double pref;
};

// One run: rows of k [k0, k0 + nk) on one tile, to partial row `row` of the job.
struct GqRun {
    int64_t k0;
    int nk, job, tile, row;
};

// warps 0-15: producers; 16: the MMAs; 17-19: coefficients; 20-23: draining
constexpr int kGqProdWarps = 16, kGqMmaWarp = 16, kGqCoefWarp = 17, kGqDrainWarp = 20;
constexpr int kGqCoefWarps = 3, kGqCoefThreads = 32 * kGqCoefWarps, kGqDrainWarps = 4;
constexpr int kGqThreads = 768;
// registers per thread: 80 at launch, moved to the draining warps
constexpr int kGqRegsProd = 64, kGqRegsMid = 48, kGqRegsDrain = 176;
static_assert(kGqRegsProd * 32 * kGqProdWarps + kGqRegsMid * 128 + kGqRegsDrain * 32 * kGqDrainWarps <= 80 * kGqThreads, "register split");
constexpr int kGqTile = 128;
constexpr int kGqStageK = 64, kGqPieceK = 384;
// K steps (16 rows of k) of a run at most: the draining warps add a run's stages of four steps in plain
// FP32, whose rounding grows with the square root of their number (3e-7 of the sum for 512)
constexpr int64_t kGqRunSteps = 4 * 512;
constexpr int kGqPieceBytes = kGqTile * kGqStageK * 2;         // one 16-bit piece of one side: 16 KB
// A stage: Y's pieces, then X's; h, l in FP16 and three stages in the ring, or h, m, l in BF16 and two.
template <bool kBf16>
struct GqForm {
    static constexpr int kPieces = kBf16 ? 3 : 2, kBufs = kBf16 ? 2 : 3;
    static constexpr int kSideBytes = kPieces * kGqPieceBytes, kBufBytes = 2 * kSideBytes;
};
constexpr int kGqRingBytes = 12 * kGqPieceBytes, kGqMaxBufs = 3;
static_assert(GqForm<false>::kBufs * GqForm<false>::kBufBytes == kGqRingBytes && GqForm<true>::kBufs * GqForm<true>::kBufBytes == kGqRingBytes, "ring");
// A piece as the warps see it.  The rings hold 8: the coefficient warps are at most two pieces
// ahead of the producers, these three stages ahead of the MMAs, and those two stages ahead of the
// draining warps.
struct GqPiece {
    float *out;                             // the tile's first sum in the run's partial row
    int W;
    int nk, nc, nr;                         // rows of k, the tile's columns and rows
    int first, last, final;                 // of the run; final: the CTA's last piece
    float scale;                            // of the products: 2^m (BF16), 2^(m - 28) (FP16)
};
struct GqSmem {
    unsigned char bufs[kGqRingBytes];
    float4 a[2][2][kGqPieceK / 2];          // [piece parity][side]: (-x, -x', -q, -q') of two rows of k
    float2 e[2][2][kGqPieceK / 2];          // exponent offsets; side 0: rows, 1: columns
    float2 pos[2][2][kGqTile];              // [run parity][side]: offsets of the tile's rows, columns
    GqPiece piece[8];
    float wmax[kGqCoefWarps];
    int2 stage_info[8];                     // piece ring slot + 8 x first + 16 x last stage of the
                                            // piece, rows of k
    uint64_t cfull[2], cempty[2], full[kGqMaxBufs], empty[kGqMaxBufs], done[2], free1[2], free2[2], idle;
    uint32_t tmem;
    int failed;
};
// What the tensor core's accumulation of a full stage drops, put back by halves of an FP32 ulp: its two
// accumulator sets take these factors in turn.  (Stages of fewer steps lose less than half an ulp.)
template <bool kBf16>
__device__ __forceinline__ float gq_unbias(int set) {
    return kBf16 ? (set ? 1.0f + 0x1p-23f : 1.0f) : (set ? 1.0f + 0x1p-22f : 1.0f + 0x1p-23f);
}
constexpr float kGqFarExp = 150.0f;         // q rho^2 from which a row of k is left out
constexpr int kGqSmemBytes = (int)sizeof(GqSmem) + 1024;
static_assert(kGqSmemBytes <= 227 * 1024, "shared memory of a CTA");

// set when a wait of the contraction gives up (its partial sums are then NaN)
static __device__ int g_grid_quad_timeout;

__device__ __forceinline__ uint32_t f16x2_rn(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float2 f16x2_to_f2(uint32_t w) {
    float2 f;
    asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %2;\n cvt.f32.f16 %0, l;\n cvt.f32.f16 %1, h;\n}\n"
        : "=f"(f.x), "=f"(f.y) : "r"(w));
    return f;
}
__device__ __forceinline__ uint32_t bf16x2_rn(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// v - the rounded pair w, exact (mixed-precision multiply-add)
__device__ __forceinline__ float2 bf16x2_rest(uint32_t w, float2 v) {
    float2 r;
    asm("{\n .reg .b16 x, y, n;\n mov.b32 {x, y}, %2;\n mov.b16 n, 0xBF80;\n"
        " fma.rn.f32.bf16 %0, x, n, %3;\n fma.rn.f32.bf16 %1, y, n, %4;\n}\n"
        : "=f"(r.x), "=f"(r.y) : "r"(w), "f"(v.x), "f"(v.y));
    return r;
}
// instruction descriptor of kind::f16: FP32 accumulator, FP16 A and B, both K-major
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void gq_mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void gq_coef_sync() { asm volatile("bar.sync 1, %0;" :: "n"(kGqCoefThreads) : "memory"); }
__device__ __forceinline__ bool gq_coef_all(bool v) {
    int r;
    asm volatile("{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n barrier.cta.red.and.pred q, 1, %2, p;\n selp.b32 %0, 1, 0, q;\n}\n"
                 : "=r"(r) : "r"((int)v), "n"(kGqCoefThreads) : "memory");
    return r != 0;
}
// Wait for the phase of the given parity: at most 2^18 probes that may suspend the thread for up
// to 1 us each (about 0.26 s).  False, with *failed set, if the wait gave up or another one had.
__device__ __forceinline__ bool gq_wait(uint64_t *bar, uint32_t parity, volatile int *failed) {
    const uint32_t addr = smem_u32(bar);
    for (int it = 0; it < (1 << 18); ++it) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (done) return true;
        if (*failed) return false;
    }
    *failed = 1;
    return false;
}
// the same for a whole warp: one answer
__device__ __forceinline__ bool gq_wait_warp(uint64_t *bar, uint32_t parity, volatile int *failed) {
    return __all_sync(0xffffffffu, gq_wait(bar, parity, failed));
}

// v 2^n for a float above the denormals; a zero turns into 2^(n - 127), which the FP16
// conversion rounds back to zero.  (On the integer pipe: the FMA pipe is the busier one.)
__device__ __forceinline__ float gq_scale(float v, int n) { return __int_as_float(__float_as_int(v) + (n << 23)); }

// Factors of 8 rows of k at one position, as 16-byte core-matrix rows one piece apart (FP16: h, -l;
// BF16: h, m, l).  a: (-x, -x', -q, -q') of four pairs of rows of k, e: their exponent offsets; the
// position is din + dfr (kSplit: dfr is added last, else the sum is in din).
template <bool kSplit, bool kBf16>
__device__ __forceinline__ void gq_factors(const float4 (&a)[4], const float2 (&e)[4], float din, float dfr,
                                           unsigned char *dst) {
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        float2 d = __fadd2_rn(f2(din, din), f2(a[u].x, a[u].y));
        if (kSplit) d = __fadd2_rn(d, f2(dfr, dfr));
        const float2 g = __ffma2_rn(f2(a[u].z, a[u].w), __fmul2_rn(d, d), e[u]);
        if (kBf16) {
            const float2 F = f2(ex2_approx(g.x), ex2_approx(g.y));
            h[u] = bf16x2_rn(F.x, F.y);
            const float2 r = bf16x2_rest(h[u], F);
            m[u] = bf16x2_rn(r.x, r.y);
            const float2 q = bf16x2_rest(m[u], r);
            l[u] = bf16x2_rn(q.x, q.y);
        } else {
            const float F0 = gq_scale(ex2_approx(g.x), 14), F1 = gq_scale(ex2_approx(g.y), 14);
            h[u] = f16x2_rn(F0, F1);
            // h - F, exact (mixed-precision subtraction)
            float r0, r1;
            asm("{\n .reg .b16 x, y;\n mov.b32 {x, y}, %2;\n sub.rn.f32.f16 %0, x, %3;\n sub.rn.f32.f16 %1, y, %4;\n}\n"
                : "=f"(r0), "=f"(r1) : "r"(h[u]), "f"(F0), "f"(F1));
            l[u] = f16x2_rn(gq_scale(r0, 11), gq_scale(r1, 11));
        }
    }
    *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
    if (kBf16) {
        *reinterpret_cast<uint4 *>(dst + kGqPieceBytes) = make_uint4(m[0], m[1], m[2], m[3]);
        *reinterpret_cast<uint4 *>(dst + 2 * kGqPieceBytes) = make_uint4(l[0], l[1], l[2], l[3]);
    } else {
        *reinterpret_cast<uint4 *>(dst + kGqPieceBytes) = make_uint4(l[0], l[1], l[2], l[3]);
    }
}
// The same for the positions of mask (bit q: din[q]), the coefficients read once.
template <bool kBf16>
__device__ __forceinline__ void gq_group(const float4 *as, const float2 *es, const float (&din)[4], const float (&dfr)[4],
                                         bool split, uint32_t mask, unsigned char *dst) {
    float4 a[4];
    float2 e[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        a[u] = as[u];
        e[u] = es[u];
    }
    if (split) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (mask & (1u << q)) gq_factors<true, kBf16>(a, e, din[q], dfr[q], dst + 512 * q);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (mask & (1u << q)) gq_factors<false, kBf16>(a, e, din[q], 0.0f, dst + 512 * q);
    }
}

// withhold (tests): no MMA is issued and no accumulator set is committed, so that the waits run
// out.
template <bool kBf16>
__global__ void __launch_bounds__(kGqThreads, 1)
grid_quad_kernel(const GqJob *__restrict__ jobs, const GqRun *__restrict__ runs, const int *__restrict__ cta_off,
                 const GqRow *__restrict__ rows, const float2 *__restrict__ ax, float *__restrict__ partial,
                 int withhold) {
    constexpr int kGqBufs = GqForm<kBf16>::kBufs, kGqBufBytes = GqForm<kBf16>::kBufBytes, kGqSideBytes = GqForm<kBf16>::kSideBytes;
    extern __shared__ unsigned char gq_raw[];
    GqSmem &sm = *reinterpret_cast<GqSmem *>((reinterpret_cast<uintptr_t>(gq_raw) + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == kGqMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" :: "r"(smem_u32(&sm.tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        if (lane == 0) {
            for (int k = 0; k < 2; ++k) {
                mbar_init(sm.cfull + k, kGqCoefWarps);
                mbar_init(sm.cempty + k, kGqProdWarps);
                mbar_init(sm.done + k, 1);
                mbar_init(sm.free1 + k, kGqDrainWarps);
                mbar_init(sm.free2 + k, kGqDrainWarps);
            }
            for (int k = 0; k < kGqBufs; ++k) {
                mbar_init(sm.full + k, kGqProdWarps);
                mbar_init(sm.empty + k, 1);
            }
            mbar_init(&sm.idle, 1);
            sm.failed = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // columns [0, 256): the leading products, by stage; [256, 512): the rest, by piece; two of each
    const uint32_t tmem = sm.tmem;
    volatile int *const failed = &sm.failed;
    // A role whose wait gives up leaves its loop; so do the others at their next wait, and the
    // draining warps write NaN to all of the CTA's sums.
    if (warp < kGqProdWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kGqRegsProd));
        // ---- the producers: warp = 8 rows of k of the row side (warps 0-7) or the column side
        const int side = warp >> 3, kg = warp & 7;
        unsigned char *const dst0 = sm.bufs + side * kGqSideBytes + kg * (kGqTile * 16) + lane * 16;
        int stage = 0, run = -1;
        float din[4], dfr[4];
        bool split = false;
        uint32_t mask = 0;                   // position groups of 32 that hold points
        for (int piece = 0;; ++piece) {
            bool ok = gq_wait_warp(sm.cfull + (piece & 1), (uint32_t)(piece >> 1) & 1u, failed);
            if (!ok) break;
            const GqPiece &P = sm.piece[piece & 7];
            const int nk = P.nk;
            if (P.first) {
                ++run;
                mask = (1u << (((side ? P.nc : P.nr) + 31) >> 5)) - 1u;
                bool exact = true;           // the offsets fit one FP32 number to 2^-28 pitch
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 v = sm.pos[run & 1][side][lane + 32 * q];
                    din[q] = v.x;
                    dfr[q] = v.y;
                    exact = exact && fabsf(((v.x + v.y) - v.x) - v.y) <= 3.7e-9f;
                }
                split = !__all_sync(0xffffffffu, exact);
                if (!split) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) din[q] += dfr[q];
                }
            }
            for (int k0 = 0; k0 < nk; k0 += kGqStageK, ++stage) {
                const int b = stage % kGqBufs;
                if (stage >= kGqBufs) ok = gq_wait_warp(sm.empty + b, (uint32_t)(stage / kGqBufs - 1) & 1u, failed);
                if (!ok) break;
                if (tid == 0)
                    sm.stage_info[stage & 7] = make_int2((piece & 7) + (k0 == 0 ? 8 : 0) + (nk - k0 <= kGqStageK ? 16 : 0),
                                                         min(nk - k0, kGqStageK));
                if (k0 + 8 * kg < ((nk + 15) & ~15))
                    gq_group<kBf16>(&sm.a[piece & 1][side][(k0 + 8 * kg) / 2], &sm.e[piece & 1][side][(k0 + 8 * kg) / 2], din, dfr,
                             split, mask, dst0 + b * kGqBufBytes);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) gq_mbar_arrive(sm.full + b);
            }
            if (!ok) break;
            const int final = P.final;
            __syncwarp();
            if (lane == 0) gq_mbar_arrive(sm.cempty + (piece & 1));
            if (final) break;
        }
    } else if (warp < kGqDrainWarp) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kGqRegsMid));
        if (warp == kGqMmaWarp) {
        // ---- the MMA thread
        if (lane == 0) {
            const uint64_t desc0 = umma_smem_desc(smem_u32(sm.bufs), kGqTile * 16, 128u);
            int piece = -1;
            for (int stage = 0;; ++stage) {
                const int b = stage % kGqBufs, set = stage & 1;
                if (!gq_wait(sm.full + b, (uint32_t)(stage / kGqBufs) & 1u, failed)) break;
                const int2 info = sm.stage_info[stage & 7];
                const GqPiece &P = sm.piece[info.x & 7];
                const int nc = (P.nc + 15) & ~15;
                const uint32_t idesc = kBf16 ? umma_idesc_bf16(kGqTile, nc) : umma_idesc_f16(kGqTile, nc);
                const bool fresh = info.x & 8, final = (info.x & 16) && P.final;
                if (fresh) {
                    ++piece;
                    if (piece >= 2 && !gq_wait(sm.free2 + (piece & 1), (uint32_t)((piece >> 1) - 1) & 1u, failed)) break;
                }
                if (stage >= 2 && !gq_wait(sm.free1 + set, (uint32_t)((stage >> 1) - 1) & 1u, failed)) break;
                tc_fence_after();
                const uint32_t d1 = tmem + 128u * set, d2 = tmem + 256u + 128u * (piece & 1);
                // descriptors count in 16 bytes; a K step is two groups of 8 rows of k
                const uint64_t y = desc0 + (uint64_t)(b * (kGqBufBytes / 16));
                constexpr uint64_t kP = kGqPieceBytes / 16, kX = kGqSideBytes / 16, kStep = 2 * kGqTile;
                const int steps = withhold ? 0 : (info.y + 15) / 16;
#pragma unroll
                for (int k = 0; k < kGqStageK / 16; ++k)
                    if (k < steps) {
                        const uint64_t yk = y + k * kStep, xk = yk + kX;
                        umma_bf16(d1, yk, xk, idesc, k > 0 ? 1 : 0);
                        umma_bf16(d2, yk, xk + kP, idesc, k > 0 || !fresh ? 1 : 0);
                        umma_bf16(d2, yk + kP, xk, idesc, 1);
                        if (kBf16) {
                            umma_bf16(d2, yk + kP, xk + kP, idesc, 1);
                            umma_bf16(d2, yk, xk + 2 * kP, idesc, 1);
                            umma_bf16(d2, yk + 2 * kP, xk, idesc, 1);
                        }
                    }
                if (!withhold) umma_commit(sm.done + set);
                umma_commit(sm.empty + b);
                if (final) break;
            }
            // no MMA in flight when the tensor memory is given back
            umma_commit(&sm.idle);
            int never = 0;
            gq_wait(&sm.idle, 0u, &never);
        }
        __syncwarp();
        } else {
        // ---- the coefficients: four rows of k per thread
        const int t = tid - 32 * kGqCoefWarp, cw = warp - kGqCoefWarp;
        const int run0 = cta_off[blockIdx.x], run1 = cta_off[blockIdx.x + 1];
        constexpr int kPer = kGqPieceK / kGqCoefThreads;
        int piece = 0;
        bool ok = true;
        for (int r = run0; r < run1 && ok; ++r) {
            const GqRun run = runs[r];
            const GqJob &J = jobs[run.job];
            const int W = J.W, shift = J.shift;
            const int c0 = (run.tile % J.n_tc) * J.tw, q0 = (run.tile / J.n_tc) * kGqTile;
            const int nc = min(J.tw, W - c0), nr = min(kGqTile, J.H - q0);
            const float4 *const srcF = J.srcF;
            const float2 *const axx = ax + J.ax_off + c0, *const axy = ax + J.ax_off + W + q0;
            float *const out = partial + J.t_off + (int64_t)run.row * J.t_stride + (int64_t)q0 * W + c0;
            // coordinates as integer offsets from the integer grid position nearest the tile's
            // first point plus fractions (visits are integers): dx within one rounding
            const float ox = rintf(axx[0].x), oy = rintf(axy[0].x);
            float x_a = (axx[0].x - ox) + axx[0].y, x_b = (axx[nc - 1].x - ox) + axx[nc - 1].y;
            float y_a = (axy[0].x - oy) + axy[0].y, y_b = (axy[nr - 1].x - oy) + axy[nr - 1].y;
            if (x_a > x_b) { const float v = x_a; x_a = x_b; x_b = v; }
            if (y_a > y_b) { const float v = y_a; y_a = y_b; y_b = v; }
            for (int kk = 0; kk < run.nk; kk += kGqPieceK, ++piece) {
                const int nk = min(kGqPieceK, run.nk - kk), par = piece & 1;
                float q[kPer], vx[kPer], vy[kPer], wf[kPer], g[kPer], p[kPer];
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const int k = t + u * kGqCoefThreads;
                    q[u] = vx[u] = vy[u] = wf[u] = p[u] = 0.0f;
                    g[u] = -INFINITY;
                    if (k < nk) {
                        const GqRow w = rows[run.k0 + kk + k];
                        const float4 v = srcF[w.vis - shift];
                        vx[u] = (v.x - ox) + v.y;
                        vy[u] = (v.z - oy) + v.w;
                        q[u] = w.q;
                        wf[u] = w.wfrac;
                        g[u] = w.wint;
                    }
                }
                // p = floor(q dxmin^2) moves from the row factor's exponent to the column
                // factor's; m: the piece's largest row exponent.  A row of k whose term is below
                // the FP32 range at every point of the tile (w < 2, so 2^-150 is) turns into
                // padding: its exponents would be differences of numbers that FP32 no longer
                // holds to within one, and its factors could pass FP16's range.
                float m = -3e38f;
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const float dx = fmaxf(0.0f, fmaxf(x_a - vx[u], vx[u] - x_b));
                    const float dy = fmaxf(0.0f, fmaxf(y_a - vy[u], vy[u] - y_b));
                    const float ex = q[u] * (dx * dx), ey = q[u] * (dy * dy);
                    if (!(ex + ey <= kGqFarExp)) {
                        q[u] = vx[u] = vy[u] = wf[u] = 0.0f;
                        g[u] = -INFINITY;
                        continue;
                    }
                    p[u] = floorf(ex);
                    g[u] -= p[u];
                    m = fmaxf(m, floorf(fmaxf(g[u] + wf[u] - ey, -3e30f)));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                // (one answer for the three warps: they share barriers)
                if (piece >= 2) ok = gq_wait(sm.cempty + par, (uint32_t)((piece >> 1) - 1) & 1u, failed);
                if (lane == 0) sm.wmax[cw] = m;
                ok = gq_coef_all(ok);
                if (!ok) break;
                m = fmaxf(fmaxf(sm.wmax[0], sm.wmax[1]), sm.wmax[2]);
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const int k = t + u * kGqCoefThreads, j = k >> 1, o = k & 1;
                    float *const a0 = reinterpret_cast<float *>(&sm.a[par][0][j]), *const a1 = reinterpret_cast<float *>(&sm.a[par][1][j]);
                    a0[o] = -vy[u]; a0[2 + o] = -q[u];
                    a1[o] = -vx[u]; a1[2 + o] = -q[u];
                    // rows of k past the piece: -inf, a zero row factor
                    reinterpret_cast<float *>(&sm.e[par][0][j])[o] = wf[u] + (g[u] - m);
                    reinterpret_cast<float *>(&sm.e[par][1][j])[o] = p[u];
                }
                if (kk == 0) {
                    for (int i = t; i < 2 * kGqTile; i += kGqCoefThreads) {
                        const int s = i >> 7, c = i & (kGqTile - 1);
                        const float2 v = s ? axx[min(c, nc - 1)] : axy[min(c, nr - 1)];
                        const float n = rintf(v.x);
                        sm.pos[(r - run0) & 1][s][c] = f2(n - (s ? ox : oy), (v.x - n) + v.y);
                    }
                }
                if (t == 0) {                // the scale is 0 below the FP32 normal range
                    const int ex = (int)fmaxf(m, -1000.0f) - (kBf16 ? 0 : 28);
                    sm.piece[piece & 7] = GqPiece{out, W, nk, nc, nr, kk == 0, kk + kGqPieceK >= run.nk,
                                                  kk + kGqPieceK >= run.nk && r + 1 == run1,
                                                  ex > -127 ? __int_as_float((ex + 127) << 23) : 0.0f};
                }
                __syncwarp();
                if (lane == 0) gq_mbar_arrive(sm.cfull + par);
                gq_coef_sync();              // wmax may be written again
            }
        }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(kGqRegsDrain));
        // ---- the draining warps: warp covers rows 32 quarter .. of the tile, lane = row
        const int quarter = warp & 3;
        const uint32_t base = tmem + ((uint32_t)(32 * quarter) << 16);
        int piece = 0;
        float acc[kGqTile];
#pragma unroll
        for (int c = 0; c < kGqTile; ++c) acc[c] = 0.0f;
        for (int stage = 0;; ++stage) {
            const int set = stage & 1;
            if (!gq_wait_warp(sm.done + set, (uint32_t)(stage >> 1) & 1u, failed)) break;
            tc_fence_after();
            const int2 stage_info = sm.stage_info[stage & 7];
            const int info = stage_info.x;
            const GqPiece &P = sm.piece[info & 7];
            const int nc = P.nc;
            const float scale = P.scale;
            // acc += scale * (the accumulator at column d)
            auto drain = [&](uint32_t d, float f) {
#pragma unroll
                for (int cb = 0; cb < kGqTile; cb += 32)
                    if (cb < nc) {
                        uint32_t v[32];
                        tmem_ld_32x32b<32>(base + d + (uint32_t)cb, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[cb + e] = fmaf(__uint_as_float(v[e]), f, acc[cb + e]);
                    }
                tc_fence_before();
                __syncwarp();
            };
            drain(128u * set, stage_info.y > kGqStageK - 16 ? scale * gq_unbias<kBf16>(set) : scale);
            if (lane == 0) gq_mbar_arrive(sm.free1 + set);
            if (!(info & 16)) continue;
            drain(256u + 128u * (piece & 1), kBf16 ? scale : scale * (-1.0f / 2048.0f));   // FP16: of -l
            const int last = P.last, final = P.final, nr = P.nr, W = P.W;
            float *const out = P.out + (int64_t)(32 * quarter + lane) * W;
            __syncwarp();
            if (lane == 0) gq_mbar_arrive(sm.free2 + (piece & 1));
            ++piece;
            if (!last) continue;
            // the run's sums: each lane its row
            if (32 * quarter + lane < nr) {
                if ((W & 3) == 0) {          // the tile's first column and the row stride are, too
#pragma unroll
                    for (int c = 0; c < kGqTile; c += 4)
                        if (c < nc) *reinterpret_cast<float4 *>(out + c) = make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
                } else {
#pragma unroll
                    for (int c = 0; c < kGqTile; ++c)
                        if (c < nc) out[c] = acc[c];
                }
            }
            __syncwarp();
            if (final) break;
#pragma unroll
            for (int c = 0; c < kGqTile; ++c) acc[c] = 0.0f;
        }
        if (__any_sync(0xffffffffu, *failed)) {
            for (int r = cta_off[blockIdx.x]; r < cta_off[blockIdx.x + 1]; ++r) {
                const GqRun run = runs[r];
                const GqJob &J = jobs[run.job];
                const int c0 = (run.tile % J.n_tc) * J.tw, q = (run.tile / J.n_tc) * kGqTile + 32 * quarter + lane;
                float *const out = partial + J.t_off + (int64_t)run.row * J.t_stride + (int64_t)q * J.W + c0;
                for (int c = 0; q < J.H && c < min(J.tw, J.W - c0); ++c) out[c] = __int_as_float(0x7FC00000);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && *failed) atomicExch(&g_grid_quad_timeout, 1);
    if (warp == kGqMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" :: "r"(tmem) : "memory");
}

__device__ __forceinline__ int gq_segment(const int64_t *__restrict__ offs, int n, int64_t g) {
    int lo = 0, hi = n - 1;                  // largest k with offs[k] <= g
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (offs[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// One thread per record, then one per table visit (its rows of k), then one per axis entry, each
// range from a whole warp on.  Bound by the latency of a record's serial chain and by FP64
// divisions.  q = q1 log2(e) e^(L u) comes from the FP64 q1 as a float-float pair and expm1.
struct GqPrep {
    const GqTable *tabs;
    const int64_t *rec_offs, *vis_offs, *ax_offs;
    const GqGrid *grids;
    int64_t n_rec, n_vis, n_ax;
    int n_tabs, n_grids;
    GqRow *rows;
    RecF32 *rec;
    float2 *ax;
};
__host__ __device__ inline int64_t gq_warps(int64_t n) { return (n + 31) / 32 * 32; }
__global__ void __launch_bounds__(64) grid_quad_prep_kernel(const GqPrep P) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < gq_warps(P.n_rec)) {
        if (g >= P.n_rec) return;
        const GqTable &S = P.tabs[gq_segment(P.rec_offs, P.n_tabs, g)];
        const int i = S.vb[kGqBands] + (int)(g - S.rec_off);
        const double dT = S.T ? S.tdim - S.T[i] : (double)(S.n_vis - i), tau = S.T ? S.TAU[i] : 1.0;
        double q1, dq, r, ell;
        pair_geometry<RecTraits<RecF32>::kFP64Ell>(dT, tau, S.s, S.kappa, q1, dq, r, ell);
        RecF32 out;
        RecTraits<RecF32>::fill(out, q1, dq, r, ell);
        P.rec[g] = out;
        return;
    }
    g -= gq_warps(P.n_rec);
    if (g >= gq_warps(P.n_vis)) {
        const int64_t a = g - gq_warps(P.n_vis);
        if (a >= P.n_ax) return;
        const GqGrid &G = P.grids[gq_segment(P.ax_offs, P.n_grids, a)];
        const int64_t i = a - G.ax_off;
        const double v = i < G.W ? __dadd_rn(__dmul_rn((double)i, G.dx), G.x0)
                                 : __dadd_rn(__dmul_rn((double)(i - G.W), G.dy), G.y0);
        const double x = v * G.inv_pitch;
        const float hi = (float)x;
        P.ax[a] = make_float2(hi, (float)(x - (double)hi));
        return;
    }
    if (g >= P.n_vis) return;
    const GqTable &S = P.tabs[gq_segment(P.vis_offs, P.n_tabs, g)];
    const int i = (int)(g - S.vis_off);
    if (i >= S.vb[kGqBands]) return;
    int b = 0;
    int64_t k = S.k_off;
    for (; b < kGqBands - 1 && i >= S.vb[b + 1]; ++b) k += (int64_t)(S.vb[b + 1] - S.vb[b]) * kGqRule.nodes[b];
    const int n = kGqRule.nodes[b], o = kGqRule.first[b];
    k += (int64_t)(i - S.vb[b]) * n;
    // the dwell is over: w0 = w1 - 4 kappa tau
    const double dT = S.T ? S.tdim - S.T[i] : (double)(S.n_vis - i), tau = S.T ? S.TAU[i] : 1.0;
    const double w1 = 2.0 * S.s + 4.0 * S.kappa * dT, w0 = 2.0 * S.s + 4.0 * S.kappa * (dT - tau);
    const double inv = 1.0 / (w0 * w1);
    const double q1 = 1.44269504088896340736 * (w0 * inv);
    const float L = log1pf((float)((4.0 * S.kappa * tau) * (w1 * inv)));
    const float qh = (float)q1, ql = (float)(q1 - (double)qh);
    for (int j = 0; j < n; ++j) {
        const float w = L * kGqRule.c[o + j];
        const int bits = __float_as_int(w);
        GqRow out;
        out.q = qh + fmaf(qh, expm1f(L * kGqRule.u[o + j]), ql);
        out.wint = (float)((bits >> 23) - 127);
        out.wfrac = log2f(__int_as_float((bits & 0x7FFFFF) | 0x3F800000));
        out.vis = i;
        P.rows[k + j] = out;
    }
}

// The recent visits at a tile of 32 columns x 16 rows (lane = column, warp = 4 rows), each at the
// cheapest series that holds it over the warp's points (the classes of the field kernel), at most
// kGqFinMost of them in one plain FP32 sum, plus the partial rows of the contraction and of earlier
// recent visits, in compensated FP32; out = pref times that.  Bound by the series' issue for many recent
// visits, by the partial rows' loads for few.
constexpr int kGqFinRows = 16, kGqFinThreads = 128, kGqFinStage = 32;
// More than kGqFinSplit recent visits of a job are split into parts of kGqFinVisits while the GPU has
// places for their CTAs: a CTA walks 0.15 us per visit, so that 65,536 of them on 64 x 64 points (8
// CTAs) took 9.8 ms in one piece each and take 0.36 ms split.  Fewer stay in one piece: a second
// launch and its fork cost the host 20 us (256 visits, 16 x 16 points, 256 snapshots: 64 us, split 85).
// More than kGqFinMost (16 stages) always are, so that no plain sum grows longer: over 2048 stages it
// rounds to 7e-7; a compensated sum in the loop instead took 2 us of 47 on the 16 x 16 case.
constexpr int kGqFinSplit = 256, kGqFinVisits = 64, kGqFinMost = 512, kGqFinResident = 8;    // CTAs per SM
__global__ void __launch_bounds__(kGqFinThreads, kGqFinResident)
grid_quad_final_kernel(const GqJob *__restrict__ jobs, const int64_t *__restrict__ tile_offs, int n_jobs,
                       const RecF32 *__restrict__ rec, const float2 *__restrict__ ax, float *partial,
                       double *__restrict__ out) {
    __shared__ float s_vx[kGqFinStage], s_vy[kGqFinStage];
    __shared__ __align__(16) RecF32 s_rec[kGqFinStage];
    const int64_t q = blockIdx.x;
    const int j = gq_segment(tile_offs, n_jobs, q);
    const GqJob J = jobs[j];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_tc = (J.W + 31) / 32, t = (int)(q - tile_offs[j]);
    const int c = (t % n_tc) * 32 + lane, row0 = (t / n_tc) * kGqFinRows + 4 * warp;
    const float2 *const axx = ax + J.ax_off, *const axy = axx + J.W;
    const float2 vx0 = axx[(t % n_tc) * 32], vy0 = axy[(t / n_tc) * kGqFinRows];
    const float ox = rintf(vx0.x), oy = rintf(vy0.x);
    const float2 px = axx[min(c, J.W - 1)];
    const float xi = rintf(px.x), xin = xi - ox, xfr = (px.x - xi) + px.y;
    float2 yin[2], yfr[2];
    float by0 = 3e38f, by1 = -3e38f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 py = axy[min(row0 + k, J.H - 1)];
        const float yi = rintf(py.x), a = yi - oy, f = (py.x - yi) + py.y;
        if (k & 1) { yin[k >> 1].y = a; yfr[k >> 1].y = f; } else { yin[k >> 1].x = a; yfr[k >> 1].x = f; }
        by0 = fminf(by0, a + f);
        by1 = fmaxf(by1, a + f);
    }
    float bx0 = xin + xfr, bx1 = bx0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        bx0 = fminf(bx0, __shfl_xor_sync(0xffffffffu, bx0, o));
        bx1 = fmaxf(bx1, __shfl_xor_sync(0xffffffffu, bx1, o));
    }
    float2 run[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
    for (int v0 = J.r0; v0 < J.r1; v0 += kGqFinStage) {
        const int cnt = min(kGqFinStage, J.r1 - v0);
        __syncthreads();
        if (tid < cnt) {
            const float4 v = J.srcF[v0 + tid];
            s_vx[tid] = (v.x - ox) + v.y;                // probe positions are integers
            s_vy[tid] = (v.z - oy) + v.w;
        }
        {
            const float4 *const src = reinterpret_cast<const float4 *>(rec + J.rec0 + (v0 - J.r0));
            float4 *const dst = reinterpret_cast<float4 *>(s_rec);
            for (int k = tid; k < cnt * (int)(sizeof(RecF32) / 16); k += kGqFinThreads) dst[k] = src[k];
        }
        __syncthreads();
        uint32_t code = kCodeSkip;                       // staged visit `lane` against the warp's box
        if (lane < cnt) {
            float r2min, r2max;
            box_rho2(s_vx[lane], s_vy[lane], bx0, bx1, by0, by1, r2min, r2max);
            const float4 v1 = s_rec[lane].v1;
            code = series_class(r2max * v1.y, r2min * v1.z, v1.y);
        }
        float2 acc[4] = {f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f)};   // [0], [1] used
        for (uint32_t m = __ballot_sync(0xffffffffu, code != kCodeSkip); m; m &= m - 1) {
            const int s = __ffs(m) - 1;
            const uint32_t cl = __shfl_sync(0xffffffffu, code, s);
            const RecF32 &R = s_rec[s];
            const float dx = (xin - s_vx[s]) + xfr, vy = s_vy[s];
            float r2[4];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float2 dy = __fadd2_rn(__fadd2_rn(yin[k], f2(-vy, -vy)), yfr[k]);
                const float2 d2 = __fmul2_rn(dy, dy);
                r2[2 * k] = fmaf(dx, dx, d2.x);
                r2[2 * k + 1] = fmaf(dx, dx, d2.y);
            }
            if (cl <= kCodeD4) {
                const float4 w0 = R.v0;
                const float g4 = R.v1.x;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const float2 r = f2(r2[2 * k], r2[2 * k + 1]);
                    float2 e = __ffma2_rn(f2(g4, g4), r, f2(w0.w, w0.w));
                    e = __ffma2_rn(e, r, f2(w0.z, w0.z));
                    e = __ffma2_rn(e, r, f2(w0.y, w0.y));
                    e = __ffma2_rn(e, r, f2(w0.x, w0.x));
                    acc[k] = __fadd2_rn(acc[k], f2(ex2_approx(e.x), ex2_approx(e.y)));
                }
            } else if (cl == kCodeD8) {
                point_pass_h2<8, 4>(acc, r2, R);
            } else if (cl == kCodeD12) {
                point_pass_h2<12, 4>(acc, r2, R);
            } else {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    acc[k].x += pair_term(r2[2 * k], R);
                    acc[k].y += pair_term(r2[2 * k + 1], R);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) run[k] = __fadd2_rn(run[k], acc[k]);
    }
    if (c >= J.W || row0 >= J.H) return;
    const int nr = min(4, J.H - row0);
    if (J.out_off < 0) {                     // the recent visits as a partial row
        float *const o = partial + J.t_off + J.row * J.t_stride + (int64_t)row0 * J.W + c;
        const float v[4] = {run[0].x, run[0].y, run[1].x, run[1].y};
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (e < nr) o[(int64_t)e * J.W] = v[e];
        return;
    }
    BlockSum<float> sum[4];
    const float *const p = partial + J.t_off + (int64_t)row0 * J.W + c;
#pragma unroll 2
    for (int k = 0; k < J.nq; ++k) {
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = e < nr ? __ldcg(p + k * J.t_stride + (int64_t)e * J.W) : 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) sum[e].add(v[e]);
    }
    sum[0].add(run[0].x);
    sum[1].add(run[0].y);
    sum[2].add(run[1].x);
    sum[3].add(run[1].y);
    double *const o = out + J.out_off + (int64_t)row0 * J.W + c;
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (e < nr) o[(int64_t)e * J.W] = J.pref * sum[e].value();
}

// Running sums over the segments of the groups: thread = a point of the group's tall grid (32
// columns x 4 rows per block).  Bound by the latency of the segments' loads, two rounds of which
// are in flight (26 us on 64 segments with four loads in flight, 21 us with these), and the stores.
constexpr int kGqShiftSegs = 64, kGqShiftAhead = 8;
__global__ void __launch_bounds__(128)
grid_quad_shift_kernel(const GqGroup *__restrict__ groups, int n_groups, const GqSegment *__restrict__ segs,
                       const float *__restrict__ partial, double *__restrict__ out) {
    __shared__ GqSegment s_seg[kGqShiftSegs];
    int k = 0;
    while (k + 1 < n_groups && groups[k + 1].block0 <= blockIdx.x) ++k;
    const GqGroup G = groups[k];
    const int n_tc = (G.W + 31) / 32, t = (int)(blockIdx.x - G.block0);
    const int c = (t % n_tc) * 32 + (threadIdx.x & 31), R = (t / n_tc) * 4 + (threadIdx.x >> 5);
    const int64_t p = (int64_t)R * G.W + c;
    BlockSum<float> acc;
    for (int s0 = 0; s0 < G.n_seg; s0 += kGqShiftSegs) {
        const int n = min(kGqShiftSegs, G.n_seg - s0);
        __syncthreads();
        for (int i = threadIdx.x; i < n * (int)(sizeof(GqSegment) / 8); i += 128)
            reinterpret_cast<int64_t *>(s_seg)[i] = reinterpret_cast<const int64_t *>(segs + G.seg0 + s0)[i];
        __syncthreads();
        if (c >= G.W) continue;
        // the first two partial rows of kGqShiftAhead segments in flight while the last ones are added
        constexpr int A = kGqShiftAhead;
        float v[A][2], w[A][2];
        auto load = [&](int i, float (&x)[A][2]) {
#pragma unroll
            for (int e = 0; e < A; ++e) {
                const GqSegment &S = s_seg[min(i + e, n - 1)];
                const int m = i + e < n && R < S.H ? S.n_part : 0;
                const float *const q = partial + S.t_off + p;
                x[e][0] = m > 0 ? __ldcg(q) : 0.0f;
                x[e][1] = m > 1 ? __ldcg(q + S.t_stride) : 0.0f;
            }
        };
        load(0, v);
        for (int i = 0; i < n; i += A) {
            load(i + A, w);
#pragma unroll
            for (int e = 0; e < A; ++e) {
                if (i + e >= n) break;
                const GqSegment &S = s_seg[i + e];
                if (R >= S.H) continue;
                acc.add(v[e][0]);
                acc.add(v[e][1]);
                for (int q = 2; q < S.n_part; ++q) acc.add(__ldcg(partial + S.t_off + q * S.t_stride + p));
                const int r = R - S.shift;
                if (r >= 0 && r < G.H) out[S.out_off + (int64_t)r * G.W + c] = G.pref * acc.result();
            }
#pragma unroll
            for (int e = 0; e < A; ++e) { v[e][0] = w[e][0]; v[e][1] = w[e][1]; }
        }
    }
}

}  // namespace ddk
