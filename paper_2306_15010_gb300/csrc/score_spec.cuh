// Filter-bank descriptions passed to the score kernels by value (kernel parameters).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace vqnnf {

constexpr int kMaxFilters = 32;
constexpr int kMaxRects = 192;

// One weighted half-open rectangle.
struct RectSpec {
    int x0, y0, x1, y1, weight;
};

// Any bank: F filters, rectangles of filter f are rect[rect_begin[f] .. rect_begin[f+1]).
struct BankSpec {
    int F;
    int rect_begin[kMaxFilters + 1];
    RectSpec rect[kMaxRects];
    float coef[kMaxFilters];      // w_f / A_f
};

// Grid bank: the window cut by column boundaries bx[0..G] and row boundaries by[0..G]
// into G x G cells (slot r * G + c), optionally with the full window (slot G * G).  Every
// filter is one cell or the full window with weight 1.
struct GridSpec {
    int G;                        // 0 = not a grid bank
    int full;
    int F;
    int ncol;
    int bx[5];
    int by[5];
    int slot_filter[17];          // slot -> filter index
    int slot_area[17];            // pixels in the slot's rectangle
    float slot_coef[17];          // w_f / A_f of the slot's filter
    int filter_slot[kMaxFilters]; // filter index -> slot
    float coef[kMaxFilters];
};

// Weighted-grid bank: every filter is an integer weighting of the 3 x 3 cells of one of up to
// four grids (cells cut by column boundaries bx[g][0..3] and row boundaries by[g][0..3]; a
// boundary may repeat, giving empty cells), at most five filters per grid.  The coarse
// Gaussian / Haar filters of the paper at sub-scales have this form.
constexpr int kMaxWGrids = 4;
constexpr int kMaxWFilters = 5;
struct WGridSpec {
    int NG;                                   // 0 = not a weighted-grid bank
    int nf[kMaxWGrids];
    int bx[kMaxWGrids][4];
    int by[kMaxWGrids][4];
    int w[kMaxWGrids][kMaxWFilters][9];       // cell weights, cell r * 3 + c
    int filt[kMaxWGrids][kMaxWFilters];       // bank index of the filter
    float coef[kMaxWGrids][kMaxWFilters];     // w_f / A_f
    int sep[kMaxWGrids];                      // every filter of the grid has equal rows or equal columns
    int rowwise[kMaxWGrids][kMaxWFilters];    // sep: 1 = weights by row w[3 r], 0 = weights by column w[c]
};

// Coarse samples of the integral image, cluster by cluster: S at rows 0, 8, 16, .. and H and at
// columns 0, 16, 32, .. and the last, element ((row index) * columns + column index) * kp + j,
// kp = k rounded up to a multiple of 4.  One coalesced read per corner tells for many clusters
// whether a region rounded out to the samples holds them.
constexpr int kCoarseX = 16, kCoarseY = 8;
__host__ __device__ inline int sat_coarse_cols(int W) { return (W + 64) / 64 * (64 / kCoarseX) + 1; }
__host__ __device__ inline int sat_coarse_pitch(int k) { return (k + 3) / 4 * 4; }
__host__ __device__ inline int sat_coarse_rows(int H) { return (H + kCoarseY - 1) / kCoarseY + 1; }
bool sat_is_u16(int th, int tw);
int sat_pitch(int W);
int sat_strips(int W);
int sat_band_rows(int H, int W, int k);
int sat_bands(int H, int W, int k);
size_t sat_bandsum_elems(int H, int W, int k);   // workspace: at least sat_bands * k * sat_pitch, never more for a smaller image
// Tensor map of the integral image for the write pass: 32 planes x 128 bytes of one row (assign_tc.cu,
// beside the other maps).
cudaError_t make_sat_map(CUtensorMap *m, void *S, bool u16, int P, int k, int rows);
int score_ncol(int tw);
bool score_grid_fits(int ncol);   // the grid kernel stages at most TXW + 256 columns
size_t sat_slack_elems(int tw);

// The maximum's key: larger for the larger value, then for the lower window index.
__device__ __forceinline__ unsigned long long pack_key(float v, unsigned idx)
{
    unsigned b = __float_as_uint(v);
    b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);   // order-preserving
    return ((unsigned long long)b << 32) | (unsigned long long)(0xFFFFFFFFu - idx);
}
// Box count from four integral-image values; exact mod 2^16 for the 16-bit table.
template <typename T>
__device__ __forceinline__ int box(int s11, int s10, int s01, int s00)
{
    const int v = s11 - s10 - s01 + s00;
    return sizeof(T) == 2 ? (v & 0xFFFF) : v;
}

// Device words of one score: the maximum's key and the probe (both zero after launch_sat), and
// the grid bank's template side.
constexpr int kMaxSlots = 17;
struct ScoreAux {
    unsigned long long amax;
    long long probe;                              // > dense_from: the dense kernel is cheaper
    int tsum[kMaxSlots];                          // per slot: sum of the positive template counts
    alignas(16) int t[kMaxSlots][256];            // the slots' template counts
};
cudaError_t launch_sat(const uint8_t *lab, int H, int W, int k, bool u16, int *carry, int *bandsum,
                       void *S, void *coarse, ScoreAux *aux, cudaStream_t s);
cudaError_t launch_filter_responses(const uint8_t *lab, int h, int w, int k, const BankSpec &bs,
                                    int32_t *counts, cudaStream_t s);
cudaError_t launch_score(const void *S, const void *coarse, bool u16, int H, int W, int k, int HO, int WO,
                         const BankSpec &bs, const GridSpec &gs, const WGridSpec &ws, const int32_t *tc, float *heat,
                         ScoreAux *aux, int32_t *argmax_yx, cudaStream_t s);
// Which kernel scores a grid bank: the dense kernel, or the one that a probe of the image's tiles
// finds cheaper (score_tiles.cu); any other bank goes over tiles.
enum ScoreRoute { kScoreTiles, kScoreDense, kScoreProbe };
ScoreRoute score_grid_route(int HO, int WO, int k, int P, int th);
cudaError_t launch_score_probe(const void *coarse, bool u16, int W, int k, int HO, int WO, const GridSpec &gs,
                               const int32_t *tc, ScoreAux *aux, long long *dense_from, cudaStream_t s);
// Whether a weighted grid over a 32-bit table is probed, and the probe: aux->probe > 0 where the dense
// kernel is cheaper (launch_score_tiles then returns at once on the device).
bool score_wgrid_probed(const WGridSpec &ws, int k, int P, int HO);
cudaError_t launch_wgrid_probe(const void *coarse, int W, int k, int HO, int WO, const WGridSpec &ws, ScoreAux *aux, cudaStream_t s);
// A grid bank only where aux->probe <= dense_from, after the probe.
cudaError_t launch_score_tiles(const void *S, const void *coarse, bool u16, int W, int k, int HO, int WO,
                               const BankSpec &bs, const GridSpec &gs, const WGridSpec &ws, const int32_t *tc, float *heat,
                               ScoreAux *aux, long long dense_from, cudaStream_t s);
cudaError_t read_and_clear_score_error(int *out);
// One-thread kernel whose mbarrier wait gives up after limit_cycles (self-test of the bounded
// waits; sets the error word that read_and_clear_score_error returns).
cudaError_t launch_wait_selftest(long long limit_cycles, cudaStream_t s);

}  // namespace vqnnf
