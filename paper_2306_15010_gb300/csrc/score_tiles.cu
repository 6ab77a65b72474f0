// Eq. 2 score over tiles of windows, visiting only the clusters that both images hold there.
//
// A warp owns a tile of 32 NX x TY windows.  For a rectangle of the bank and a cluster j, let t be
// the template's count and n the count of a window of the query.  Then
//     sum_j |t_j - n_j| = area + sum_{t_j > 0} t_j - 2 sum_{t_j > 0} min(t_j, n_j)
// (every query pixel carries one label, so sum_j n_j = area), and min(t_j, n_j) = 0 for every
// window of the tile when the rectangle, swept over the tile, meets no pixel labelled j.  A
// four-corner sum of the integral image over the swept region, rounded out to the coarse samples,
// tells; a sum of zero is proof, so skipping is exact.  Labels are piecewise constant: on the
// 2048 x 2048, k = 128 workload with a 128 x 128 template about 95 of the 1,280 (rectangle,
// cluster) pairs of a 64 x 4 tile remain, against 486 that the template's counts alone leave.  The
// other two bank forms use the same test with the box of a grid or a filter: a cluster that is
// absent adds |t|.
//
// What bounds it: instruction issue and the corner rows' way from L2 into shared memory, in that
// order (ncu, 2048 x 2048: 70 % and 60 % of peak before the pair list, 2.3 KB per pair and tile).
// Tiles of 64 x 4 windows with three staged pairs take 0.43 ms there, 12 blocks to an SM (18.9 KB of
// shared memory each, 80 registers); with 72 registers, and 20 bytes of spills, for 14 blocks that
// shared memory does not hold 0.45, with 96 for 10 blocks 0.46 ms.  64 x 8
// took 0.46 to 0.51, 128 x 4 0.52, 32 x 4 0.54 ms, two staged pairs 0.49 ms, loads from global memory
// straight into registers 0.48 ms and more, a table laid out by 64-column strips the same.  The
// dense kernel (sat_score.cu: every cluster, staged for 512 windows) takes 1.13 ms.  Testing against
// the full-size table (a gather from 32 planes per corner) cost 0.34 ms by itself, against the
// coarse samples 0.06 ms; they leave 101 pairs where the exact region leaves 93.
#include "common.cuh"
#include "ptx.cuh"
#include "score_spec.cuh"

namespace vqnnf {
namespace {

constexpr int TW = 2;              // warps per block, their tiles side by side in x
constexpr int NST = 3;             // staged pairs of a warp

// The integral image, element (y, j, x) at (y * k + j) * P + x, and its coarse samples.
template <typename T>
struct Sat {
    const T *S, *coarse;
    int P, k, ccols, kp;
};

// The clusters that the region [x0, x1) x [y0, y1) of the image, rounded out to the coarse
// samples, holds.
template <typename T>
struct Region {
    const T *p00, *p01, *p10, *p11;
    __device__ __forceinline__ Region(const Sat<T> &s, int x0, int y0, int x1, int y1)
    {
        const int cx0 = x0 / kCoarseX, cx1 = (x1 + kCoarseX - 1) / kCoarseX;
        const T *top = s.coarse + (size_t)(y0 / kCoarseY) * s.ccols * s.kp;
        const T *bot = s.coarse + (size_t)((y1 + kCoarseY - 1) / kCoarseY) * s.ccols * s.kp;
        p00 = top + (size_t)cx0 * s.kp, p01 = top + (size_t)cx1 * s.kp;
        p10 = bot + (size_t)cx0 * s.kp, p11 = bot + (size_t)cx1 * s.kp;
    }
    // bit u: cluster j + u, j a multiple of 4
    __device__ __forceinline__ unsigned holds4(int j) const
    {
        struct __align__(4 * sizeof(T)) Four { T v[4]; };
        const Four a = *reinterpret_cast<const Four *>(p11 + j), b = *reinterpret_cast<const Four *>(p10 + j);
        const Four c = *reinterpret_cast<const Four *>(p01 + j), d = *reinterpret_cast<const Four *>(p00 + j);
        unsigned h = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) h |= (box<T>(a.v[u], b.v[u], c.v[u], d.v[u]) != 0 ? 1u : 0u) << u;
        return h;
    }
};

// Whether the count of a region of w x h pixels, rounded out, stays below the table's modulus (one
// that could reach it is not tested: every cluster is visited).
template <typename T>
__host__ __device__ inline bool testable(int w, int h)
{
    return sizeof(T) > 2 || (long long)(w + 2 * (kCoarseX - 1)) * (h + 2 * (kCoarseY - 1)) <= 65535;
}

// The clusters a tile visits, as bits: word g = 4 G + u, bit b is cluster 128 G + 4 b + u (a lane
// reads four clusters' samples at once).  Here: those that the region holds, or every one where
// the region is not tested.
template <typename T>
__device__ __forceinline__ void visit_words(unsigned *act, int k, bool test, const Region<T> &reg)
{
    const int lane = threadIdx.x & 31;
    for (int j0 = 0; j0 < k; j0 += 128) {
        const int j = j0 + 4 * lane;
        const unsigned h = j >= k ? 0u : test ? reg.holds4(j) : 15u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned m = __ballot_sync(0xffffffffu, j + u < k && ((h >> u) & 1u));
            if (lane == 0) act[j0 / 32 + u] = m;
        }
    }
}
__device__ __forceinline__ int word_cluster(int w, unsigned m) { return 128 * (w >> 2) + 4 * (__ffs(m) - 1) + (w & 3); }
__device__ __forceinline__ int words_of(int k) { return (k + 127) / 128 * 4; }

// Corner rows and columns of a grid bank's slot: cell q, or the full window (q = G G).
struct Slot {
    int x0, x1, y0, y1;
    __device__ __forceinline__ Slot(const GridSpec &gs, int q)
    {
        const int G = gs.G;
        const bool full = q == G * G;
        x0 = gs.bx[full ? 0 : q % G], x1 = gs.bx[full ? G : q % G + 1];
        y0 = gs.by[full ? 0 : q / G], y1 = gs.by[full ? G : q / G + 1];
    }
};

__device__ __forceinline__ void warp_argmax(unsigned long long best, unsigned long long *amax)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
        best = other > best ? other : best;
    }
    if ((threadIdx.x & 31) == 0 && best) atomicMax(amax, best);
}

// Writes this lane's column of the tile, its first `rows` rows; the larger of `best` and its values' keys.
template <int TY>
__device__ __forceinline__ unsigned long long put_tile(const float (&hs)[TY], int X, int Y0, int WO,
                                                       float *__restrict__ heat, unsigned long long best, int rows = TY)
{
    if (X < WO) {
#pragma unroll
        for (int r = 0; r < TY; ++r) {
            if (r >= rows) break;                            // uniform
            const unsigned idx = (unsigned)((Y0 + r) * WO + X);
            heat[idx] = -hs[r];
            const unsigned long long key = pack_key(-hs[r], idx);
            best = key > best ? key : best;
        }
    }
    return best;
}

// Grid bank: the shape of a warp's tile and of one staged pair: the four corner blocks of TY rows,
// each row 32 NX columns from a 16-byte boundary on.
template <typename T, int NX, int TY>
struct GridTile {
    static constexpr int E = 16 / (int)sizeof(T);            // elements of a 16-byte chunk
    static constexpr int CPR = 32 * NX / E + 1;              // chunks per row
    static constexpr int NCH = 4 * TY * CPR;                 // chunks per pair
    static constexpr int PER = (NCH + 31) / 32;              // per lane
    static constexpr int STAGE = NCH * 16;
};
// A pair to visit: slot, cluster and template count.  Where the table is 16-bit no window's count
// exceeds 65,535, so a larger template count (a caller's own) gives the same minimum cut to that.
template <typename T> struct PairOf;
template <> struct PairOf<uint16_t> {
    uint32_t v;
    PairOf() = default;
    __device__ __forceinline__ PairOf(int q, int j, int t) : v((uint32_t)min(t, 65535) << 16 | (uint32_t)q << 8 | (uint32_t)j) {}
    __device__ __forceinline__ int t() const { return (int)(v >> 16); }
    __device__ __forceinline__ int q() const { return (int)(v >> 8 & 255u); }
    __device__ __forceinline__ int j() const { return (int)(v & 255u); }
};
template <> struct PairOf<uint32_t> {
    uint2 v;
    PairOf() = default;
    __device__ __forceinline__ PairOf(int q, int j, int t) : v(make_uint2((uint32_t)q << 8 | (uint32_t)j, (uint32_t)t)) {}
    __device__ __forceinline__ int t() const { return (int)v.y; }
    __device__ __forceinline__ int q() const { return (int)(v.x >> 8); }
    __device__ __forceinline__ int j() const { return (int)(v.x & 255u); }
};
constexpr int kGridY = 4;         // window rows of a grid bank's tile, 64 wide
constexpr int kPairs = 512;        // a warp's list: at least the pairs of four slots of 128 clusters

// `test`: the slots whose region is tested.
template <typename T, int NX, int TY>
__global__ void __launch_bounds__(32 * TW, sizeof(T) == 2 ? 12 : 1) score_grid_tile_kernel(Sat<T> sat, int HO, int WO, GridSpec gs, unsigned test,
                                                                  float *__restrict__ heat, ScoreAux *aux,
                                                                  long long dense_from)
{
    using L = GridTile<T, NX, TY>;
    ptx::pdl_enter();
    if (aux->probe > dense_from) return;                     // the dense kernel takes this image
    __shared__ __align__(16) uint8_t stage_s[TW][NST][L::STAGE];
    __shared__ PairOf<T> list_s[TW][kPairs];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int nslot = gs.G * gs.G + gs.full, k = sat.k;
    const int X0 = ((int)blockIdx.x * TW + wi) * 32 * NX;
    if (X0 >= WO) return;                                    // uniform over the warp
    const int Y0 = min((int)blockIdx.y * TY, HO - TY);       // the last tile moves up to stay whole
    const int xe = min(X0 + 32 * NX - 1, WO - 1);            // last window column of the tile
    PairOf<T> *list = list_s[wi];
    // the tile's rows start here; offsets from it in 16-byte units stay below 2^32 (checked on the host)
    const uint4 *S16 = reinterpret_cast<const uint4 *>(sat.S + (size_t)Y0 * k * sat.P);
    const uint32_t plane16 = (uint32_t)(sat.P / L::E);
    uint32_t off[L::PER];                                    // this lane's chunks of a slot
    float hs[NX][TY];
    int acc[NX][TY];
#pragma unroll
    for (int c = 0; c < NX; ++c)
#pragma unroll
        for (int r = 0; r < TY; ++r) hs[c][r] = 0.f, acc[c][r] = 0;
    auto fold = [&](int q) {                                  // H = - sum_q coef_q L1_q, slot by slot
        const float coef = gs.slot_coef[q];
        const int base = gs.slot_area[q] + aux->tsum[q];
#pragma unroll
        for (int c = 0; c < NX; ++c)
#pragma unroll
            for (int r = 0; r < TY; ++r) {
                hs[c][r] = fmaf(coef, (float)(base - 2 * acc[c][r]), hs[c][r]);
                acc[c][r] = 0;
            }
    };
    const uint32_t st0 = ptx::smem_u32(stage_s[wi][0]) + lane * 16;
    const T *sm = reinterpret_cast<const T *>(stage_s[wi][0]) + lane;
    int q = 0, da = 0, db = 0;                               // slot; its columns' places in their staged rows
    bool entered = false;
    auto visit = [&](int n) {
        int iq = -1, ib = 0;
        auto issue = [&](int p) {
            if (p < n) {
                const PairOf<T> e = list[p];
                if (e.q() != iq) {
                    iq = e.q();
                    const Slot sl(gs, iq);
                    const int xa = (X0 + sl.x0) & ~(L::E - 1), xb = (X0 + sl.x1) & ~(L::E - 1);
#pragma unroll
                    for (int i = 0; i < L::PER; ++i) {
                        const int idx = lane + 32 * i, row = idx / L::CPR, ch = idx % L::CPR;
                        const int blk = row / TY, r = row % TY;   // blocks: top a, top b, bottom a, bottom b
                        const int x = min(((blk & 1) ? xb : xa) + ch * L::E, sat.P - L::E);
                        const int y = ((blk & 2) ? sl.y1 : sl.y0) + r;
                        off[i] = (uint32_t)y * (uint32_t)k * plane16 + (uint32_t)(x / L::E);
                    }
                }
                const uint4 *src = S16 + (uint32_t)e.j() * plane16;
                const uint32_t dst = st0 + (uint32_t)ib * L::STAGE;
#pragma unroll
                for (int i = 0; i < L::PER; ++i)
                    if (32 * i + 32 <= L::NCH || lane + 32 * i < L::NCH) ptx::cp16(dst + 32 * 16 * i, src + off[i]);
            }
            ptx::cp_commit();
            ib = ib + 1 < NST ? ib + 1 : 0;
        };
#pragma unroll
        for (int p = 0; p < NST - 1; ++p) issue(p);
        int b = 0;
        for (int p = 0; p < n; ++p) {
            ptx::cp_wait<NST - 2>();
            __syncwarp();                                    // every lane's copies have landed, the oldest buffer is read
            issue(p + NST - 1);
            const PairOf<T> e = list[p];
            if (e.q() != q || !entered) {
                while (q < e.q()) fold(q++);
                entered = true;
                const Slot sl(gs, q);
                da = (X0 + sl.x0) & (L::E - 1);
                db = (X0 + sl.x1) & (L::E - 1);
            }
            const int t = e.t();
            constexpr int RP = L::CPR * L::E;                // elements between rows
            const T *ta = sm + b * (L::STAGE / (int)sizeof(T)) + da, *tb = sm + b * (L::STAGE / (int)sizeof(T)) + db;
#pragma unroll
            for (int c = 0; c < NX; ++c)
#pragma unroll
                for (int r = 0; r < TY; ++r)
                    acc[c][r] += min(t, box<T>(tb[(3 * TY + r) * RP + 32 * c], ta[(2 * TY + r) * RP + 32 * c],
                                               tb[(TY + r) * RP + 32 * c], ta[r * RP + 32 * c]));
            b = b + 1 < NST ? b + 1 : 0;
        }
        __syncwarp();                                        // the list may be rewritten
    };
    // the clusters to visit, four words' samples in flight at a time: four slots of at most 128
    // clusters, or two of more
    constexpr int QB = 4;
    const int two = k > 128, qb = QB >> two;
    int n = 0;
    for (int q0 = 0; q0 < nslot; q0 += qb) {
        unsigned h[QB];
        int4 t[QB];
#pragma unroll
        for (int i = 0; i < QB; ++i) {
            const int s = min(q0 + (i >> two), nslot - 1), j = 128 * (i & two) + 4 * lane;
            const Slot sl(gs, s);
            const Region<T> reg(sat, X0 + sl.x0, Y0 + sl.y0, xe + sl.x1, Y0 + TY - 1 + sl.y1);
            h[i] = j >= k || q0 + (i >> two) >= nslot ? 0u : (test >> s) & 1 ? reg.holds4(j) : 15u;
            t[i] = *reinterpret_cast<const int4 *>(&aux->t[s][j]);
        }
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < QB; ++i) {
            h[i] &= (t[i].x > 0 ? 1u : 0u) | (t[i].y > 0 ? 2u : 0u) | (t[i].z > 0 ? 4u : 0u) | (t[i].w > 0 ? 8u : 0u);
            cnt += __popc(h[i]);
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (n + cnt > kPairs) {
            __syncwarp();
            visit(n);
            n = 0;
        }
#pragma unroll
        for (int i = 0; i < QB; ++i) {
            const int s = q0 + (i >> two), j = 128 * (i & two) + 4 * lane;
            const int tv[4] = {t[i].x, t[i].y, t[i].z, t[i].w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned m = __ballot_sync(0xffffffffu, (h[i] >> u) & 1u);
                if ((h[i] >> u) & 1u) list[n + __popc(m & ((1u << lane) - 1u))] = PairOf<T>(s, j + u, tv[u]);
                n += __popc(m);
            }
        }
    }
    __syncwarp();
    visit(n);
    while (q < nslot) fold(q++);
    unsigned long long best = 0ull;
#pragma unroll
    for (int c = 0; c < NX; ++c) best = put_tile<TY>(hs[c], X0 + 32 * c + lane, Y0, WO, heat, best);
    warp_argmax(best, &aux->amax);
}

// Weighted-grid bank (WGridSpec): grid by grid, the clusters present in the grid's box add
// |t - R|, R the filter's integer weighting of the cell counts, to a filter's sum of the other
// clusters' |t|.  Where every filter weights whole columns or whole rows of cells (the Gaussian and
// Haar filters with equal bin weights: SEP), the three column and three row counts come from the 12
// corners on the box's edge; otherwise the nine cell counts from all 16.
// Bound by the copies: a staged (grid, cluster) is 16 rows, each the 32 columns at every boundary or all
// columns between, eight lanes to a row, so that an instruction's copies lie in few lines.  Calls on a
// 720 x 1280 query with every cluster in every window (k = 128, the paper's 15 filters, templates of
// 110 x 100 to 110 x 250): 1.45 to 1.63 ms at any width; whole rows alone, two lanes each, 1.68 to 2.84 ms;
// the kernel that visited every cluster for 512 windows 2.41 to 2.49 ms.  Labels in 12-pixel cells with
// 2 % noise 1.19 to 1.45, 1.37 to 2.51 ms.  32-bit table (700 x 100 to 700 x 250 template, 900 x 800 query,
// k = 64) 0.33 to 0.39, 0.41 to 0.69 and 0.47 ms.  With exponential bin weights (all 16 corners) 1.72 to
// 1.88, 2.03 to 2.70 and 2.42 to 2.50 ms; 0.33 to 0.40, 0.40 to 0.70 and 0.48 ms.
constexpr int kWY = 4;             // tile: 32 x kWY windows
constexpr int WNST = 2;
// A staged pair: kWY rows for each boundary row a, then the pair's template counts.  A row has room for
// the 32 columns at each boundary column that is read (SEP: the outer two alone in the box's inner rows),
// each from a 16-byte boundary on; or it holds all columns from the first boundary's to the last's,
// where these are fewer.
template <typename T, bool SEP>
struct WTile {
    static constexpr int E = 16 / (int)sizeof(T);              // elements of a 16-byte chunk
    static constexpr int CPR = (32 + E - 2) / E + 1;           // chunks per row
    static constexpr int R0 = 4 * CPR, R1 = SEP ? 2 * CPR : R0;   // chunks of an outer and of an inner row
    static constexpr int NCH = 2 * kWY * (R0 + R1);            // chunks per pair
    static constexpr int STAGE = NCH * 16 + 32;
    // first chunk of boundary row a, tile row r
    __host__ __device__ static constexpr int row(int a, int r)
    {
        return a == 0 ? r * R0 : a == 3 ? kWY * (R0 + 2 * R1) + r * R0 : kWY * (R0 + (a - 1) * R1) + r * R1;
    }
    // chunks of all columns of a grid `w` columns wide
    __device__ static __forceinline__ int whole(int w) { return (w + 30 + E) / E + 1; }
};

template <typename T, bool SEP>
__global__ void __launch_bounds__(32 * TW) score_wgrid_tile_kernel(Sat<T> sat, int HO, int WO, WGridSpec ws, unsigned test,
                                                                   const int32_t *__restrict__ tcounts,
                                                                   float *__restrict__ heat, unsigned long long *amax,
                                                                   const long long *probe)
{
    using L = WTile<T, SEP>;
    constexpr int E = L::E, TY = kWY;
    ptx::pdl_enter();
    if (sizeof(T) == 4 && probe && *probe > 0) return;       // the dense kernel takes this image
    __shared__ __align__(16) uint8_t stage_s[TW][WNST][L::STAGE];
    __shared__ uint16_t list_s[TW][kMaxWGrids * kMaxK];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int k = sat.k, NG = ws.NG;
    const int X0 = ((int)blockIdx.x * TW + wi) * 32;
    if (X0 >= WO) return;
    const int rows = min(TY, HO);                            // fewer window rows than a tile: the last one repeated
    const int Y0 = min((int)blockIdx.y * TY, HO - rows);
    const int xe = min(X0 + 31, WO - 1);
    uint16_t *list = list_s[wi];                             // grid << 8 | cluster, grid by grid
    int n = 0;
    for (int g = 0; g < NG; ++g) {
        const Region<T> reg(sat, X0 + ws.bx[g][0], Y0 + ws.by[g][0], xe + ws.bx[g][3], Y0 + rows - 1 + ws.by[g][3]);
        for (int j0 = 0; j0 < k; j0 += 128) {
            const int j = j0 + 4 * lane;
            const unsigned h = j >= k ? 0u : (test >> g) & 1 ? reg.holds4(j) : 15u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool v = j + u < k && ((h >> u) & 1u);
                const unsigned m = __ballot_sync(0xffffffffu, v);
                if (v) list[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(g << 8 | (j + u));
                n += __popc(m);
            }
        }
    }
    __syncwarp();
    // the tile's rows start here; offsets from it in 16-byte units stay below 2^32 (checked on the host)
    const uint4 *S16 = reinterpret_cast<const uint4 *>(sat.S + (size_t)Y0 * k * sat.P);
    const uint32_t plane16 = (uint32_t)(sat.P / E);
    // Eight lanes copy a row (of one a), chunk c, c + 8, ..: an instruction's four rows lie in few lines.
    // The last chunks may end past the table's row, and past the table by less than its slack.
    const int c = lane & 7, r0 = lane >> 3;
    S16 += X0 / E + (uint32_t)min(r0, rows - 1) * (uint32_t)k * plane16 + c;
    const uint32_t st0 = ptx::smem_u32(stage_s[wi][0]) + 16 * c;
    int ig = -1, ib = 0, cw = 0;                             // grid of the copies, the chunks of its whole rows
    int nfg = 0;                                             // its filters, and this lane's filter's counts
    const int32_t *tcf = tcounts;
    uint32_t ya[4], xq[4];                                   // its boundary rows and columns, in chunks
    auto issue = [&](int p) {
        if (p < n) {
            const int g = list[p] >> 8, j = list[p] & 255;
            if (g != ig) {
                ig = g;
                cw = L::whole(ws.bx[g][3] - ws.bx[g][0]);
                nfg = ws.nf[g];
                tcf = tcounts + (size_t)ws.filt[g][min(lane, kMaxWFilters - 1)] * k;
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    ya[a] = (uint32_t)ws.by[g][a] * (uint32_t)k * plane16;
                    xq[a] = (uint32_t)(ws.bx[g][a] / E);
                }
            }
            const uint4 *src = S16 + (uint32_t)j * plane16;
            const uint32_t dst = st0 + (uint32_t)ib * L::STAGE;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const bool outer = a == 0 || a == 3;
                const int R = outer ? L::R0 : L::R1;
                const uint4 *from = src + ya[a];
                const uint32_t to = dst + 16 * (L::row(a, 0) + r0 * R);
                if (cw <= R) {
                    from += xq[0];
#pragma unroll
                    for (int h = 0; h < R; h += 8)
                        if (c + h < cw) ptx::cp16(to + 16 * h, from + h);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (SEP && !outer && (q == 1 || q == 2)) continue;
                        const int sg = SEP && !outer ? q / 3 : q;
#pragma unroll
                        for (int h = 0; h < L::CPR; h += 8)
                            if (c + h < L::CPR) ptx::cp16(to + 16 * (sg * L::CPR + h), from + (xq[q] + h));
                    }
                }
            }
            if (lane < nfg) ptx::cp4(dst - 16 * c + lane * 4 + 16 * L::NCH, tcf + j);
        }
        ptx::cp_commit();
        ib = ib + 1 < WNST ? ib + 1 : 0;
    };
    float hs[TY];
#pragma unroll
    for (int r = 0; r < TY; ++r) hs[r] = 0.f;
#pragma unroll
    for (int p = 0; p < WNST - 1; ++p) issue(p);
    int p = 0, b = 0;
#pragma unroll 1
    for (int g = 0; g < NG; ++g) {
        const int nf = ws.nf[g];
        int acc[kMaxWFilters][TY];                           // |t| of the clusters not visited, then |t - R| of the others
#pragma unroll
        for (int f = 0; f < kMaxWFilters; ++f) {
            int ts = 0;
            if (f < nf) {
                const int32_t *tc = tcounts + (size_t)ws.filt[g][f] * k;
                for (int j = lane; j < k; j += 32) ts += abs(tc[j]);
                for (int q = p + lane; q < n && (list[q] >> 8) == g; q += 32) ts -= abs(tc[list[q] & 255]);
                ts = __reduce_add_sync(0xffffffffu, ts);
            }
#pragma unroll
            for (int r = 0; r < TY; ++r) acc[f][r] = ts;
        }
        const int cw = L::whole(ws.bx[g][3] - ws.bx[g][0]);
        int col[4], last;                                    // places in an outer row, and of the last column in an inner row
        {
            const int x0 = X0 + ws.bx[g][0], s0 = x0 & (E - 1), s3 = (X0 + ws.bx[g][3]) & (E - 1);
            const int end = lane + ws.bx[g][3] - ws.bx[g][0] + s0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                col[q] = lane + (cw <= L::R0 ? ws.bx[g][q] - ws.bx[g][0] + s0 : q * L::CPR * E + ((X0 + ws.bx[g][q]) & (E - 1)));
            last = !SEP ? col[3] : cw <= L::R1 ? end : lane + L::CPR * E + s3;
        }
#pragma unroll 1
        for (; p < n && (list[p] >> 8) == g; ++p) {
            ptx::cp_wait<WNST - 2>();
            __syncwarp();
            issue(p + WNST - 1);
            const T *v = reinterpret_cast<const T *>(stage_s[wi][b]);
            const int *ts = reinterpret_cast<const int *>(stage_s[wi][b] + 16 * L::NCH);
            constexpr int NN = SEP ? 6 : 9;
            int m[TY][NN];                                   // column and row counts, or cell counts
            auto at = [&](int a, int q, int r) { return (int)v[L::row(a, r) * E + (q == 3 && (a == 1 || a == 2) ? last : col[q])]; };
#pragma unroll
            for (int r = 0; r < TY; ++r) {
                if (SEP) {
                    int top[4], bot[4], lft[4], rgt[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        top[i] = at(0, i, r);
                        bot[i] = at(3, i, r);
                        lft[i] = at(i, 0, r);
                        rgt[i] = at(i, 3, r);
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        m[r][i] = box<T>(bot[i + 1], bot[i], top[i + 1], top[i]);
                        m[r][3 + i] = box<T>(rgt[i + 1], lft[i + 1], rgt[i], lft[i]);
                    }
                } else {
                    int cr[4][4];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int i = 0; i < 4; ++i) cr[a][i] = at(a, i, r);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int i = 0; i < 3; ++i)
                            m[r][(a * 3 + i) % NN] = box<T>(cr[a + 1][i + 1], cr[a + 1][i], cr[a][i + 1], cr[a][i]);
                }
            }
#pragma unroll
            for (int f = 0; f < kMaxWFilters; ++f) {
                if (f >= nf) break;
                const int t = ts[f];
                if (SEP) {
                    const bool rowwise = ws.rowwise[g][f];
                    const int w0 = ws.w[g][f][0], w1 = ws.w[g][f][rowwise ? 3 : 1], w2 = ws.w[g][f][rowwise ? 6 : 2];
                    if (rowwise) {
#pragma unroll
                        for (int r = 0; r < TY; ++r)
                            acc[f][r] = (int)__sad(t, w0 * m[r][3] + w1 * m[r][4] + w2 * m[r][5], (unsigned)acc[f][r]);
                    } else {
#pragma unroll
                        for (int r = 0; r < TY; ++r)
                            acc[f][r] = (int)__sad(t, w0 * m[r][0] + w1 * m[r][1] + w2 * m[r][2], (unsigned)acc[f][r]);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < TY; ++r) {
                        int R = 0;
#pragma unroll
                        for (int i = 0; i < 9; ++i) R += ws.w[g][f][i] * m[r][i % NN];
                        acc[f][r] = (int)__sad(t, R, (unsigned)acc[f][r]);
                    }
                }
            }
            b = b + 1 < WNST ? b + 1 : 0;
        }
#pragma unroll
        for (int f = 0; f < kMaxWFilters; ++f) {
            if (f >= nf) break;
#pragma unroll
            for (int r = 0; r < TY; ++r) hs[r] = fmaf(ws.coef[g][f], (float)acc[f][r], hs[r]);
        }
    }
    warp_argmax(put_tile<TY>(hs, X0 + lane, Y0, WO, heat, 0ull, rows), amax);
}

// Any bank (weighted half-open rectangles, filter by filter): corners straight from global memory.
// Sums in 64 bits: only each filter's counts are known to fit 32.
// Bound by the corners' loads; a filter's template counts wait in shared memory, since between them the
// corners leave L1 no room (32-bit table, 1024 x 1024, k = 128, ten filters over a 200 x 400 template:
// 1.83 ms, read where they are used and their |t| added up by every lane 3.46; the kernel that staged every
// cluster for 512 windows 3.30).  Tiles of four rows share loads of neighbouring rows' lines, but
// below 13 of their warps per SM too few are in flight, and one row a warp is faster: 700 x 700, k =
// 128, 300 x 300 template (1,313 warps) 1.11 against 1.63 ms, 200 x 200, k = 32, ten filters of six
// rectangles (258) 0.40 against 0.75; 720 x 1280, k = 128, 240 x 250 template (3,993), two filters, 1.20
// against 0.79.
constexpr int kGenericWarps = 1976;   // 13 per SM
template <typename T, int TY>
__global__ void __launch_bounds__(32 * TW) score_generic_kernel(Sat<T> sat, int HO, int WO, BankSpec bs,
                                                                const int32_t *__restrict__ tcounts,
                                                                float *__restrict__ heat, unsigned long long *amax)
{
    ptx::pdl_enter();
    __shared__ unsigned act_s[TW][kMaskWords];
    __shared__ int tc_s[TW][kMaxK];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const int k = sat.k, nw = words_of(k);
    const int X0 = ((int)blockIdx.x * TW + wi) * 32;
    if (X0 >= WO) return;
    const int Y0 = min((int)blockIdx.y * TY, HO - TY);
    const int xe = min(X0 + 31, WO - 1), xl = min(X0 + lane, WO - 1);
    const size_t down = (size_t)k * sat.P;                   // one image row further
    unsigned *act = act_s[wi];
    float hs[TY];
#pragma unroll
    for (int r = 0; r < TY; ++r) hs[r] = 0.f;
    for (int f = 0; f < bs.F; ++f) {
        const int32_t *tc = tcounts + (size_t)f * k;
        int bx0 = 1 << 30, by0 = 1 << 30, bx1 = 0, by1 = 0;  // the filter's bounding box
        for (int q = bs.rect_begin[f]; q < bs.rect_begin[f + 1]; ++q) {
            bx0 = min(bx0, bs.rect[q].x0), by0 = min(by0, bs.rect[q].y0);
            bx1 = max(bx1, bs.rect[q].x1), by1 = max(by1, bs.rect[q].y1);
        }
        __syncwarp();                                        // the words of the filter before are read
        visit_words<T>(act, k, testable<T>(bx1 - bx0 + 31, by1 - by0 + TY - 1),
                       Region<T>(sat, X0 + bx0, Y0 + by0, xe + bx1, Y0 + TY - 1 + by1));
        __syncwarp();
        long long ts = 0, acc[TY];
        for (int j = lane; j < k; j += 32) {
            const int t = tc[j];
            tc_s[wi][j] = t;
            ts += abs(t);
        }
        __syncwarp();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ts += __shfl_xor_sync(0xffffffffu, ts, o);
#pragma unroll
        for (int r = 0; r < TY; ++r) acc[r] = ts;
        int w = 0;
        unsigned m = act[0];
        while (true) {
            while (m == 0 && ++w < nw) m = act[w];
            if (m == 0) break;
            const int j = word_cluster(w, m), t = tc_s[wi][j];
            m &= m - 1;
            const T *base = sat.S + ((size_t)Y0 * k + j) * sat.P + xl;
            int v[TY];
#pragma unroll
            for (int r = 0; r < TY; ++r) v[r] = 0;
            for (int q = bs.rect_begin[f]; q < bs.rect_begin[f + 1]; ++q) {
                const RectSpec &rc = bs.rect[q];
                const T *top = base + rc.y0 * down, *bot = base + rc.y1 * down;
#pragma unroll
                for (int r = 0; r < TY; ++r)
                    v[r] += rc.weight * box<T>(bot[r * down + rc.x1], bot[r * down + rc.x0], top[r * down + rc.x1],
                                               top[r * down + rc.x0]);
            }
#pragma unroll
            for (int r = 0; r < TY; ++r) acc[r] += abs(t - v[r]) - abs(t);
        }
#pragma unroll
        for (int r = 0; r < TY; ++r) hs[r] = fmaf(bs.coef[f], (float)acc[r], hs[r]);
    }
    warp_argmax(put_tile<TY>(hs, X0 + lane, Y0, WO, heat, 0ull), amax);
}

// Cost of the tile kernel less that of the dense kernel, over a sample of 64 x 4 tiles: in
// hundredths of a nanosecond on the full GPU, a visited pair costs 27 (0.244 to 0.307 ns measured
// at 2048 x 2048 on random and on coherent labels), and in the dense kernel a cluster 25 and each
// of its template-present pairs 10 (1.13 ms for 14,400 tiles of 128 clusters with 3.8 pairs each).
// One warp per (sampled tile, slot).  The warps of the first tile also leave their slot's template
// side: its counts in rows of 256, and the sum of the positive ones.
template <typename T>
__global__ void __launch_bounds__(128) score_probe_kernel(Sat<T> sat, int HO, int WO, int ntx, int nsample, int step,
                                                          GridSpec gs, unsigned test, const int32_t *__restrict__ tcounts,
                                                          ScoreAux *aux)
{
    ptx::pdl_enter();
    const int lane = threadIdx.x & 31, k = sat.k, nslot = gs.G * gs.G + gs.full;
    const int id = blockIdx.x * 4 + (threadIdx.x >> 5), q = id % nslot, i = id / nslot;
    if (i >= nsample) return;
    const long long tile = (long long)i * step;
    const int X0 = (int)(tile % ntx) * 64, Y0 = min((int)(tile / ntx) * 4, HO - 4), xe = min(X0 + 63, WO - 1);
    const Slot sl(gs, q);
    const Region<T> reg(sat, X0 + sl.x0, Y0 + sl.y0, xe + sl.x1, Y0 + 3 + sl.y1);
    const int32_t *tc = tcounts + (size_t)gs.slot_filter[q] * k;
    int present = 0, visited = 0, ts = 0;
    for (int j0 = 0; j0 < k; j0 += 128) {
        const int j = j0 + 4 * lane;
        const unsigned h = j >= k ? 0u : (test >> q) & 1 ? reg.holds4(j) : 15u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = j + u < k ? tc[j + u] : 0;
            ts += max(t, 0);
            present += t > 0;
            visited += t > 0 && ((h >> u) & 1u);
            if (i == 0) aux->t[q][j + u] = t;
        }
    }
    const int d = __reduce_add_sync(0xffffffffu, 27 * visited - 10 * present);
    ts = __reduce_add_sync(0xffffffffu, ts);
    if (lane == 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&aux->probe), (unsigned long long)(long long)d);
        if (i == 0) aux->tsum[q] = ts;
    }
}

// The same for a weighted grid over a 32-bit table: one warp per sampled 32 x 4 tile and grid.  With
// every cluster visited a pair costs a tile 0.80 to 1.35 ns, and the dense kernel 0.51 to 0.67 ns and 0.09 to
// 0.10 for every further filter of the grid (1024 x 1024 to 2048 x 2048, templates of 300 x 256 to 800 x
// 100, 1 to 5 filters a grid); `dense` has the latter, in hundredths of a nanosecond, per grid.
constexpr int kWTileCost = 110;    // of a pair that a tile visits
struct WGridCost {
    int dense[kMaxWGrids];
};
__global__ void __launch_bounds__(128) wgrid_probe_kernel(Sat<uint32_t> sat, int HO, int WO, int ntx, int nsample, int step, WGridSpec ws,
                                                          WGridCost cost, ScoreAux *aux)
{
    ptx::pdl_enter();
    const int lane = threadIdx.x & 31, k = sat.k;
    const int id = blockIdx.x * 4 + (threadIdx.x >> 5), g = id % ws.NG, i = id / ws.NG;
    if (i >= nsample) return;
    const long long tile = (long long)i * step;
    const int X0 = (int)(tile % ntx) * 32, rows = min(4, HO), Y0 = min((int)(tile / ntx) * 4, HO - rows), xe = min(X0 + 31, WO - 1);
    const Region<uint32_t> reg(sat, X0 + ws.bx[g][0], Y0 + ws.by[g][0], xe + ws.bx[g][3], Y0 + rows - 1 + ws.by[g][3]);
    int visited = 0;
    for (int j = 4 * lane; j < k; j += 128) visited += __popc(reg.holds4(j) & (k - j >= 4 ? 15u : (1u << (k - j)) - 1u));
    visited = __reduce_add_sync(0xffffffffu, visited);
    if (lane == 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(&aux->probe),
                  (unsigned long long)(long long)(kWTileCost * visited - cost.dense[g] * k));
}

// Slots whose region, swept over a tile of w x h windows, is tested.
template <typename T>
unsigned slot_tests(const GridSpec &gs, int w, int h)
{
    unsigned test = 0;
    for (int q = 0; q <= gs.G * gs.G; ++q) {
        const bool full = q == gs.G * gs.G;
        const int sw = full ? gs.bx[gs.G] : gs.bx[q % gs.G + 1] - gs.bx[q % gs.G];
        const int sh = full ? gs.by[gs.G] : gs.by[q / gs.G + 1] - gs.by[q / gs.G];
        test |= (unsigned)testable<T>(sw + w - 1, sh + h - 1) << q;
    }
    return test;
}

// A weighted-grid bank whose tiles' rows are within 32-bit offsets in 16-byte units (a table of 64 GiB or
// more under the template's rows is not; such a bank goes filter by filter).
bool wgrid_fits(const WGridSpec &ws, int k, int plane16)
{
    int h = 0;
    for (int g = 0; g < ws.NG; ++g) h = ws.by[g][3] > h ? ws.by[g][3] : h;
    return ws.NG > 0 && (long long)(h + kWY) * k * plane16 < (1ll << 32);
}

template <typename T>
unsigned wgrid_tests(const WGridSpec &ws)
{
    unsigned test = 0;
    for (int g = 0; g < ws.NG; ++g)
        test |= (unsigned)testable<T>(ws.bx[g][3] - ws.bx[g][0] + 31, ws.by[g][3] - ws.by[g][0] + kWY - 1) << g;
    return test;
}

template <typename T>
cudaError_t launch_wgrid(const Sat<T> &sat, int HO, int WO, const WGridSpec &ws, const int32_t *tc, float *heat,
                         ScoreAux *aux, cudaStream_t s)
{
    bool sep = true;
    for (int g = 0; g < ws.NG; ++g) sep = sep && ws.sep[g];
    const long long *probe = sizeof(T) == 4 && score_wgrid_probed(ws, sat.k, sat.P, HO) ? &aux->probe : nullptr;
    return launch_pdl(sep ? score_wgrid_tile_kernel<T, true> : score_wgrid_tile_kernel<T, false>,
                      dim3((WO + 32 * TW - 1) / (32 * TW), (HO + kWY - 1) / kWY), dim3(32 * TW), 0, s, sat, HO, WO, ws,
                      wgrid_tests<T>(ws), tc, heat, &aux->amax, probe);
}

template <typename T>
Sat<T> make_sat(const void *S, const void *coarse, int W, int k)
{
    return Sat<T>{static_cast<const T *>(S), static_cast<const T *>(coarse), sat_pitch(W), k, sat_coarse_cols(W),
                  sat_coarse_pitch(k)};
}

template <typename T>
cudaError_t launch_tiles_t(const Sat<T> &sat, int HO, int WO, const BankSpec &bs, const GridSpec &gs, const WGridSpec &ws,
                           const int32_t *tc, float *heat, ScoreAux *aux, long long dense_from, cudaStream_t s)
{
    unsigned long long *amax = &aux->amax;
    if (gs.G > 0)
        return launch_pdl(score_grid_tile_kernel<T, 2, kGridY>, dim3((WO + 64 * TW - 1) / (64 * TW), (HO + kGridY - 1) / kGridY), dim3(32 * TW),
                          0, s, sat, HO, WO, gs, slot_tests<T>(gs, 64, kGridY), heat, aux, dense_from);
    if (wgrid_fits(ws, sat.k, sat.P / WTile<T, true>::E)) return launch_wgrid<T>(sat, HO, WO, ws, tc, heat, aux, s);
    if (HO >= 4 && (long long)((WO + 31) / 32) * ((HO + 3) / 4) >= kGenericWarps)
        return launch_pdl(score_generic_kernel<T, 4>, dim3((WO + 32 * TW - 1) / (32 * TW), (HO + 3) / 4), dim3(32 * TW), 0, s,
                          sat, HO, WO, bs, tc, heat, amax);
    return launch_pdl(score_generic_kernel<T, 1>, dim3((WO + 32 * TW - 1) / (32 * TW), HO), dim3(32 * TW), 0, s, sat, HO, WO,
                      bs, tc, heat, amax);
}

}  // namespace

// The tile kernel needs whole tiles and 32-bit offsets between a tile's rows.  Below 512 tiles (a
// 256 x 256 query: 16 us dense, 24 us in tiles) a tile's chain of pairs is longer than the dense
// kernel's whole run, and with at most 16 clusters nearly every cluster is in every window
// (1019 x 972, k = 8: 38 us dense, 60 us in tiles); both stay dense without a probe.
ScoreRoute score_grid_route(int HO, int WO, int k, int P, int th)
{
    const long long tiles = (long long)((WO + 63) / 64) * ((HO + 3) / 4);
    const bool far = (long long)(th + 4) * k * (P / 4) >= (1ll << 32);
    return HO < 4 || k <= 16 || tiles < 512 || far ? kScoreDense : kScoreProbe;
}

// Where every filter weights whole rows or columns, three or more of them a grid, the tiles are the faster
// with every cluster visited too (300 x 256 template, 1024 x 1024, k = 64, five filters: 0.81 against 0.91
// ms), and there is no probe (3 us, and 3 for the kernel that returns).  The dense grid has a row of blocks
// per window row.
bool score_wgrid_probed(const WGridSpec &ws, int k, int P, int HO)
{
    int F = 0;
    bool sep = true;
    for (int g = 0; g < ws.NG; ++g) {
        F += ws.nf[g];
        sep = sep && ws.sep[g];
    }
    return wgrid_fits(ws, k, P / WTile<uint32_t, true>::E) && HO <= 65535 && !(sep && F >= 3 * ws.NG);
}

cudaError_t launch_wgrid_probe(const void *coarse, int W, int k, int HO, int WO, const WGridSpec &ws, ScoreAux *aux, cudaStream_t s)
{
    const int ntx = (WO + 31) / 32;
    const long long ntile = (long long)ntx * ((HO + 3) / 4);
    const int step = (int)(ntile / 509 > 1 ? (ntile / 509) | 1 : 1);      // about 500 tiles
    const int n = (int)((ntile + step - 1) / step);
    // below two blocks per SM of 512 windows each the dense kernel has too few in flight
    const bool few = (long long)HO * ((WO + 511) / 512) < 304;
    WGridCost cost;
    for (int g = 0; g < kMaxWGrids; ++g) cost.dense[g] = (45 + 10 * ws.nf[g]) * (few ? 16 : 10) / 10;
    return launch_pdl(wgrid_probe_kernel, dim3((unsigned)((n * ws.NG + 3) / 4)), dim3(128), 0, s,
                      make_sat<uint32_t>(nullptr, coarse, W, k), HO, WO, ntx, n, step, ws, cost, aux);
}

cudaError_t launch_score_probe(const void *coarse, bool u16, int W, int k, int HO, int WO, const GridSpec &gs,
                               const int32_t *tc, ScoreAux *aux, long long *dense_from, cudaStream_t s)
{
    const int ntx = (WO + 63) / 64, nslot = gs.G * gs.G + gs.full;
    const long long ntile = (long long)ntx * ((HO + 3) / 4);
    const int step = (int)(ntile / 509 > 1 ? (ntile / 509) | 1 : 1);      // about 500 tiles
    const int n = (int)((ntile + step - 1) / step);
    *dense_from = 25ll * k * n;
    const dim3 grid((unsigned)((n * nslot + 3) / 4)), block(128);
    return u16 ? launch_pdl(score_probe_kernel<uint16_t>, grid, block, 0, s, make_sat<uint16_t>(nullptr, coarse, W, k), HO, WO,
                            ntx, n, step, gs, slot_tests<uint16_t>(gs, 64, 4), tc, aux)
               : launch_pdl(score_probe_kernel<uint32_t>, grid, block, 0, s, make_sat<uint32_t>(nullptr, coarse, W, k), HO, WO,
                            ntx, n, step, gs, slot_tests<uint32_t>(gs, 64, 4), tc, aux);
}

cudaError_t launch_score_tiles(const void *S, const void *coarse, bool u16, int W, int k, int HO, int WO,
                               const BankSpec &bs, const GridSpec &gs, const WGridSpec &ws, const int32_t *tc, float *heat,
                               ScoreAux *aux, long long dense_from, cudaStream_t s)
{
    return u16 ? launch_tiles_t(make_sat<uint16_t>(S, coarse, W, k), HO, WO, bs, gs, ws, tc, heat, aux, dense_from, s)
               : launch_tiles_t(make_sat<uint32_t>(S, coarse, W, k), HO, WO, bs, gs, ws, tc, heat, aux, dense_from, s);
}

}  // namespace vqnnf
