// k_vote_rows.cu -- the distinct-layer Hough vote (the track path) on row
// masks.
//
// Each hit casts exactly the votes of the plain vote (Section 5 of
// arXiv:1309.6275); a cell counts the distinct detector layers among the
// hits voting in it, since a track leaves at most one hit per layer and the
// peak finder is tuned for tracks of at least seven hits (Section 7).
//
// Only the layer bits of a cell matter, so a tile keeps one bit per (layer,
// row, bin): word (l, w, j) of shared memory holds layer l's bits of the 32
// rho rows 32 w .. 32 w + 31 in d0 bin j, and one atomicOr votes in as many of
// those rows as a hit's curve spends in the bin.  A tile is one phi0 column x
// a band of 32 NWB rows x all bins x kRes layers.
//
// Along a column the root d0 of a hit falls with rho, so its curve is a run
// of rows per bin, and the runs' ends are where the curve crosses the bin
// edges: at edge d0 = d the circle equation is linear in rho, rho = -2 w /
// (w^2 + c^2) with w = d + s -- one reciprocal per bin instead of a
// reciprocal and a reciprocal square root per row.  Near the axis of the
// detector a curve spends whole words in one bin (layer at 4 cm: 0.6 bins
// over 256 rows; 27 cm: 28 bins; 74 cm: 270).
//
// A warp takes 32 hits, one per lane, computes their column constants and
// sorts them into four kinds:
//   walk  curves that keep a bin for a word of rows or more: 32 / NWB hits per
//         step, one lane per (hit, word), each lane walking its word's bins;
//   edge  steeper ones up to kEdgeSlope bins per row: 8, 16 or 32 lanes per
//         hit, a lane per bin (two beyond 32 bins), whose rows lie between its
//         own crossing and the previous lane's;
//   row   the steepest, in the A-form of tiles.cuh: one hit per step, one
//         lane per row of the hit's row window (the rows whose circles can
//         reach the axis);
//   item  the rest (rows where the second root can reach the axis or the
//         discriminant can vanish, c near 0): eval32, a lane per row.
// The first three cover the rows up to a |rho| at which the hit's first root
// is safely the only one; the rows of its window beyond that are items.  The
// warp then votes them from its own slots of shared memory: no barrier
// until the tile is complete.  Rows that float32 cannot prove go to the
// warp's redo slots and through the double-float and float64 tiers, 32 at a
// time.
//
// Why here: the tile kernel this replaces evaluated every (hit, row) of a
// column (52.7 thread instructions per vote; 29.5 lanes) and built each (hit,
// column) item three times, once per 64-row tile.  Of a 17k-hit event's 24.5k
// votes per hit, 5.0k runs of rows remain.  Issue-bound now (70% of the slots;
// 19.8k warp instructions per 10k-hit event's hit, 27.8 lanes).
// Vote stage with hit index, GB300, 25 events of 2k-60k hits (256 x 128 x 512
// cells): 18.3 -> 8.6 ms; 25 of 10k: 11.2 -> 5.3; with top-8 region sets 14.6
// -> 6.0; two of 50k (512 x 256 x 1024): 32.2 -> 17.8.  With dense layers cell by
// cell (below) the first takes 7.5 and the last 14.1.
//
// Constants, each measured on those batches: kEdgeSlope 0.5 (0.45 to 0.6
// equal, 1.0 5% slower: a steep curve has fewer rows than bins); kWalkSlope
// 1/64 (1/16 2% slower); two bins per lane beyond 32 bins (one: 10% slower);
// 3 CTAs of 320 threads (256: 4% slower, 384: 5%); kRes 10 layers resident
// keep three CTAs, and the detector has ten.
//
// Cell by cell.  Where many hits of a layer can vote in a column, going
// through them costs more than going through the column's cells, and that
// cost does not grow with the hits.  For one radius r the circle of (rho, d0)
// meets the layer at s = -S, S(rho, d0) = (rho (d0^2 + r^2) + 2 d0) / (2 (1 +
// rho d0)), so a cell holds a hit's root iff the hit's -s lies between S at
// the bin's two edges.  The index keeps each layer in azimuth order
// (k_hidx_sort) and -s is sorted along it, so an edge's place among the hits is
// a table lookup over s and a step or two along them, and the bits of 32 rows
// (a lane each) of a bin are one ballot.  Only where a bin depends on a hit
// within the error bound of an edge is that hit evaluated by the definition.
// The number of votes telescopes: per row, the hits between the axis' ends.
// A layer's rows where S is not monotone (tight curls) keep the hit-by-hit
// vote, as do sparse layers (kCellMin: 160, 300 and 500 time alike), layers
// whose radii spread, and smaller events.  kCellHits lies where the two cost the
// same: 8 events on 256 x 128 x 512 cells, cell by cell and hit by hit, of 20k
// hits 4.18 and 3.33 ms, 24k 4.30 and 3.91, 28k 4.41 and 4.55, 32k 4.53 and
// 5.20, 60k 5.40 and 9.58; two on 512 x 256 x 1024, of 20k 9.50 and 7.52, 30k
// 11.05 and 10.91, 50k 14.1 and 17.8.  (25 of 2k-60k hits: 12000 8.23 ms, 16000
// 7.83, 20000 7.52, 24000 7.43, 28000 7.50, 32000 7.41, none 8.61.)  It is bound
// by instructions (1.53 G for 3 events of 30k hits, the issue slots 69% busy).
//
// In the batch the hits come from the (layer, azimuth) index of
// k_hitindex.cu: a column scans, per layer, the run of azimuth cells whose
// hits can reach it, and a warp's hits have about the same curve, so its
// lanes walk about the same number of bins.  The single-event call has no
// scratch for an index: each tile goes through the event in the caller's
// order, and a warp's hits that can vote in it wait in shared memory until they
// fill the warp's lanes.  One event of 50k hits (512 x 256 x 1024): 20.6 -> 15.4
// ms; 20k hits (256 x 128 x 512): 1.19 -> 0.93.
#include <cooperative_groups.h>

#include "tiles.cuh"

namespace ht {
namespace {

namespace cg = cooperative_groups;

constexpr int kVrCluster = 8;         // columns whose counts one event's tiles exchange
// Threads of a tile: 320, three tiles per SM; cell by cell 512, two.  A single
// event's tiles of at most two words of rows take 256, four per SM, where three
// per SM are not one wave: 512 columns, 20k hits, 1 row 210 -> 155 us, 8 rows
// 376 -> 272, 48 rows 556 -> 469; where shared memory allows only three anyway
// (512 bins) they would lose: 646 -> 723.
constexpr int kVrThreads = 320, kClThreads = 512, kVrNarrow = 256;
constexpr int kRes = 10;              // layers resident in a tile (more: a second round)
constexpr int kKept = 16 - kRes;      // its first free place: the first round's counts, four bits
static_assert(kKept + 4 <= kRes, "the second round's layers leave room for the counts");
constexpr int kVrRedo = 96;           // redo slots per warp
constexpr int kVrPad = 4;             // words between rows of words: spreads one bin's words over banks
constexpr float kWalkSlope = 1.0f / 64.0f;   // bins per row up to which a curve is walked
constexpr float kEdgeSlope = 0.5f;    // and up to which a lane takes a bin
constexpr float kWalkEps = 8.0f;      // rows of uncertainty at a crossing
constexpr float kEdgeEps = 0.25f;     // (an edge lane's at most one row)
constexpr size_t kVrBitmap = 43 * 1024;
constexpr int kGather = 64;           // hits a single event's warp looks at per step, at most
constexpr int kClMaxHits = 4096;      // hits of a layer in a column's window, at most
constexpr int kCellMin = 160;         // and at least, to go cell by cell
constexpr int kClTab = 2048;          // table entries over a layer's s

// Where a tile's hits come from: the batch's hit index (offs set), or an
// event's arrays in the caller's order (offs null, n hits).
struct HitSource {
    const float *x, *y;
    const int *h;             // event-local hit index of a position (index only)
    const uint8_t *l;         // layer of a position
    const int *offs;
    const unsigned *rmm;
    int n;
    const int *unsorted;      // cells: layers not in azimuth order (index only)
};

struct VrSlot {
    float4 a, b;
};

// Shared memory of a tile (dynamic), in this order.
struct VrSmem {
    uint32_t *bm;             // [kRes][NWB][ND + kVrPad]
    VrSlot *slot;             // [warps][32]
    int4 *item;               // [warps][32]: item rows, layer | flags, position
    int2 *redo;               // [warps][kVrRedo]: position, row << 4 | layer
    float *sig;               // CELLS: [kClMaxHits + 1] a layer's -s, over the slots
    uint16_t *tab;            // CELLS: [kClTab] hits certainly below a bin of s
    float *rho;               // [32 NWB]
    unsigned long long *hm;   // HIT: [warps][32] region sets of the slots
    uint32_t *rowmask;        // HIT: [NWB][8] rows of the word in or next to rho block b
    uint32_t *rowblk;         // HIT: [32 NWB] rho blocks (x 8) of rows i - 1, i, i + 1
    uint8_t *jmask;           // HIT: [ND] d0 blocks of bins j - 1, j, j + 1
};

__host__ __device__ constexpr size_t vr_smem(int nwb, int nd, bool hit, bool cells, int threads)
{
    const size_t rows = (size_t)32 * nwb;
    const size_t warps = threads / 32;
    size_t b = warps * 32 * (sizeof(VrSlot) + 16) + warps * kVrRedo * 8 +
               (size_t)kRes * nwb * (nd + kVrPad) * 4 + rows * 4;
    b = (b + 15) / 16 * 16;
    if (hit) b += warps * 32 * 8 + (size_t)nwb * 32 + rows * 4 + (nd + 15) / 16 * 16;
    if (cells) b += (size_t)kClTab * 2;
    return b;
}
static_assert(kClThreads * (sizeof(VrSlot) + 16) >= (kClMaxHits + 1) * sizeof(float),
              "a layer's hits fit the slots' space");

// Words of rows per band: the largest power of two whose bitmap fits, at
// most 8 (32 rows x 8 words keep three tiles per SM at 128 bins) and no more
// than the geometry's rows need.
__host__ __device__ inline int vr_nwb(int n_rho, int nd)
{
    int nwb = 8;
    while (nwb > 1 && ((size_t)kRes * nwb * (nd + kVrPad) * 4 > kVrBitmap ||
                       (nwb / 2) * 32 >= n_rho))
        nwb /= 2;
    return nwb;
}

template <int NWB, bool HIT, bool CELLS, int kThr>
__device__ __forceinline__ VrSmem vr_carve(unsigned char *p, int nd)
{
    constexpr size_t warps = kThr / 32;
    VrSmem S{};
    // 16-byte items first: the slots, then the rest
    S.slot = reinterpret_cast<VrSlot *>(p);
    S.sig = reinterpret_cast<float *>(p);
    p += warps * 32 * sizeof(VrSlot);
    S.item = reinterpret_cast<int4 *>(p);
    p += warps * 32 * 16;
    if (HIT) {
        S.hm = reinterpret_cast<unsigned long long *>(p);
        p += warps * 32 * 8;
    }
    S.redo = reinterpret_cast<int2 *>(p);
    p += warps * kVrRedo * 8;
    S.bm = reinterpret_cast<uint32_t *>(p);
    p += (size_t)kRes * NWB * (nd + kVrPad) * 4;
    S.rho = reinterpret_cast<float *>(p);
    p += (size_t)32 * NWB * 4;
    if (CELLS) {
        S.tab = reinterpret_cast<uint16_t *>(p);
        p += (size_t)kClTab * 2;
    }
    if (HIT) {
        S.rowmask = reinterpret_cast<uint32_t *>(p);
        p += (size_t)NWB * 32;
        S.rowblk = reinterpret_cast<uint32_t *>(p);
        p += (size_t)32 * NWB * 4;
        S.jmask = p;
    }
    return S;
}

// Azimuth cells [b0, b1] of a layer's hits (radii in [rmin, rmax]) that can
// vote in a column at phik: the window of hit_cos_window, whose first angle
// grows with r and whose second falls, c > 0 bounding their sum by pi / 2;
// 4e-3 rad cover the float32 rounding (asin near 1 for argument errors below
// 5e-6 included) and that of the cells.
__device__ __forceinline__ void vote_cells(const DevGeom &G, float phik, float rmin, float rmax,
                                           bool &full, bool &empty, int &b0, int &b1)
{
    full = false;
    empty = !(rmin <= rmax);
    b0 = b1 = 0;
    if (empty) return;
    if (!(rmin >= 1e-3f)) {
        full = true;
        return;
    }
    const float a = fminf(1.0f, G.rho_max_f * (rmax + G.dmax_f) * 0.5f);
    const float b = fminf(1.0f, G.dmax_f / rmin);
    const float w = fminf(asinf(a) + asinf(b), 1.57079633f) + 4e-3f;
    const float k = kIdxAz / 6.28318531f;
    b0 = (int)floorf((phik - w + 3.14159265f) * k);
    b1 = (int)floorf((phik + w + 3.14159265f) * k);
    full = b1 - b0 + 1 >= kIdxAz;
}

// Second-root reach of rows with |rho| <= rt (TileCtx::init of tiles.cuh).
__device__ __forceinline__ bool needs_b(const DevGeom &G, float rt, float s, float c, float eS)
{
    if (!(rt > 0.0f)) return false;
    const float ir = __frcp_rn(rt);
    const float sB = fmaf(ir - G.dext_f, 1.0f - 1e-6f, -0.01f);
    const float cB = fmaf(sqrtf(fmaxf(fmaf(ir, ir, -G.dext_f * G.dext_f), 0.0f)), 1.0f - 1e-6f,
                          -0.05f);
    return fabsf(s) + eS >= sB && c + eS >= cB;
}

// s = x sn - y cs and c = x cs + y sn of a hit in a column, with the tables'
// float32 remainders and the products' and sum's rounding errors carried:
// within 1.01 2^-24 of their own size plus a few 2^-48 (|x| + |y|) of the
// exact values, instead of 3 2^-24 (|x| + |y|).
__device__ __forceinline__ float dot2(float a, float p, float plo, float b, float q, float qlo)
{
    const float u = __fmul_rn(a, p), eu = fmaf(a, p, -u);   // (never fused into the sum)
    const float v = __fmul_rn(b, q), ev = fmaf(b, q, -v);
    const F2 h = two_sum(u, v);
    return h.hi + (h.lo + (eu + ev) + fmaf(a, plo, b * qlo));
}

// Bound on the error of dot2's s (or c).
__device__ __forceinline__ float dot2_err(float v, float R1)
{
    return fmaf(1.25f * kEps, fabsf(v), 1e-13f * R1);
}

// Bound (rows) on the row coordinate of an edge crossing,
//   t = tc - kr w / (w^2 + c^2),  w = s + (edge - off) delta,
// against the exact crossing of the float64 definition's curve (first order,
// u = 2^-24, kSafe on the sum).  w is off by eS (the float32 s) plus
// u (|d| + |w|) from the edge and the sum, |dt/dw| <= kr / c^2; c^2 is off by
// 2 eC / c + u relative, |dt/d(c^2)| <= kr |w| / c^4 with |w| <= rt c^2 at the
// rows' edges and kr rt <= n_rho; the sum of squares, the reciprocal, the
// products and the last sum add 6u |t - tc| + u |t| <= 8u n_rho.  The
// definition's own rounding is a few 2^-53 of rho R1^2 + 2 R1 in d0 (e64).
__device__ __forceinline__ float walk_eps(const DevGeom &G, float c, float R1, float eS, float eC)
{
    const float ic = rcp_approx(c) * 1.001f;
    const float e64 = 1e-13f * R1;
    return kSafe * (G.kr_f * ic * ic * fmaf(kEps, G.dmax_f + c, eS + e64) +
                    (float)G.n_rho * fmaf(2.0f * eC, ic, 9.0f * kEps));
}

// The A-form record of tiles.cuh ({A0, c^2, c2d, eA} and eB) for s and c with
// errors eS and eC (make_aform takes 4e-7 R1 for both).
__device__ __forceinline__ float4 make_aform2(const DevGeom &G, float s, float c, float R1,
                                              float rt, float eS, float eC, float &eB)
{
    const float c2 = c * c;
    const float t = rt * rt * c2 * 1.001f;
    const float A0 = fmaf(-s, G.inv_delta_f, G.off_f);
    const float c2d = c2 * G.inv_delta_f;
    const float rc = 2.0f * eC * rcp_approx(c) * 1.001f;
    const float dD = fmaf(t, rc + 5.0f * kEps, kEps);
    const float isD = rsqrt_approx(1.0f - t) * 1.001f;
    const float aA = fabsf(A0);
    const float e64 = 1.6e-14f * fmaf(rt * R1, R1, 2.0f * R1) * G.inv_delta_f +
                      4e-15f * (aA + rt * c2d + G.off_f);
    const float eA = (kSafe * 1.001f) * (fmaf(kEps, fabsf(s), eS) * G.inv_delta_f +
                                         2.0f * kEps * aA) + e64;
    eB = (kSafe * 1.001f) * c2d * (rc + 14.3f * kEps + dD * isD);
    return make_float4(A0, c2, c2d, eA);
}

// The definition's bins of one (hit, row, column) through the double-float
// and float64 tiers: (first + 1) | (second + 1) << 16, 0 for none.  One
// copy of the code for every caller.
static __device__ __noinline__ unsigned redo_packed(const DevGeom &G, float xf, float yf, int i,
                                                    int k)
{
    int jj[2] = {-1, -1};
    const int nv = redo_bins(G, xf, yf, i, k, jj);
    return (nv > 0 ? (unsigned)(jj[0] + 1) : 0u) | (nv > 1 ? (unsigned)(jj[1] + 1) << 16 : 0u);
}

// Floors of t - eps and t + eps, rounded outwards (|t| small).
__device__ __forceinline__ void crossing(float t, float eps, int &lo, int &hi)
{
    lo = __float_as_int(__fadd_rd(__fsub_rd(t, eps), kMagic)) - kMagicBits;
    hi = __float_as_int(__fadd_rd(__fadd_ru(t, eps), kMagic)) - kMagicBits;
}

// Row coordinate (within the band, tc = the row of rho = 0) at which the
// curve of a hit (s, c) crosses d0 = jo delta: the rows up to it have their
// root at or above that edge.  Edges below -c are below every row's root;
// the clamp puts their crossing beyond the rows.  |t - tc| <= kr / (2 c).
__device__ __forceinline__ float cross_row(const DevGeom &G, float jo, float s, float c, float c2,
                                           float tc)
{
    const float w = fmaxf(fmaf(jo, G.delta_f, s), -c);
    return fmaf(-G.kr_f * w, rcp_approx(fmaf(w, w, c2)), tc);
}

// Bin coordinate of a hit's root in a row (A-form, no bound).
__device__ __forceinline__ float row_coord(const DevGeom &G, float s, float c2, float rho)
{
    const float D = fmaf(-rho * rho, c2, 1.0f);
    const float den = fmaf(D, rsqrt_approx(D), 1.0f);
    return fmaf(-rho * c2 * G.inv_delta_f, rcp_approx(den), fmaf(-s, G.inv_delta_f, G.off_f));
}

// One tile of one event: votes, then the layer counts.
// PLANES: out is the event's bit planes (see k_peak_planes.cu); otherwise the
// accumulator of OutT counts.
template <int NWB, bool HIT, bool PLANES, bool CELLS, int kThr, typename OutT>
__device__ __forceinline__ void vr_tile(const DevGeom &G, const HitSource &H, int e,
                                        const unsigned long long *__restrict__ hmask,
                                        void *__restrict__ out,
                                        unsigned long long *__restrict__ stats, int k, int band)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kWarps = kThr / 32;
    // runs of positions [rs, re) (index: layer << 2 | part << 1 | side), chunks
    // before each, rows first | last << 16 they vote in
    __shared__ int s_rs[64], s_re[64], s_cp[65], s_row[64];
    __shared__ int s_next, s_more, s_full, s_any;
    __shared__ int s_nredo[kWarps];
    __shared__ unsigned long long s_stats[2];
    __shared__ int s_ws[32], s_we[32];   // CELLS: window runs (layer << 1 | part)
    __shared__ int s_bad, s_val[16];   // CELLS: a cell layer's rows first | last << 16, else -1
    // single event: the warps' hits that can vote here and wait for a full warp
    __shared__ int s_wait[PLANES ? 1 : kWarps][32 + kGather];
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kBand = 32 * NWB;
    constexpr int IPW = 32 / NWB;                  // hits per walk step
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ND = G.n_d0, NDp = ND + kVrPad, NW = (G.n_rho + 31) / 32;
    const VrSmem S = vr_carve<NWB, HIT, CELLS, kThr>(smem, ND);
    const int i0 = band * kBand, nrow = min(kBand, G.n_rho - i0);
    const float tc = 0.5f * (float)(G.n_rho - 1) - (float)i0;   // row of rho = 0

    for (int r = threadIdx.x; r < nrow; r += kThr) S.rho[r] = G.rho32[i0 + r];
    if (HIT) {
        const int NR = G.n_rho;
        for (int j = threadIdx.x; j < ND; j += kThr)
            S.jmask[j] = (uint8_t)((1u << region_block(max(j - 1, 0), ND)) |
                                   (1u << region_block(j, ND)) |
                                   (1u << region_block(min(j + 1, ND - 1), ND)));
        for (int r = threadIdx.x; r < kBand; r += kThr) {
            const int i = min(i0 + r, NR - 1);
            S.rowblk[r] = (8u * region_block(max(i - 1, 0), NR)) |
                          (8u * region_block(i, NR) << 8) |
                          (8u * region_block(min(i + 1, NR - 1), NR) << 16);
        }
        for (int q = threadIdx.x; q < NWB * 8; q += kThr) {
            const int b = q & 7, f = i0 + 32 * (q >> 3);
            // rows [first of b - 1, first of b + 1] of the word; empty blocks hold none
            const int lo = max(block_first(b, NR) - 1 - f, 0);
            const int hi = min(block_first(b + 1, NR) - f, 31);
            const bool has = block_first(b + 1, NR) > block_first(b, NR);
            S.rowmask[q] = has && lo <= hi && lo < 32 && hi >= 0
                               ? (kAll << lo) & (kAll >> (31 - hi)) : 0u;
        }
    }
    if (threadIdx.x < 2) s_stats[threadIdx.x] = 0ull;
    int my_cast = 0;   // votes (cell rows subtract what lies below the axis)
    int my_fb = 0;

#pragma unroll 1
    for (int l0 = 0; l0 < 16; l0 += kRes) {
        const int l1 = min(l0 + kRes, 16);
        // ---- the runs of positions that hold the column's hits
        __syncthreads();   // the previous round's counts are out
        if (warp == 0) {
            int start = 0, end = 0;
            if (H.offs) {
                const int l = lane >> 1, part = lane & 1;
                const float rmin = __uint_as_float(H.rmm[2 * (e * 16 + l)]);
                const float rmax = __uint_as_float(H.rmm[2 * (e * 16 + l) + 1]);
                const bool all16 = __all_sync(kAll, rmin <= rmax);
                if (lane == 0) s_full = all16;
                if (l >= l0 && l < l1) {
                    bool full, empty;
                    int b0, b1;
                    vote_cells(G, G.phi32[k], rmin, rmax, full, empty, b0, b1);
                    const int *o = H.offs + (e * 16 + l) * kIdxAz;
                    if (full) {
                        if (part == 0) {
                            start = o[0];
                            end = o[kIdxAz];
                        }
                    } else if (!empty) {
                        const int b0m = ((b0 % kIdxAz) + kIdxAz) % kIdxAz, nb = b1 - b0 + 1;
                        const bool wrap = b0m + nb > kIdxAz;
                        if (part == 0) {
                            start = o[b0m];
                            end = o[wrap ? kIdxAz : b0m + nb];
                        } else if (wrap) {
                            start = o[0];
                            end = o[b0m + nb - kIdxAz];
                        }
                    }
                }
            } else if (lane == 0 && (l0 == 0 || s_more)) {
                end = H.n;
            }
            s_ws[lane] = start;
            s_we[lane] = end;
            const bool any = __any_sync(kAll, end > start);
            if (lane == 0) {
                s_any = any;
                s_cp[0] = 0;
                s_next = 0;
            }
            __syncwarp();
            if (lane == 0 && l0 == 0) s_more = 0;
        }
        if (threadIdx.x < kWarps) s_nredo[threadIdx.x] = 0;
        if (CELLS && threadIdx.x < 16) s_val[threadIdx.x] = -1;
        __syncthreads();
        if (l0 > 0 && !s_any) continue;   // uniform
        {
            uint4 *z4 = reinterpret_cast<uint4 *>(S.bm);
            // (NDp is a multiple of 2, kRes and kKept too; the kept counts stay)
            const int n4 = (!PLANES && l0 > 0 ? kKept : kRes) * NWB * NDp / 4;
            for (int t = threadIdx.x; t < n4; t += kThr) z4[t] = make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
        VrSlot *const slot = S.slot + warp * 32;
        int4 *const imeta = S.item + warp * 32;
        unsigned long long *const shm = HIT ? S.hm + warp * 32 : nullptr;
        int2 *const redo = S.redo + warp * kVrRedo;
        auto set_hm = [&](int p) -> unsigned long long { return hmask[H.h ? H.h[p] : p]; };
        // word of (layer, row word, bin 0)
        auto word0 = [&](int l, int w) -> uint32_t * {
            return S.bm + ((l - l0) * NWB + w) * NDp;
        };
        // the definition's votes of one (position, row), any tier
        auto redo_row = [&](int p, int r, int l, bool counted) {
            const unsigned pk = redo_packed(G, H.x[p], H.y[p], i0 + r, k);
            unsigned rb = 0u;
            if (HIT) rb = halo_row_blocks(set_hm(p), i0 + r, G.n_rho);
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const int j = (int)((pk >> (16 * v)) & 0xffffu) - 1;
                if (j < 0 || (HIT && !(rb & S.jmask[j]))) continue;
                atomicOr(word0(l, r >> 5) + j, 1u << (r & 31));
                if (counted) ++my_cast;
            }
        };
        constexpr int kNotCounted = 1 << 30;   // the row's vote is counted already
        auto push = [&](int p, int r, int l, int flag = 0) {
            ++my_fb;
            const int q = atomicAdd(&s_nredo[warp], 1);
            if (q < kVrRedo) redo[q] = make_int2(p, (r << 4) | l | flag);
            else redo_row(p, r, l, flag == 0);
        };
        auto drain = [&]() {   // the warp's redos, a lane each (all lanes call)
            __syncwarp();
            const int nr = min(s_nredo[warp], kVrRedo);
#pragma unroll 1
            for (int t = lane; t < nr; t += 32) {
                const int y = redo[t].y;
                redo_row(redo[t].x, (y & ~kNotCounted) >> 4, y & 15, !(y & kNotCounted));
            }
            __syncwarp();
            if (lane == 0) s_nredo[warp] = 0;
            __syncwarp();
        };
        // rows [r, last] of word wd (in-word rows) allowed to the set hs in a
        // bin with d0 blocks jm
        auto allowed = [&](unsigned long long hs, unsigned jm, int wd) -> uint32_t {
            uint32_t al = 0u;
#pragma unroll
            for (int bb = 0; bb < 8; ++bb)
                if ((unsigned)(hs >> (8 * bb)) & jm) al |= S.rowmask[wd * 8 + bb];
            return al;
        };

        if constexpr (CELLS) {
            for (int l = l0; l < l1; ++l) {   // uniform
                const int st0 = s_ws[2 * l], n0 = s_we[2 * l] - st0;
                const int st1 = s_ws[2 * l + 1], n = n0 + s_we[2 * l + 1] - st1;
                if (n < kCellMin || n > kClMaxHits || H.unsorted[e * 16 + l] != 0) continue;
                const float rmin = __uint_as_float(H.rmm[2 * (e * 16 + l)]);
                const float rmax = __uint_as_float(H.rmm[2 * (e * 16 + l) + 1]);
                const float dmax = G.dext_f;
                if (!(rmin >= 1e-3f) || !(rmax < 1e6f)) continue;
                // |rho| up to which S is monotone over the axis: with u = 1 - |rho| dmax,
                // 1 + u^2 - rho^2 r^2 >= 0.05 (then dS/dd0 > 0 and sqrt(D) > 0.01)
                const float rv = fminf(1.95f / (dmax + sqrtf(fmaxf(fmaf(1.95f * rmax, rmax,
                                                                        -0.95f * dmax * dmax), 0.0f))),
                                       0.95f / dmax) * 0.9999f;
                const int vA = (int)fmaxf(ceilf(fmaf(-rv, G.inv_drho_f, tc)), 0.0f);
                const int vB = (int)fminf(floorf(fmaf(rv, G.inv_drho_f, tc)), (float)(nrow - 1));
                if (vB - vA < 32) continue;
                // bound on S at an edge against -s of a hit (cm), first order: S's own
                // rounding, the layer's spread in r^2, the hit's float32 s; and by how much
                // hits can be out of order in s: the spread in r, atan2f's 3 ulp at a cell
                // boundary (twice), the rounding of s
                const float rt = fmaxf(fabsf(S.rho[vA]), fabsf(S.rho[vB]));
                const float iu = 0.5f / (1.0f - rt * dmax);
                const float r2 = 0.5f * fmaf(rmin, rmin, rmax * rmax);
                const float eE = kEps * fmaf(iu, fmaf(8.0f * rt, fmaf(rmax, rmax, dmax * dmax), 12.0f * dmax),
                                             4.0f * rmax);
                const float eR2 = rt * iu * (0.51f * (rmax - rmin) * (rmax + rmin) +
                                             8.0f * kEps * rmax * rmax);
                const float eta = 1.01f * (rmax - rmin) + 2.3e-6f * rmax;   // how far out of order
                const float eps = fmaf(kSafe, eE + eR2 + dot2_err(rmax, 2.0f * rmax), eta);
                if (!(eps <= 0.05f * G.delta_f)) continue;
                // ---- the layer's -s in azimuth order; hits with c <= 0 beyond its ends
                __syncthreads();
                if (threadIdx.x == 0) s_bad = 0;
                __syncthreads();
                {
                    const float sk = G.sn32[k], ck = G.cs32[k], sl = G.snlo[k], cl = G.cslo[k];
                    for (int t = threadIdx.x; t < n; t += kThr) {
                        const int p = t < n0 ? st0 + t : st1 + t - n0;
                        const float xf = H.x[p], yf = H.y[p];
                        const float c = dot2(xf, ck, cl, yf, sk, sl);
                        const float s = dot2(xf, sk, sl, -yf, ck, cl);
                        const float Ec = (kSafe * 3.0f * kEps) * (fabsf(xf) + fabsf(yf));
                        if (!(fabsf(c) > Ec)) s_bad = 1;   // sign of c not proven (or NaN)
                        S.sig[t] = c > 0.0f ? -s : s < 0.0f ? 3.0e38f : -3.0e38f;
                    }
                    if (threadIdx.x == 0) S.sig[n] = 3.4e38f;
                }
                __syncthreads();
                if (s_bad) continue;   // uniform
                // ---- the table: below[q] = hits certainly before bin q = [q, q + 1) / kap - R
                const float Rr = rmax * 1.001f, kap = (float)kClTab / (2.0f * Rr), k0 = Rr * kap;
                const float ef = fmaf(2e-6f, Rr, eps + eta);   // and the rounding of a table bin
                auto tbin = [&](float v) -> int {
                    return (int)fminf(fmaxf(floorf(fmaf(v, kap, k0)), -1.0f), (float)(kClTab - 1));
                };
                for (int t = threadIdx.x; t <= n; t += kThr) {
                    const int a1 = t < n ? tbin(S.sig[t] + ef) : kClTab - 1;
                    const int a0 = t > 0 ? tbin(S.sig[t - 1] + ef) : -1;
                    for (int q = a0 + 1; q <= a1; ++q) S.tab[q] = (uint16_t)t;
                }
                __syncthreads();
                // the first hit not below v, from rank r on (a value past every edge ends
                // the hits)
                auto first_at = [&](float v, int r, float &t) -> int {
                    const float q = fminf(fmaxf(fmaf(v, kap, k0), 0.0f), (float)(kClTab - 1));
                    r = max(r, (int)S.tab[(int)q]);
                    t = S.sig[r];
                    while (t < v) t = S.sig[++r];
                    return r;
                };
                // ---- units of one row word x 32 bins, a lane per row
                const int nj = (ND + 31) >> 5;
                for (int u = warp; u < NWB * nj; u += kWarps) {
                    const int wd = u % NWB, j0 = (u / NWB) << 5, jn = min(32, ND - j0);
                    const int row = 32 * wd + lane;
                    const bool ok = row >= vA && row <= vB;
                    const float rho = S.rho[min(max(row, vA), vB)], rr = rho * r2, rho2 = 2.0f * rho;
                    uint32_t mine = 0u;
                    auto hit = [&](int q) -> int { return q < n0 ? st0 + q : st1 + q - n0; };
                    auto at = [&](int j) -> float {
                        const float d = ((float)j - G.off_f) * G.delta_f;
                        return fmaf(fmaf(rho, d, 2.0f), d, rr) * rcp_approx(fmaf(rho2, d, 2.0f));
                    };
                    // r: hits below the edge or within the bound of it; those from open on
                    // are within it and not settled yet
                    const float v0 = at(j0);
                    int r = n, open = n;
                    if (ok) {
                        float t;
                        open = r = first_at(v0 - eps, 0, t);
                        while (t <= v0 + eps) t = S.sig[++r];
                        if (j0 == 0) {   // the axis' lower end: these are not counted below
                            my_cast -= r;
                            for (; open < r; ++open) push(hit(open), row, l);
                        }
                    }
                    bool prev = false;   // the bin below surely holds a hit
                    for (int jj = 0; jj < jn; ++jj) {
                        const float v1 = at(j0 + jj + 1);
                        const int r0 = r;
                        float t;
                        r = first_at(v1 - eps, r0, t);
                        const bool bit = r > r0;
                        if (open < r0 && !(prev && bit))   // one of the two bins depends on them
                            for (int q = open; q < r0; ++q) push(hit(q), row, l, kNotCounted);
                        open = r;
                        while (t <= v1 + eps) t = S.sig[++r];
                        prev = bit;
                        const uint32_t word = __ballot_sync(kAll, bit);
                        if (lane == jj) mine = word;
                    }
                    if (ok) {
                        const bool end = j0 + jn == ND;   // the axis' upper end
                        if (end) my_cast += open;
                        for (; open < r; ++open) push(hit(open), row, l, end ? 0 : kNotCounted);
                    }
                    if (mine) atomicOr(word0(l, wd) + j0 + lane, mine);
                    __syncwarp();
                    if (s_nredo[warp] >= 32) drain();
                }
                if (threadIdx.x == 0) s_val[l] = vA | (vB << 16);   // the other rows go hit by hit
            }
            __syncthreads();
        }
        // (single event: of a size that gives every warp as many chunks)
        int step = 32;
        if (!PLANES) {
            const int rounds = max((H.n + kGather * kWarps - 1) / (kGather * kWarps), 1);
            step = max((H.n + rounds * kWarps - 1) / (rounds * kWarps), 1);
        }
        // ---- chunks of step hits of the runs; a cell layer's runs twice, below and
        // above its rows
        if (warp == 0) {
            int n[2];
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int q = 2 * lane + side;   // layer << 2 | part << 1 | side
                int r0 = 0, r1 = nrow - 1;
                bool use = side == 0;
                if (CELLS && s_val[lane >> 1] >= 0) {
                    if (side) r0 = (s_val[lane >> 1] >> 16) + 1;
                    else r1 = (s_val[lane >> 1] & 0xffff) - 1;
                    use = r0 <= r1;
                }
                s_rs[q] = s_ws[lane];
                s_re[q] = use ? s_we[lane] : s_ws[lane];
                s_row[q] = r0 | (max(r1, 0) << 16);
                n[side] = (s_re[q] - s_rs[q] + step - 1) / step;
            }
            int incl = n[0] + n[1];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kAll, incl, o);
                if (lane >= o) incl += v;
            }
            s_cp[2 * lane + 1] = incl - n[1];
            s_cp[2 * lane + 2] = incl;
        }
        __syncthreads();
        const int nchunk = s_cp[64];
        auto pop = [&]() -> int {
            int ch = 0;
            if (lane == 0) ch = atomicAdd(&s_next, 1);
            return __shfl_sync(kAll, ch, 0);
        };
        int nwait = 0;   // single event: hits in s_wait

        for (;;) {
            int run = 0, p = 0;
            bool live = false;
            if constexpr (PLANES) {
                const int ch = pop();
                if (ch >= nchunk) break;
                int hi = 63;   // the last run with s_cp[run] <= ch
                while (run < hi) {
                    const int mid = (run + hi + 1) >> 1;
                    if (s_cp[mid] <= ch) run = mid;
                    else hi = mid - 1;
                }
                p = s_rs[run] + (ch - s_cp[run]) * 32 + lane;
                live = p < s_re[run];
            } else {
                // The event's hits in the caller's order: those of this round's layers
                // that can vote in the tile's rows (the tests below, on the plain s and
                // c that the filters' margins are for) wait until they fill the warp.
                const float sk = G.sn32[k], ck = G.cs32[k];
                while (nwait < 32) {
                    const int ch = pop();
                    if (ch >= nchunk) break;
                    bool keep[kGather / 32];
#pragma unroll
                    for (int u = 0; u < kGather / 32; ++u) {
                        const int q = ch * step + 32 * u + lane;
                        const bool in = 32 * u + lane < step && q < H.n;
                        const int l = in ? H.l[q] & 15 : 0;
                        const float xf = in ? H.x[q] : 0.0f, yf = in ? H.y[q] : 0.0f;
                        if (l >= l1) s_more = 1;
                        const float c = fmaf(xf, ck, yf * sk), s = fmaf(xf, sk, -(yf * ck));
                        const float R1 = fabsf(xf) + fabsf(yf);
                        keep[u] = in && l >= l0 && l < l1 &&
                                  !(c < hit_cos_window(G, fmaf(xf, xf, yf * yf))) &&
                                  !(c < -(kSafe * 3.0f * kEps) * R1);
                        if (nrow < G.n_rho && keep[u] && c > 1.0f) {   // more than one band
                            float gmin, gmax;
                            rho_range(G, s, c, 4e-7f * R1, gmin, gmax);
                            const float fa = floorf(fmaf(gmin, G.inv_drho_f, tc - 0.5f));
                            const float fb = ceilf(fmaf(gmax, G.inv_drho_f, tc + 0.5f));
                            keep[u] = fa <= (float)(nrow - 1) && fb >= 0.0f;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kGather / 32; ++u) {
                        const unsigned m = __ballot_sync(kAll, keep[u]);
                        if (keep[u])
                            s_wait[warp][nwait + __popc(m & ((1u << lane) - 1u))] =
                                ch * step + 32 * u + lane;
                        nwait += __popc(m);
                    }
                }
                if (nwait == 0) break;
                __syncwarp();
                const int take = min(nwait, 32);
                nwait -= take;
                live = lane < take;
                if (live) p = s_wait[warp][nwait + lane];
                __syncwarp();   // the places are free again
            }
            // ---- one hit per lane: its kind and its constants
            enum { kWalk, kEdge8, kEdge16, kEdge32, kEdge64, kRow, kKinds, kNone = kKinds };
            int kind = kNone;
            // item rows: the window's (bytes 0 and 3) without bytes 1 .. 2 (all when 1 > 2)
            unsigned rest = 0u;
            bool item = false;
            float4 ma = make_float4(0.f, 0.f, 0.f, 0.f), mb = ma;
            unsigned long long hm = 0ull;
            if (live) {
                const int l = PLANES ? run >> 2 : H.l[p] & 15;
                const float sk = G.sn32[k], ck = G.cs32[k], sl = G.snlo[k], cl = G.cslo[k];
                const float xf = H.x[p], yf = H.y[p];
                const float c = dot2(xf, ck, cl, yf, sk, sl);
                const float s = dot2(xf, sk, sl, -yf, ck, cl);
                const float R1 = fabsf(xf) + fabsf(yf);
                const float Ec = (kSafe * 3.0f * kEps) * R1;
                const float eR = 4e-7f * R1;   // what the shared filters take for s and c
                if (c < -Ec) live = false;
                float hwlo = G.d0lo_f, hwhi = G.d0hi_f;
                int jhi = ND;   // the highest bin of interest, plus one
                if (HIT && live) {
                    // the hit's d0 blocks over the band's rows and their halo
                    hm = set_hm(p);
                    const int NR = G.n_rho;
                    const int rb0 = region_block(max(i0 - 1, 0), NR);
                    const int rb1 = region_block(min(i0 + nrow, NR - 1), NR);
                    unsigned tb = 0u;
                    for (int b = rb0; b <= rb1; ++b) tb |= (unsigned)(hm >> (8 * b)) & 0xffu;
                    live = tb != 0u;
                    if (live) {
                        const int lo = max(block_first(__ffs(tb) - 1, ND) - 1, 0);
                        const int hib = min(block_first(32 - __clz(tb), ND), ND - 1);
                        hwlo = fmaf((float)lo - G.off_f, G.delta_f, -0.01f);
                        hwhi = fmaf((float)(hib + 1) - G.off_f, G.delta_f, 0.01f);
                        jhi = hib + 1;
                    }
                }
                if (live) {
                    // rows whose circles can reach the (hit's part of the) axis
                    int ra = CELLS ? s_row[run] & 0xffff : 0;
                    int rb = CELLS ? s_row[run] >> 16 : nrow - 1;
                    if (c > 1.0f) {
                        float gmin, gmax;
                        rho_range_w(hwlo + s, hwhi + s, c, eR, gmin, gmax);
                        const float fa = floorf(fmaf(gmin, G.inv_drho_f, tc - 0.5f));
                        const float fb = ceilf(fmaf(gmax, G.inv_drho_f, tc + 0.5f));
                        if (!(fa <= (float)rb && fb >= (float)ra)) live = false;
                        ra = (int)fmaxf(fa, (float)ra);
                        rb = (int)fminf(fb, (float)rb);
                    }
                    if (live) {
                        // |rho| up to which root B is out of the axis (the conditions of
                        // needs_b solved for rt), b = 1 + rho s > 0 and D > 0
                        const float sp = fmaf(fabsf(s) + eR, 1.000004f, 0.0102f);
                        const float cp = fmaf(c + eR, 1.000004f, 0.0502f);
                        float rok = fmaxf(rcp_approx(G.dext_f + sp),
                                          rsqrt_approx(fmaf(cp, cp, G.dext_f * G.dext_f)));
                        rok = fminf(rok, 0.985f * rcp_approx(fmaxf(c, fabsf(s) + eR))) * 0.9997f;
                        const int rA = (int)fmaxf(ceilf(fmaf(-rok, G.inv_drho_f, tc)), (float)ra);
                        const int rB = (int)fminf(floorf(fmaf(rok, G.inv_drho_f, tc)), (float)rb);
                        mb.z = __int_as_float((l << 16) | ((l - l0) * NWB * NDp));
                        mb.w = __int_as_float(p);
                        item = true;
                        rest = (unsigned)ra | (1u << 8) | ((unsigned)rb << 24);   // every row
                        const float rt = rA <= rB ? fmaxf(fabsf(S.rho[rA]), fabsf(S.rho[rB])) * 1.0001f
                                                  : 0.0f;
                        if (rA <= rB && c > Ec && !needs_b(G, rt, s, c, eR) &&
                            aform_ok(G, s, c, R1, rt)) {
                            rest = (unsigned)ra | ((unsigned)rA << 8) | ((unsigned)rB << 16) |
                                   ((unsigned)rb << 24);
                            item = ra < rA || rB < rb;
                            mb.y = __int_as_float(rA | (rB << 16));
                            kind = kRow;
                            const float c2 = c * c;
                            const float eS = dot2_err(s, R1), eC = dot2_err(c, R1);
                            float eB;
                            ma = make_aform2(G, s, c, R1, rt, eS, eC, eB);
                            mb.x = eB;
                            // bins per row at rho = 0; crossings also need the clamp
                            // at -c two rows beyond the rows
                            const float slope = 0.5f * G.drho_f * c2 * G.inv_delta_f;
                            if (slope <= kEdgeSlope && c * fmaf(2.0f, G.drho_f, rt) <= 0.97f &&
                                fmaf(rt, eB, ma.w) <= 0.01f) {
                                const float eps = walk_eps(G, c, R1, eS, eC);
                                // bins of the rows: from the first row's (or the next
                                // one up when its coordinate is within 0.02 of it: the
                                // bound is below 0.01) to the last row's
                                const float uh = row_coord(G, s, c2, S.rho[rA]);
                                const float ul = row_coord(G, s, c2, S.rho[rB]);
                                const float jt = floorf(fminf(uh + 0.02f, (float)jhi));
                                const float nbin = jt - fmaxf(floorf(ul - 0.02f), 0.0f) + 1.0f;
                                const bool flat = slope <= kWalkSlope;
                                if (!(jt >= 0.0f)) {
                                    kind = kNone;   // below the axis
                                } else if (flat ? eps <= kWalkEps
                                                : eps <= kEdgeEps && c > 2.4e-7f * G.kr_f) {
                                    kind = flat ? kWalk : nbin <= 8.0f ? kEdge8
                                           : nbin <= 16.0f ? kEdge16
                                           : nbin <= 32.0f ? kEdge32 : kEdge64;
                                    ma = make_float4(s, c, eps, jt - G.off_f);
                                    mb.x = nbin;
                                    mb.z = __int_as_float(__float_as_int(mb.z) + (int)jt);
                                }
                            }
                        }
                    }
                }
            }
            // Slots of 32 bytes in the order of the kinds.  walk, edge: {s, c, bound
            // (rows), first bin - off}, {bins, rows, layer << 16 | word of (layer,
            // row word 0, first bin), position}; row: {A-form}, {eB, rows, layer << 16
            // | word of (layer, 0, 0), position}.  first[t] = the first of kind t
            int first[kKinds + 1];
            first[0] = 0;
            int q_of = 0;
#pragma unroll
            for (int t = 0; t < kKinds; ++t) {
                const unsigned m = __ballot_sync(kAll, kind == t);
                if (kind == t) q_of = first[t] + __popc(m & ((1u << lane) - 1u));
                first[t + 1] = first[t] + __popc(m);
            }
            if (kind != kNone) {
                slot[q_of].a = ma;
                slot[q_of].b = mb;
                if (HIT) shm[q_of] = hm;
            }
            __syncwarp();

            // ---- walk: lane = (hit, word)
            for (int q0 = 0; q0 < first[kEdge8]; q0 += IPW) {
                const int q = q0 + lane / NWB, wd = lane % NWB;
                if (q < first[kEdge8]) {
                    const float4 a = slot[q].a, b = slot[q].b;
                    const float s = a.x, c = a.y, eps = a.z, c2 = c * c;
                    const int rab = __float_as_int(b.y), l = __float_as_int(b.z) >> 16;
                    int r = max((rab & 0xffff) - 32 * wd, 0);           // rows of the word
                    const int r1 = min((rab >> 16) - 32 * wd, 31);
                    const int jtop = (int)(a.w + G.off_f);
                    unsigned long long hs = 0ull;
                    if (HIT) hs = shm[q];
                    if (r <= r1) {
                        const float tw = tc - (float)(32 * wd);
                        const float u = row_coord(G, s, c2, S.rho[32 * wd + r]);
                        // bin jtop (at most n_d0) stands for everything above it too
                        int j = min((int)floorf(fmaxf(u + 0.02f, -1.0f)), jtop);
                        uint32_t *wp = word0(l, wd) + j;
                        float jo = (float)j - G.off_f;
                        while (j >= 0 && r <= r1) {
                            int lo, hi;
                            const float t = cross_row(G, jo, s, c, c2, tw);
                            crossing(fminf(fmaxf(t, -16.0f), 48.0f), eps, lo, hi);
                            const int last = min(lo, r1);
                            if (last >= r) {
                                if (j < ND) {
                                    uint32_t m = (kAll << r) & (kAll >> (31 - last));
                                    if (HIT) m &= allowed(hs, S.jmask[j], wd);
                                    atomicOr(wp, m);
                                    my_cast += __popc(m);
                                }
                                r = last + 1;
                            }
                            if (hi > lo) {   // rows within the bound of this edge
                                const int hi2 = min(hi, r1);
                                for (int rr = max(lo + 1, r); rr <= hi2; ++rr)
                                    push(__float_as_int(b.w), 32 * wd + rr, l);
                                r = max(r, hi2 + 1);
                            }
                            --j;
                            --wp;
                            jo -= 1.0f;
                        }
                    }
                }
            }
            __syncwarp();

            // ---- edge: lane = (hit, bin)
            const float jcap = (float)ND - G.off_f - 0.25f;
            // votes rows r .. last (in one word, or two, or more) of the bin of word wp
            // (lower edge jo); the virtual bin above the axis has none
            auto emit = [&](uint32_t *wp, int r, int last, float jo, unsigned long long hs) {
                if (!(r <= last && jo < jcap)) return;
                uint32_t m = kAll << (r & 31), m2 = kAll >> (31 - (last & 31));
                const int w0 = r >> 5, w1 = last >> 5;
                if (w0 == w1) m &= m2;
                if (HIT) {
                    const unsigned jm = S.jmask[(int)(jo + G.off_f + 0.25f)];
                    m &= allowed(hs, jm, w0);
                    m2 = w1 > w0 ? m2 & allowed(hs, jm, w1) : 0u;
                    my_cast += __popc(m) + __popc(m2);
                } else {
                    my_cast += last - r + 1;
                }
                atomicOr(wp + w0 * NDp, m);
                if (w1 > w0) {
                    atomicOr(wp + w1 * NDp, m2);
                    for (int w = w0 + 1; w < w1; ++w) {   // a run over a whole word
                        uint32_t mm = kAll;
                        if (HIT) {
                            mm = allowed(hs, S.jmask[(int)(jo + G.off_f + 0.25f)], w);
                            my_cast += __popc(mm);
                        }
                        atomicOr(wp + w * NDp, mm);
                    }
                }
            };
            // up to 32 bins: 2^lg lanes per hit
#pragma unroll 1
            for (int lg = 3; lg <= 5; ++lg) {
                const int qb = lg == 3 ? first[kEdge8] : lg == 4 ? first[kEdge16] : first[kEdge32];
                const int qe = lg == 3 ? first[kEdge16] : lg == 4 ? first[kEdge32] : first[kEdge64];
                const int width = 1 << lg, sub = lane & (width - 1);
                const float fsub = (float)sub;
#pragma unroll 1
                for (int q0 = qb; q0 < qe; q0 += 32 >> lg) {
                    const bool act = q0 + (lane >> lg) < qe;
                    const int q = act ? q0 + (lane >> lg) : q0;
                    const float4 a = slot[q].a, b = slot[q].b;
                    const int rab = __float_as_int(b.y), ra1 = (rab & 0xffff) - 1, rb = rab >> 16;
                    unsigned long long hs = 0ull;
                    if (HIT) hs = shm[q];
                    const float jo = a.w - fsub;   // the lane's lower edge, in bins from d0 = 0
                    int lo, hi;
                    crossing(cross_row(G, jo, a.x, a.y, a.y * a.y, tc), a.z, lo, hi);
                    const int pv = __shfl_up_sync(kAll, hi, 1, width);
                    const int before = sub == 0 ? ra1 : max(pv, ra1);   // rows settled above
                    if (act && fsub < b.x) {
                        emit(S.bm + (__float_as_int(b.z) & 0xffff) - sub, before + 1, min(lo, rb), jo, hs);
                        // one row within the bound of this edge
                        if (hi > lo && lo >= before && lo < rb)
                            push(__float_as_int(b.w), lo + 1, __float_as_int(b.z) >> 16);
                    }
                }
            }
            // more: a lane takes two bins
#pragma unroll 1
            for (int q = first[kEdge64]; q < first[kRow]; ++q) {
                const float4 a = slot[q].a, b = slot[q].b;
                const int rab = __float_as_int(b.y), rb = rab >> 16;
                const float s = a.x, c = a.y, c2 = c * c;
                unsigned long long hs = 0ull;
                if (HIT) hs = shm[q];
                int up = (rab & 0xffff) - 1;             // rows settled by the edges above
                float jo = a.w - (float)(2 * lane), left = b.x - (float)(2 * lane);
                uint32_t *wp = S.bm + (__float_as_int(b.z) & 0xffff) - 2 * lane;
#pragma unroll 1
                for (;;) {
                    int lo0, hi0, lo1, hi1;
                    crossing(cross_row(G, jo, s, c, c2, tc), a.z, lo0, hi0);
                    crossing(cross_row(G, jo - 1.0f, s, c, c2, tc), a.z, lo1, hi1);
                    const int pv = __shfl_up_sync(kAll, hi1, 1);
                    const int before = lane == 0 ? up : max(pv, up);
                    const int mid = max(hi0, before);
                    if (left > 0.5f) emit(wp, before + 1, min(lo0, rb), jo, hs);
                    if (left > 1.5f) emit(wp - 1, mid + 1, min(lo1, rb), jo - 1.0f, hs);
                    if (hi0 > lo0 || hi1 > lo1) {        // a row within the bound of an edge
                        const int l = __float_as_int(b.z) >> 16, pp = __float_as_int(b.w);
                        if (hi0 > lo0 && left > 0.5f && lo0 >= before && lo0 < rb) push(pp, lo0 + 1, l);
                        if (hi1 > lo1 && left > 1.5f && lo1 >= mid && lo1 < rb) push(pp, lo1 + 1, l);
                    }
                    if (!(__shfl_sync(kAll, left, 31) > 2.5f)) break;   // uniform
                    up = __shfl_sync(kAll, hi1, 31);
                    jo -= 64.0f;
                    left -= 64.0f;
                    wp -= 64;
                }
            }
            __syncwarp();

            // ---- row: lane = row of the window; a lane's bit and the step of its word
            // are the same for all its rows
            // (a band of one word: as many hits per step as their rows fit the lanes;
            // 8 rows, 20k hits: 564 -> 376 us)
            const int lgr = NWB > 1 ? 5 : 32 - __clz(nrow - 1);   // nrow = 1: 0
#pragma unroll 1
            for (int q0 = first[kRow]; q0 < first[kKinds]; q0 += 32 >> lgr) {
                const int q = NWB > 1 ? q0 : q0 + (lane >> lgr);
                if (NWB == 1 && q >= first[kKinds]) continue;
                const float4 a = slot[q].a, b = slot[q].b;
                const int rend = __float_as_int(b.y) >> 16;
                const int sub = NWB > 1 ? lane : lane & ((1 << lgr) - 1);
                int row = (__float_as_int(b.y) & 0xffff) + sub;
                const uint32_t bit = 1u << (row & 31);
                uint32_t *wp = S.bm + (__float_as_int(b.z) & 0xffff) + (row >> 5) * NDp;
                unsigned long long hs = 0ull;
                if (HIT) hs = shm[q];
                auto one = [&](int rw, uint32_t *w) {
                    if (rw > rend) return;
                    const float rho = S.rho[rw];
                    const float D = fmaf(-(rho * rho), a.y, 1.0f);
                    const float den = fmaf(D, rsqrt_approx(D), 1.0f);
                    const float u = fmaf(-(rho * a.z), rcp_approx(den), a.x);
                    const float e = fmaf(fabsf(rho), b.x, a.w);
                    const float lo = __fadd_rd(__fsub_rd(u, e), kMagic);
                    const float hi = __fadd_rd(__fadd_ru(u, e), kMagic);
                    const int j = __float_as_int(lo) - kMagicBits;
                    if (lo == hi) {
                        bool ok = (unsigned)j < (unsigned)ND;
                        if (HIT && ok) {
                            const unsigned sh = S.rowblk[rw];
                            const unsigned bits = (unsigned)((hs >> (sh & 63)) | (hs >> ((sh >> 8) & 63)) |
                                                             (hs >> ((sh >> 16) & 63))) & 0xffu;
                            ok = (bits & S.jmask[j]) != 0u;
                        }
                        if (ok) {
                            atomicOr(w + j, bit);
                            ++my_cast;
                        }
                    } else if (hi >= kMagic && lo < kMagic + (float)ND) {   // not certainly outside
                        push(__float_as_int(b.w), rw, __float_as_int(b.z) >> 16);
                    }
                };
                if (NWB == 1) {
                    one(row, wp);
                    continue;
                }
#pragma unroll 1
                for (int left = rend - (row - lane); left >= 0; left -= 64) {   // uniform
                    one(row, wp);
                    if (left >= 32) one(row + 32, wp + NDp);
                    row += 64;
                    wp += 2 * NDp;
                }
            }
            __syncwarp();

            // ---- item: the general evaluation, lane = row
            const unsigned mi = __ballot_sync(kAll, item);
            if (mi) {
                if (item) {
                    const int q = __popc(mi & ((1u << lane) - 1u));
                    const float sk = G.sn32[k], ck = G.cs32[k];
                    const float xf = H.x[p], yf = H.y[p];
                    const float c = fmaf(xf, ck, yf * sk), s = fmaf(xf, sk, -(yf * ck));
                    const float R1 = fabsf(xf) + fabsf(yf);
                    const float rt = fmaxf(fabsf(S.rho[rest & 0xff]), fabsf(S.rho[rest >> 24])) * 1.0001f;
                    const Item it = make_item(G, s, c, fmaf(xf, xf, yf * yf), R1, rt);
                    slot[q].a = make_float4(it.s, it.c, it.r2, it.eD);
                    slot[q].b = make_float4(it.E1, it.E2, it.Qa, it.Qb);
                    const bool sure = c > (kSafe * 3.0f * kEps) * R1;   // sign of c proven
                    const bool nb = needs_b(G, rt, s, c, 4e-7f * R1);
                    imeta[q] = make_int4((int)rest, (PLANES ? run >> 2 : H.l[p] & 15) |
                                                        (sure ? 32 : 0) | (nb ? 64 : 0), p, 0);
                    if (HIT) shm[q] = hm;
                }
                __syncwarp();
#pragma unroll 1
                for (int q = 0; q < __popc(mi); ++q) {
                    const float4 a = slot[q].a, b = slot[q].b;
                    const int4 m = imeta[q];
                    const Item it{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
                    const unsigned rs = (unsigned)m.x;
                    const int pp = m.z, l = m.y & 15;
                    const bool sure = m.y & 32, nb = m.y & 64;
                    const int ra = rs & 0xff, rA = (rs >> 8) & 0xff, rB = (rs >> 16) & 0xff, rb = rs >> 24;
                    // rows ra .. rA - 1, then rB + 1 .. rb (every row when rA > rB)
                    const int n1 = rA > rB ? rb - ra + 1 : rA - ra, n = rA > rB ? n1 : n1 + rb - rB;
#pragma unroll 1
                    for (int t = lane; t < n; t += 32) {
                        const int row = t < n1 ? ra + t : rB + 1 + (t - n1);
                        const float rho = S.rho[row];
                        const float ir = G.invrho32[i0 + row];   // 0 where rho = 0
                        int jA = -1, jB = -1, res = kRedo;
                        if (sure) {
                            if (nb && ir != 0.0f)
                                res = eval32<true>(G, rho, fabsf(ir) * G.err_scale, ir, it, jA, jB);
                            else
                                res = eval32<false>(G, rho, 0.0f, ir, it, jA, jB);
                        }
                        if (res != kDecided) {
                            push(pp, row, l);
                            continue;
                        }
                        unsigned rbl = 0u;
                        if (HIT) rbl = halo_row_blocks(shm[q], i0 + row, G.n_rho);
                        uint32_t *const wp = word0(l, row >> 5);
                        if (jA >= 0 && (!HIT || (rbl & S.jmask[jA]))) {
                            atomicOr(wp + jA, 1u << (row & 31));
                            ++my_cast;
                        }
                        if (jB >= 0 && (!HIT || (rbl & S.jmask[jB]))) {
                            atomicOr(wp + jB, 1u << (row & 31));
                            ++my_cast;
                        }
                    }
                }
            }
            // ---- the warp's redos, once they fill its lanes (or its last chunk is done)
            __syncwarp();
            if (s_nredo[warp] >= 32) drain();
        }
        __syncthreads();
        // every warp's remaining redos, by all threads
        {
            int n = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) n += min(s_nredo[w], kVrRedo);
#pragma unroll 1
            for (int t = threadIdx.x; t < n; t += kThr) {
                int w = 0, q = t;
                while (q >= min(s_nredo[w], kVrRedo)) q -= min(s_nredo[w++], kVrRedo);
                const int2 d = S.redo[w * kVrRedo + q];
                redo_row(d.x, (d.y & ~kNotCounted) >> 4, d.y & 15, !(d.y & kNotCounted));
            }
        }
        __syncthreads();

        // ---- the counts: carry-save sum of the layers' bits, 32 rows at a time
        for (int t = threadIdx.x; t < NWB * ND; t += kThr) {
            const int w = t / ND, j = t - w * ND, wg = band * NWB + w;
            if (wg >= NW) continue;
            uint32_t n0 = 0, n1 = 0, n2 = 0, n3 = 0, n4 = 0;
            if (!PLANES && l0 > 0) {   // on from the first round's counts
                n0 = S.bm[(kKept * NWB + w) * NDp + j];
                n1 = S.bm[((kKept + 1) * NWB + w) * NDp + j];
                n2 = S.bm[((kKept + 2) * NWB + w) * NDp + j];
                n3 = S.bm[((kKept + 3) * NWB + w) * NDp + j];
#pragma unroll
                for (int l = 0; l < kKept; ++l) {
                    uint32_t x = S.bm[(l * NWB + w) * NDp + j], y;
                    y = n0 & x; n0 ^= x; x = y;
                    y = n1 & x; n1 ^= x; x = y;
                    y = n2 & x; n2 ^= x; x = y;
                    y = n3 & x; n3 ^= x; n4 |= y;
                }
                S.bm[(4 * NWB + w) * NDp + j] = n4;
            } else {
#pragma unroll
                for (int l = 0; l < kRes; ++l) {
                    uint32_t x = S.bm[(l * NWB + w) * NDp + j], y;
                    y = n0 & x; n0 ^= x; x = y;
                    y = n1 & x; n1 ^= x; x = y;
                    y = n2 & x; n2 ^= x; x = y;
                    n3 ^= x;
                }
            }
            if (PLANES) {
                uint32_t *o = reinterpret_cast<uint32_t *>(out) + ((size_t)k * kPlanes * NW + wg) * ND + j;
                const size_t ps = (size_t)NW * ND;
                if (l0 > 0) {   // add to the first round's counts
                    uint32_t a0 = o[0], a1 = o[ps], a2 = o[2 * ps], a3 = o[3 * ps], x, y;
                    x = a0 & n0; n0 ^= a0;
                    y = (a1 & n1) | (x & (a1 ^ n1)); n1 ^= a1 ^ x; x = y;
                    y = (a2 & n2) | (x & (a2 ^ n2)); n2 ^= a2 ^ x; x = y;
                    y = (a3 & n3) | (x & (a3 ^ n3)); n3 ^= a3 ^ x; n4 = y;
                }
                o[0] = n0;
                o[ps] = n1;
                o[2 * ps] = n2;
                o[3 * ps] = n3;
                if (s_full) o[4 * ps] = n4;   // read only where 16 layers hold hits
            } else {   // this thread was the only reader of (l, w, j)
                uint32_t *o = S.bm + w * NDp + j;
                if (l0 == 0 && s_more) o += kKept * NWB * NDp;   // kept for the second round
                o[0] = n0;
                o[NWB * NDp] = n1;
                o[2 * NWB * NDp] = n2;
                o[3 * NWB * NDp] = n3;
            }
        }
        if constexpr (!PLANES) {
            // hits on layers of the second round (uniform over the cluster: every tile
            // looks at all hits): their votes first, then one write of the counts
            if (l0 == 0 && s_more) continue;
            // The accumulator is phi0-fastest: the cluster's eight columns exchange
            // their bit planes through distributed shared memory, and each tile
            // writes an eighth of the (word, bin)s, eight counts of a row at a time
            // (one column at a time would write every 32-byte sector 16 times).
            cg::cluster_group cluster = cg::this_cluster();
            cluster.sync();
            const int q = (int)cluster.block_rank(), k0 = k - q, npair = NWB * ND;
            for (int t = threadIdx.x; t < (npair + kVrCluster - 1) / kVrCluster * 4; t += kThr) {
                const int pr = (t >> 2) * kVrCluster + q, w = pr / ND, j = pr - w * ND;
                const int wg = band * NWB + w;
                if (pr >= npair || wg >= NW) continue;
                uint32_t pl[kVrCluster][4];
#pragma unroll
                for (int v = 0; v < kVrCluster; ++v) {
                    const uint32_t *rb = cluster.map_shared_rank(S.bm, v) + w * NDp + j;
#pragma unroll
                    for (int pp = 0; pp < 4; ++pp) pl[v][pp] = rb[pp * NWB * NDp] >> (8 * (t & 3));
                }
                const int r0 = wg * 32 + 8 * (t & 3), nr = min(8, G.n_rho - r0);
                for (int r = 0; r < nr; ++r) {
                    OutT *d = reinterpret_cast<OutT *>(out) + ((size_t)(r0 + r) * ND + j) * G.n_phi0 + k0;
                    __align__(16) OutT o[kVrCluster];
#pragma unroll
                    for (int v = 0; v < kVrCluster; ++v)
                        o[v] = (OutT)(((pl[v][0] >> r) & 1u) | (((pl[v][1] >> r) & 1u) << 1) |
                                      (((pl[v][2] >> r) & 1u) << 2) | (((pl[v][3] >> r) & 1u) << 3));
                    constexpr int NV = kVrCluster * (int)sizeof(OutT) / 16;
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        reinterpret_cast<uint4 *>(d)[v] = reinterpret_cast<const uint4 *>(o)[v];
                }
                if (l0 > 0) {   // cells of all 16 layers (the other bits are 0)
#pragma unroll 1
                    for (int v = 0; v < kVrCluster; ++v) {
                        uint32_t m = cluster.map_shared_rank(S.bm, v)[(4 * NWB + w) * NDp + j];
                        m = (m >> (8 * (t & 3))) & 0xffu;
                        for (; m; m &= m - 1u) {
                            const size_t cell = (size_t)(r0 + __ffs(m) - 1) * ND + j;
                            reinterpret_cast<OutT *>(out)[cell * G.n_phi0 + k0 + v] = (OutT)16;
                        }
                    }
                }
            }
            cluster.sync();   // the others have read this tile's planes
        }
    }
    if (stats) {
        unsigned long long v = (unsigned long long)(long long)my_cast;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v += __shfl_xor_sync(kAll, v, o);
            my_fb += __shfl_xor_sync(kAll, my_fb, o);
        }
        if (lane == 0) {
            atomicAdd(&s_stats[0], v);
            atomicAdd(&s_stats[1], (unsigned long long)my_fb);
        }
        __syncthreads();
        if (threadIdx.x < 2) atomicAdd(&stats[threadIdx.x], s_stats[threadIdx.x]);
    }
    __syncthreads();
}

// Persistent over the (event, band, column) tiles of a batch's events, in the
// order given (largest first): CELLS the first *d_ncell (dense layers cell by
// cell), else the others up to *d_nev (d_ncell null: all).  out: the events'
// bit planes, out_stride words apart.
template <int NWB, bool HIT, bool CELLS>
__global__ void __launch_bounds__(CELLS ? kClThreads : kVrThreads, CELLS ? 2 : 3)
k_vote_rows_batch(DevGeom G, HitSource H, const int *__restrict__ off,
                  const int *__restrict__ order, const int *__restrict__ d_nev,
                  const int *__restrict__ d_ncell, uint32_t *__restrict__ out, size_t out_stride,
                  unsigned long long *__restrict__ stats, int *__restrict__ head,
                  const unsigned long long *__restrict__ masks)
{
    __shared__ int s_item;
    const int nb = (G.n_rho + 32 * NWB - 1) / (32 * NWB), nt = nb * G.n_phi0;
    const int first = CELLS || !d_ncell ? 0 : *d_ncell;
    const int total = ((CELLS ? *d_ncell : *d_nev) - first) * nt;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(head, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= total) break;
        const int e = order[first + item / nt], t = item % nt;
        vr_tile<NWB, HIT, true, CELLS, CELLS ? kClThreads : kVrThreads, uint16_t>(
            G, H, e, HIT ? masks + off[e] : nullptr, out + (size_t)e * out_stride,
            stats ? stats + 2 * e : nullptr, t % G.n_phi0, t / G.n_phi0);
    }
}

// One event (hits in the caller's order), one CTA per tile, clusters of
// neighbouring columns (n_phi0 is a multiple of 8).
template <int NWB, int kThr, typename OutT>
__global__ void __cluster_dims__(kVrCluster, 1, 1)
__launch_bounds__(kThr, kThr == kVrNarrow ? 4 : 3)
k_vote_rows(DevGeom G, HitSource H, OutT *__restrict__ acc,
            unsigned long long *__restrict__ stats)
{
    vr_tile<NWB, false, false, false, kThr, OutT>(G, H, 0, nullptr, acc, stats, blockIdx.x,
                                                  blockIdx.y);
}

}  // namespace

size_t layer_planes_words(const DevGeom &G)
{
    return (size_t)G.n_phi0 * kPlanes * ((G.n_rho + 31) / 32) * G.n_d0;
}

cudaError_t launch_vote_layers(const DevGeom &G, const float *x, const float *y,
                               const uint8_t *layer, int n, void *acc,
                               unsigned long long *stats, cudaStream_t st)
{
    const HitSource H{x, y, nullptr, layer, nullptr, nullptr, n, nullptr};
    int nwb = vr_nwb(G.n_rho, G.n_d0);
    const long long sms = device_sms();
    auto bands = [&]() { return (G.n_rho + 32 * nwb - 1) / (32 * nwb); };
    // Few columns: narrower bands, until every SM has a tile (each band goes
    // through all hits).  256 rows x 128 bins, 20k hits: 8 columns 362 -> 117 us
    // (4 words of rows to 1), 64 columns 364 -> 186 (to 2).
    while (nwb > 1 && (long long)G.n_phi0 * bands() < sms) nwb /= 2;
    const dim3 grid(G.n_phi0, bands());
    const long long tiles = (long long)grid.x * grid.y;
    const bool narrow = nwb <= 2 && tiles > 3 * sms &&
                        vr_smem(nwb, G.n_d0, false, false, kVrNarrow) <= 50 * 1024;
    const size_t sm = vr_smem(nwb, G.n_d0, false, false, narrow ? kVrNarrow : kVrThreads);
#define HT_VR(N, THR)                                                                         \
    do {                                                                                      \
        if (G.count_bits == 16)                                                               \
            k_vote_rows<N, THR, uint16_t><<<grid, THR, sm, st>>>(                             \
                G, H, reinterpret_cast<uint16_t *>(acc), stats);                              \
        else                                                                                  \
            k_vote_rows<N, THR, int32_t><<<grid, THR, sm, st>>>(                              \
                G, H, reinterpret_cast<int32_t *>(acc), stats);                               \
    } while (0)
    if (nwb == 8) HT_VR(8, kVrThreads);
    else if (nwb == 4) HT_VR(4, kVrThreads);
    else if (nwb == 2 && narrow) HT_VR(2, kVrNarrow);
    else if (nwb == 2) HT_VR(2, kVrThreads);
    else if (narrow) HT_VR(1, kVrNarrow);
    else HT_VR(1, kVrThreads);
#undef HT_VR
    return cudaGetLastError();
}

namespace {

template <int NWB, bool HIT, bool CELLS>
void run_vote_batch(const DevGeom &G, const HitSource &H, const int *off, const int *order,
                    const int *d_nev, const int *d_ncell, uint32_t *planes, size_t stride,
                    unsigned long long *stats, int *head, int sms,
                    const unsigned long long *hit_masks, cudaStream_t st)
{
    constexpr int threads = CELLS ? kClThreads : kVrThreads;
    const size_t sm = vr_smem(NWB, G.n_d0, HIT, CELLS, threads);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_vote_rows_batch<NWB, HIT, CELLS>, threads,
                                                  sm);
    k_vote_rows_batch<NWB, HIT, CELLS><<<sms * (occ > 0 ? occ : 1), threads, sm, st>>>(
        G, H, off, order, d_nev, d_ncell, planes, stride, stats, head, hit_masks);
}

template <int NWB>
cudaError_t run_votes(const DevGeom &G, const HitIndex &I, const int *off, const int *order,
                      const int *d_nev, const int *d_ncell, uint32_t *planes, size_t stride,
                      unsigned long long *stats, int *heads, int sms,
                      const unsigned long long *hit_masks, cudaStream_t st)
{
    const HitSource H{I.x, I.y, I.h, I.l, I.offs, I.rmm, 0, I.unsorted};
    if (hit_masks) {   // a hit's regions restrict its votes: hit by hit
        run_vote_batch<NWB, true, false>(G, H, off, order, d_nev, nullptr, planes, stride, stats,
                                         heads, sms, hit_masks, st);
    } else {
        const cudaError_t e = launch_hit_sort(I, order, d_ncell, sms, st);
        if (e != cudaSuccess) return e;
        run_vote_batch<NWB, false, true>(G, H, off, order, d_nev, d_ncell, planes, stride, stats,
                                         heads, sms, nullptr, st);
        run_vote_batch<NWB, false, false>(G, H, off, order, d_nev, d_ncell, planes, stride, stats,
                                          heads + 1, sms, nullptr, st);
    }
    return cudaGetLastError();
}

}  // namespace

// order lists the batch's events, largest first; the first *d_ncell have at
// least kCellHits hits.  heads: two counters, zero at launch.
cudaError_t launch_vote_batch_layers(const DevGeom &G, const HitIndex &I, const int *off,
                                     const int *order, const int *d_nev, const int *d_ncell,
                                     uint32_t *planes, size_t stride, unsigned long long *stats,
                                     int *heads, int sms, const unsigned long long *hit_masks,
                                     cudaStream_t st)
{
    const int nwb = vr_nwb(G.n_rho, G.n_d0);
#define HT_VRB(N)                                                                             \
    if (nwb == N)                                                                             \
        return run_votes<N>(G, I, off, order, d_nev, d_ncell, planes, stride, stats, heads,   \
                            sms, hit_masks, st)
    HT_VRB(8);
    HT_VRB(4);
    HT_VRB(2);
    HT_VRB(1);
#undef HT_VRB
    return cudaErrorInvalidValue;
}

cudaError_t prepare_layer_vote_kernels(int max_smem)
{
#define HT_VRP(N)                                                                             \
    (const void *)k_vote_rows<N, kVrThreads, uint16_t>,                                       \
        (const void *)k_vote_rows<N, kVrThreads, int32_t>,                                    \
        (const void *)k_vote_rows_batch<N, false, false>,                                     \
        (const void *)k_vote_rows_batch<N, true, false>,                                      \
        (const void *)k_vote_rows_batch<N, false, true>
    const void *fns[] = {HT_VRP(8),
                         HT_VRP(4),
                         HT_VRP(2),
                         HT_VRP(1),
                         (const void *)k_vote_rows<2, kVrNarrow, uint16_t>,
                         (const void *)k_vote_rows<2, kVrNarrow, int32_t>,
                         (const void *)k_vote_rows<1, kVrNarrow, uint16_t>,
                         (const void *)k_vote_rows<1, kVrNarrow, int32_t>};
#undef HT_VRP
    return allow_smem(fns, (int)(sizeof fns / sizeof fns[0]), max_smem);
}

}  // namespace ht
