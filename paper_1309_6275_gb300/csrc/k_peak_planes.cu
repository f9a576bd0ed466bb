// k_peak_planes.cu -- 3x3x3 local maxima of a batch's layer counts, on bit
// planes (Sections 5-7 of arXiv:1309.6275: candidates are the local maxima
// of the vote space), for the batched track path.
//
// The distinct-layer vote leaves an event's counts as bit planes
// (k_vote_rows.cu): one word holds one bit of the counts of 32 rho rows.  A
// bit-sliced maximum of two counts is eight three-input logic operations for
// 32 cells (four for the comparison, four for the choice), so the 26
// comparisons of a cell cost a few instructions instead of one per
// neighbour, and an event's 16.8 M cells are 10.5 MB of planes, read once,
// instead of 33.5 MB.
//
//  * A warp owns a word of rows, 30 d0 bins (lanes 1 .. 30; lanes 0 and 31
//    carry the neighbouring bins) and a segment of kSegCols phi0 columns,
//    which it sweeps.  Row neighbours are funnel shifts with the words above
//    and below, bin neighbours are shuffles, column neighbours are kept from
//    the previous steps.  Of each column it keeps two maxima, over the
//    neighbours that precede a cell in logical index and over those that
//    follow: a cell is a peak when it reaches the threshold, exceeds every
//    preceding neighbour and is at least every following one.
//  * Compaction keeps increasing logical index l = (i n_d0 + j) n_phi0 + k:
//    the sweep writes a word of peak bits per (column, row word, bin) and the
//    peaks per (row, bin, segment); one scan over the batch turns those into
//    positions; a second sweep over the peak bits writes the peaks, each at
//    its segment's position plus its rank, in column order.
//
// Bound by issue and by the latency of the sweep's loads.  Peak stage, GB300,
// 25 events of 256 x 128 x 512 cells: 1.75 -> 0.44 ms (the launches were five
// per event, the stencil 49 us of each event); two of 512 x 256 x 1024: 0.80
// -> 0.29.
#include <cuda_runtime.h>
#include <stdint.h>

#include "ht_internal.cuh"

namespace ht {
namespace {

// Short segments give few events enough warps (one event of 2000 hits: its
// batch 384 us with 128 columns, 321 with 64, 293 with 32); the two columns
// more that a segment reads cost 25 events less than their fuller last wave
// gains (peak stage 512, 436, 444 us).  A row's peaks in a segment fit a byte.
constexpr int kSegCols = 32;
constexpr int kPpWarps = 4, kPpThreads = 32 * kPpWarps;
constexpr int kLaneBins = 30;
constexpr unsigned kAll = 0xffffffffu;

// counts of 32 cells, N bits each
template <int N>
struct Cells {
    uint32_t v[N];
};

template <int N>
__device__ __forceinline__ uint32_t gt(const Cells<N> &a, const Cells<N> &b)
{
    uint32_t g = 0u;
#pragma unroll
    for (int p = 0; p < N; ++p) g = (a.v[p] & ~b.v[p]) | (~(a.v[p] ^ b.v[p]) & g);
    return g;
}

template <int N>
__device__ __forceinline__ Cells<N> vmax(const Cells<N> &a, const Cells<N> &b)
{
    const uint32_t g = gt(a, b);
    Cells<N> r;
#pragma unroll
    for (int p = 0; p < N; ++p) r.v[p] = (g & a.v[p]) | (~g & b.v[p]);
    return r;
}

template <int N>
__device__ __forceinline__ Cells<N> up1(const Cells<N> &a)   // the previous bin's
{
    Cells<N> r;
#pragma unroll
    for (int p = 0; p < N; ++p) r.v[p] = __shfl_up_sync(kAll, a.v[p], 1);
    return r;
}

template <int N>
__device__ __forceinline__ Cells<N> down1(const Cells<N> &a)   // the next bin's
{
    Cells<N> r;
#pragma unroll
    for (int p = 0; p < N; ++p) r.v[p] = __shfl_down_sync(kAll, a.v[p], 1);
    return r;
}

// A column as the sweep keeps it: the counts, and the maxima over the
// neighbours (this column's) that precede and follow a cell.
template <int N>
struct Column {
    Cells<N> v, before, after;
};

// The words a lane loads of a column: its own, the one above, the one below.
template <int N>
struct Raw {
    Cells<N> v, prev, next;
};

struct Task {
    int e, w, j, ks;
    bool bin;   // the lane's bin exists
};

struct PpShape {
    int NR, ND, NP, NW, njg, nks;
};

__host__ __device__ inline PpShape pp_shape(const DevGeom &G)
{
    PpShape s;
    s.NR = G.n_rho;
    s.ND = G.n_d0;
    s.NP = G.n_phi0;
    s.NW = (G.n_rho + 31) / 32;
    s.njg = (G.n_d0 + kLaneBins - 1) / kLaneBins;
    s.nks = (G.n_phi0 + kSegCols - 1) / kSegCols;
    return s;
}

// Task t of a batch (row word fastest, then bins, segments, events).
__device__ __forceinline__ Task task_of(const PpShape &S, long long t, int lane)
{
    Task k;
    k.w = (int)(t % S.NW);
    t /= S.NW;
    k.j = (int)(t % S.njg) * kLaneBins - 1 + lane;
    t /= S.njg;
    k.ks = (int)(t % S.nks);
    k.e = (int)(t / S.nks);
    k.bin = k.j >= 0 && k.j < S.ND;
    return k;
}

// Bits of an event's counts: 5 planes when all 16 layers hold hits, else 4.
__device__ __forceinline__ bool five_planes(const unsigned *__restrict__ rmm, int e, int lane)
{
    const int l = lane & 15;
    return __all_sync(kAll, __uint_as_float(rmm[2 * (e * 16 + l)]) <=
                                __uint_as_float(rmm[2 * (e * 16 + l) + 1]));
}

template <int N>
__device__ __forceinline__ void load_raw(const PpShape &S, const uint32_t *__restrict__ ev,
                                         const Task &T, int k, Raw<N> &r)
{
    const size_t ps = (size_t)S.NW * S.ND;
    const uint32_t *p0 = ev + (size_t)k * kPlanes * ps + (size_t)T.w * S.ND + T.j;
#pragma unroll
    for (int p = 0; p < N; ++p) {
        const uint32_t *q = p0 + p * ps;
        r.v.v[p] = T.bin ? __ldg(q) : 0u;
        r.prev.v[p] = T.bin && T.w > 0 ? __ldg(q - S.ND) : 0u;
        r.next.v[p] = T.bin && T.w < S.NW - 1 ? __ldg(q + S.ND) : 0u;
    }
}

template <int N>
__device__ __forceinline__ void make_column(const Raw<N> &r, Column<N> &c)
{
    Cells<N> u, d;   // the counts one row up (i - 1) and one down
#pragma unroll
    for (int p = 0; p < N; ++p) {
        u.v[p] = __funnelshift_l(r.prev.v[p], r.v.v[p], 1);
        d.v[p] = __funnelshift_r(r.v.v[p], r.next.v[p], 1);
    }
    c.v = r.v;
    c.before = vmax(vmax(u, down1(u)), up1(vmax(u, r.v)));
    c.after = vmax(vmax(d, up1(d)), down1(vmax(d, r.v)));
}

template <int N>
__device__ __forceinline__ void sweep(const PpShape &S, const uint32_t *__restrict__ ev,
                                      uint32_t *__restrict__ flags, const Task &T, int thr,
                                      uint8_t *cnt, int lane)
{
    const int k0 = T.ks * kSegCols, k1 = min(k0 + kSegCols, S.NP);
    const bool mine = T.bin && lane >= 1 && lane <= kLaneBins;
    uint32_t tm[N];
#pragma unroll
    for (int p = 0; p < N; ++p) tm[p] = (thr >> p) & 1 ? kAll : 0u;
    const bool none = thr >= (1 << N);   // above any count
    Column<N> A, B, C;
    Raw<N> r;
    load_raw<N>(S, ev, T, k0 > 0 ? k0 - 1 : S.NP - 1, r);
    make_column(r, A);
    load_raw<N>(S, ev, T, k0, r);
    make_column(r, B);
    load_raw<N>(S, ev, T, k0 + 1 < S.NP ? k0 + 1 : 0, r);
    // peaks of column k, between column k - 1 (a) and column k + 1 (c, made here)
    auto step = [&](int k, const Column<N> &a, const Column<N> &b, Column<N> &c) {
        make_column(r, c);
        int kn = k + 2;
        kn -= kn >= S.NP ? S.NP : 0;
        if (k + 1 < k1) load_raw<N>(S, ev, T, kn, r);
        Cells<N> before = vmax(vmax(a.before, b.before), c.before);
        Cells<N> after = vmax(vmax(a.after, b.after), c.after);
        // the column neighbours of the same row and bin: k - 1 precedes and
        // k + 1 follows, except across the phi0 wrap
        if (k > 0) before = vmax(before, a.v);
        else after = vmax(after, a.v);
        if (k < S.NP - 1) after = vmax(after, c.v);
        else before = vmax(before, c.v);
        uint32_t ge = kAll;
#pragma unroll
        for (int p = 0; p < N; ++p)
            ge = (tm[p] & (b.v.v[p] & ge)) | (~tm[p] & (b.v.v[p] | ge));
        uint32_t pk = none || !mine ? 0u : ge & gt(b.v, before) & ~gt(after, b.v);
        if (mine) flags[((size_t)k * S.NW + T.w) * S.ND + T.j] = pk;
        while (pk) {
            const int i = __ffs(pk) - 1;
            pk &= pk - 1u;
            ++cnt[i * 32 + lane];
        }
    };
    for (int k = k0; k < k1; k += 3) {
        step(k, A, B, C);
        if (k + 1 < k1) step(k + 1, B, C, A);
        if (k + 2 < k1) step(k + 2, C, A, B);
    }
}

__global__ void __launch_bounds__(kPpThreads)
k_plane_peaks(DevGeom G, const uint32_t *__restrict__ planes, size_t stride, size_t flag_at,
              const unsigned *__restrict__ rmm, const int *__restrict__ thr, int e0, int n_ev,
              int *__restrict__ segcnt)
{
    __shared__ uint8_t s_cnt[kPpWarps][32 * 32];
    const PpShape S = pp_shape(G);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t = (long long)blockIdx.x * kPpWarps + warp;
    if (t >= (long long)n_ev * S.NW * S.njg * S.nks) return;
    const Task T = task_of(S, t, lane);
    const int e = e0 + T.e;
    uint8_t *cnt = s_cnt[warp];
    for (int i = 0; i < 32; ++i) cnt[i * 32 + lane] = 0;
    const uint32_t *ev = planes + (size_t)e * stride;
    uint32_t *flags = const_cast<uint32_t *>(ev) + flag_at;
    if (five_planes(rmm, e, lane)) sweep<5>(S, ev, flags, T, thr[e], cnt, lane);
    else sweep<4>(S, ev, flags, T, thr[e], cnt, lane);
    if (!T.bin || lane < 1 || lane > kLaneBins) return;
    for (int r = 0; r < min(32, S.NR - 32 * T.w); ++r)
        segcnt[(((size_t)T.e * S.NR + 32 * T.w + r) * S.ND + T.j) * S.nks + T.ks] =
            cnt[r * 32 + lane];
}

__global__ void __launch_bounds__(kPpThreads)
k_plane_write(DevGeom G, const uint32_t *__restrict__ planes, size_t stride, size_t flag_at,
              const unsigned *__restrict__ rmm, int e0, int n_ev,
              const int *__restrict__ segoff, ht_peak *__restrict__ peaks, int cap,
              int *__restrict__ counts)
{
    __shared__ uint8_t s_cnt[kPpWarps][32 * 32];
    const PpShape S = pp_shape(G);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t = (long long)blockIdx.x * kPpWarps + warp;
    const long long per = (long long)S.NW * S.njg * S.nks;
    if (t >= n_ev * per) return;
    const Task T = task_of(S, t, lane);
    const int e = e0 + T.e;
    const size_t nseg = (size_t)S.NR * S.ND * S.nks;
    const int first = segoff[T.e * nseg];
    if (t % per == 0 && lane == 0) counts[e] = segoff[(T.e + 1) * nseg] - first;
    uint8_t *cnt = s_cnt[warp];
    for (int i = 0; i < 32; ++i) cnt[i * 32 + lane] = 0;
    const uint32_t *ev = planes + (size_t)e * stride;
    const uint32_t *flags = ev + flag_at;
    const int np = five_planes(rmm, e, lane) ? 5 : 4;
    if (!T.bin || lane < 1 || lane > kLaneBins) return;
    const size_t ps = (size_t)S.NW * S.ND, at = (size_t)T.w * S.ND + T.j;
    const int k0 = T.ks * kSegCols, k1 = min(k0 + kSegCols, S.NP);
    constexpr int U = 8;   // words in flight; n_phi0 is a multiple of 8
    for (int kb = k0; kb < k1; kb += U) {
        uint32_t f[U];
#pragma unroll
        for (int q = 0; q < U; ++q) f[q] = __ldg(flags + (kb + q) * ps + at);
#pragma unroll
        for (int q = 0; q < U; ++q) {
            uint32_t pk = f[q];
            while (pk) {
                const int r = __ffs(pk) - 1, k = kb + q, i = 32 * T.w + r;
                pk &= pk - 1u;
                const int pos = segoff[(((size_t)T.e * S.NR + i) * S.ND + T.j) * S.nks + T.ks] -
                                first + cnt[r * 32 + lane]++;
                if (pos >= cap) continue;
                int v = 0;
                for (int p = 0; p < np; ++p)
                    v |= (int)((ev[((size_t)k * kPlanes + p) * ps + at] >> r) & 1u) << p;
                peaks[(size_t)e * cap + pos] = ht_peak{i, T.j, k, v};
            }
        }
    }
}

// Events per scan: their segment counts stay far below 2^31.
int pp_group(const DevGeom &G, int max_events)
{
    const PpShape S = pp_shape(G);
    const size_t nseg = (size_t)S.NR * S.ND * S.nks;
    const size_t g = ((size_t)1 << 28) / nseg;
    return (int)(g < 1 ? 1 : g < (size_t)max_events ? g : (size_t)max_events);
}

}  // namespace

// Segment counts and offsets of one group of events, and the scan's scratch.
size_t plane_peaks_bytes(const DevGeom &G, int max_events)
{
    const PpShape S = pp_shape(G);
    const size_t n = (size_t)S.NR * S.ND * S.nks * pp_group(G, max_events);
    return 2 * align256((n + 1) * 4) + scan_tmp_bytes((int)n);
}

size_t plane_flag_words(const DevGeom &G)
{
    return (size_t)G.n_phi0 * ((G.n_rho + 31) / 32) * G.n_d0;
}

cudaError_t launch_plane_peaks(const DevGeom &G, const uint32_t *planes, size_t stride,
                               const unsigned *rmm, const int *thr, int n_ev, int max_events,
                               ht_peak *peaks, int cap, int *counts, void *ws, cudaStream_t st)
{
    const PpShape S = pp_shape(G);
    const size_t nseg = (size_t)S.NR * S.ND * S.nks, flag_at = layer_planes_words(G);
    const int g = pp_group(G, max_events);
    char *p = reinterpret_cast<char *>(ws);
    int *segcnt = reinterpret_cast<int *>(p);
    int *segoff = reinterpret_cast<int *>(p + align256((nseg * g + 1) * 4));
    void *tmp = p + 2 * align256((nseg * g + 1) * 4);
    for (int e0 = 0; e0 < n_ev; e0 += g) {
        const int ne = n_ev - e0 < g ? n_ev - e0 : g;
        const long long tasks = (long long)ne * S.NW * S.njg * S.nks;
        const unsigned grid = (unsigned)((tasks + kPpWarps - 1) / kPpWarps);
        k_plane_peaks<<<grid, kPpThreads, 0, st>>>(G, planes, stride, flag_at, rmm, thr, e0, ne,
                                                   segcnt);
        const cudaError_t e = scan_exclusive(segcnt, segoff, nullptr, (int)(nseg * ne), nullptr,
                                             nullptr, tmp, st);
        if (e != cudaSuccess) return e;
        k_plane_write<<<grid, kPpThreads, 0, st>>>(G, planes, stride, flag_at, rmm, e0, ne, segoff,
                                                   peaks, cap, counts);
    }
    return cudaGetLastError();
}

}  // namespace ht
