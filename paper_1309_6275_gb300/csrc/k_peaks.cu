// k_peaks.cu -- 3x3x3 local-maximum peak finding over the accumulator with
// order-preserving compaction (Sections 5-7 of arXiv:1309.6275: candidates
// are the local maxima of the vote space; the threshold reflects the peak
// finder's tuning for tracks of at least seven hits).
//
// Design (GB300):
//  * A CTA of 256 threads owns one tile: 16 d0 bins x 256 phi0 columns of a
//    rho row.  It reads the tile's own cells with 16-byte loads and counts
//    those at or above the threshold.  Few events fill their accumulator, so
//    most tiles hold none (a 400-hit event: 45%, and 5 cells on average): such
//    a tile costs one read of its cells.
//  * Up to kSparse such cells: a thread per cell compares it with its 26
//    neighbours, read where they lie (cached lines of tiles next to it).
//  * More: the CTA stages rows i-1..i+1 x bins j0-1..j0+16 x its columns plus
//    one wrapped column on each side in shared memory, all loads issued
//    before any is used; absent rows and bins read as 0.  Then thread = phi0
//    column walks the bins keeping, per row and bin of the rolling 3 x 3 x 3
//    window, the largest of its three columns (9 shared loads and 3
//    three-input maxima per cell); the 26 comparisons become two against the
//    maxima of the preceding and of the following neighbours.  About 100
//    instructions per cell: the instruction rate bounds it.
//  * Compaction keeps increasing logical index l = (i n_d0 + j) n_phi0 + k:
//    the tile leaves a bit per cell and the count of each (i, j, block of 256
//    columns) segment, a device-wide scan turns the counts into offsets (and
//    the total), and a second kernel writes each bit's peak at its segment's
//    offset plus its rank.  Segments are ordered by l, so the output is too.
//    A caller whose scratch has no room for the bits gets the tile kernel
//    again as its second one, writing instead of counting.
//  * Several events (a batch's, a vertex search's) take one launch of each
//    kernel: the event is a grid dimension.
// Measured: 25 events of 400 hits, 256 x 128 x 512 uint16 counts (0.84 GB):
// tiles 322 us + write 22 us (every tile staged and walked, a launch per
// event: 1109 + 157 us).  One event of 10k hits (87% of the cells at or above
// the threshold, all staged) pays the walk once instead of twice: 99 -> about
// 50 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include "ht_internal.cuh"

namespace ht {

constexpr int kPkThreads = 256;   // phi0 columns per CTA

namespace {

constexpr int kJB = 16;                         // d0 bins per CTA
constexpr int kSlices = 3 * (kJB + 2);          // staged (row, bin) slices

// A staged slice holds the CTA's columns at [kOff, kOff + 256) -- 16-byte
// aligned, so a 16-byte global load lands in one 16-byte shared store --
// with the wrapped neighbour columns at kOff - 1 and kOff + ncol.
template <typename T>
struct Stage {
    static constexpr int kOff = 16 / (int)sizeof(T);
    static constexpr int kSW = kPkThreads + 2 * kOff;   // elements per slice
    static constexpr size_t kBytes = (size_t)kSlices * kSW * sizeof(T);
};
constexpr size_t kPkSmemMax = Stage<int32_t>::kBytes;

constexpr int kFlagWords = kPkThreads / 32;     // peak bits of a segment
// Cells compared one by one, at most: 128, 256, 384 and 510 cells of a tile's 4096
// take 46, 58, 61 and 71 us (256 x 128 x 512 uint16 cells; 62, 76, 82 and 96 int32),
// staging the window 77 (105) however many.
constexpr int kSparse = 512;

// Count pass: tile (rho row i, 16 d0 bins from j0, 256 phi0 columns from k0)
// of event e; the peak bits (flags given) and the segment counts.  Scratch of event e lies
// e * ws_stride bytes after event 0's.
//
// MASKED: only cells inside masks[e] (a learned proposal's regions) can be
// peaks; a tile whose bins are all outside reads nothing.  An inside cell's
// 26 neighbours lie in the mask's halo, which the masked vote fills exactly.
// WRITE: the second pass without peak bits; seg holds the segments' offsets
// and the peaks go to out.
template <typename T, bool MASKED, bool WRITE>
__global__ void __launch_bounds__(kPkThreads)
k_peaks_tile(DevGeom G, const T *__restrict__ acc, size_t acc_stride, int *__restrict__ segs,
             uint32_t *__restrict__ flags, size_t ws_stride,
             const unsigned long long *__restrict__ masks, ht_peak *__restrict__ out, int cap)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint32_t s_flag[kJB][kFlagWords];
    __shared__ int s_n, s_at;
    __shared__ uint16_t s_hot[kSparse];
    constexpr int kOff = Stage<T>::kOff, kSW = Stage<T>::kSW;
    T *const sw = reinterpret_cast<T *>(smraw);
    const int NP = G.n_phi0, ND = G.n_d0, NR = G.n_rho, thr = G.threshold;
    const int nkb = (NP + kPkThreads - 1) / kPkThreads;
    const int kb = blockIdx.x % nkb, jb = blockIdx.x / nkb, i = blockIdx.y, e = blockIdx.z;
    acc += e * acc_stride;
    segs = reinterpret_cast<int *>(reinterpret_cast<char *>(segs) + e * ws_stride);
    if (flags)
        flags = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(flags) + e * ws_stride);
    const int k0 = kb * kPkThreads, ncol = min(kPkThreads, NP - k0);
    const int j0 = jb * kJB, j1 = min(j0 + kJB, ND), nj = j1 - j0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned inside = 0xffu;   // d0 blocks inside the mask in row i's rho block
    bool any = true;
    if (MASKED) {
        inside = (unsigned)(masks[e] >> (8 * region_block(i, NR))) & 0xffu;
        const int b0 = region_block(j0, ND), b1 = region_block(j1 - 1, ND);
        any = (inside & ((2u << b1) - 1u) & ~((1u << b0) - 1u)) != 0u;
    }
    if (threadIdx.x < kJB * kFlagWords) (&s_flag[0][0])[threadIdx.x] = 0u;
    if (threadIdx.x == 0) s_n = s_at = 0;
    __syncthreads();

    // ---- the tile's own cells, and which of them reach the threshold
    constexpr int VEC = 16 / (int)sizeof(T), kRowVec = kPkThreads / VEC, NV = kJB / VEC;
    uint4 u[NV];
    unsigned hot[NV];
#pragma unroll
    for (int n = 0; n < NV; ++n) {
        const int v = threadIdx.x + n * kPkThreads, jl = v / kRowVec, q = v % kRowVec;
        u[n] = make_uint4(0, 0, 0, 0);
        if (any && jl < nj && q * VEC < ncol)            // ncol is a multiple of 8
            u[n] = *reinterpret_cast<const uint4 *>(acc + ((size_t)i * ND + j0 + jl) * NP + k0 +
                                                    q * VEC);
    }
    int nhot = 0;
#pragma unroll
    for (int n = 0; n < NV; ++n) {
        const uint32_t w[4] = {u[n].x, u[n].y, u[n].z, u[n].w};
        const int jl = (threadIdx.x + n * kPkThreads) / kRowVec;
        hot[n] = 0u;
#pragma unroll
        for (int b = 0; b < VEC; ++b) {
            const int c = sizeof(T) == 2 ? (int)((w[b >> 1] >> (16 * (b & 1))) & 0xffffu)
                                         : (int)w[b & 3];
            hot[n] |= (unsigned)(c >= thr) << b;
        }
        if (MASKED && jl < nj && !((inside >> region_block(j0 + jl, ND)) & 1u)) hot[n] = 0u;
        nhot += __popc(hot[n]);
    }
    const int wsum = __reduce_add_sync(0xffffffffu, nhot);
    if (lane == 0 && wsum) atomicAdd(&s_n, wsum);
    __syncthreads();
    const int total = s_n;
    if (total > 0 && total <= kSparse) {
        // ---- few: list them, a thread each
        if (nhot) {
            int at = atomicAdd(&s_at, nhot);
#pragma unroll
            for (int n = 0; n < NV; ++n)
                for (unsigned h = hot[n]; h; h &= h - 1u)
                    s_hot[at++] =
                        (uint16_t)((threadIdx.x + n * kPkThreads) * VEC + __ffs(h) - 1);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < total; t += kPkThreads) {
            const int jl = s_hot[t] / kPkThreads, c = s_hot[t] % kPkThreads;
            const int j = j0 + jl, k = k0 + c;
            const int km = k == 0 ? NP - 1 : k - 1, kp = k == NP - 1 ? 0 : k + 1;
            auto row = [&](int ii, int jj, int &a, int &m, int &b) {
                a = m = b = 0;
                if (ii < 0 || ii >= NR || jj < 0 || jj >= ND) return;
                const T *r = acc + ((size_t)ii * ND + jj) * NP;
                a = (int)r[km];
                m = (int)r[k];
                b = (int)r[kp];
            };
            int a[9], m[9], b[9];
#pragma unroll
            for (int r = 0; r < 9; ++r) row(i - 1 + r / 3, j - 1 + r % 3, a[r], m[r], b[r]);
            int before = 0, after = 0;
#pragma unroll
            for (int r = 0; r < 4; ++r) before = max(before, __vimax3_s32(a[r], m[r], b[r]));
#pragma unroll
            for (int r = 5; r < 9; ++r) after = max(after, __vimax3_s32(a[r], m[r], b[r]));
            // the column neighbours of the own bin: across the wrap their order flips
            before = __vimax3_s32(before, k == 0 ? 0 : a[4], k == NP - 1 ? b[4] : 0);
            after = __vimax3_s32(after, k == 0 ? a[4] : 0, k == NP - 1 ? 0 : b[4]);
            if (m[4] > before && m[4] >= after) atomicOr(&s_flag[jl][c >> 5], 1u << (c & 31));
        }
    } else if (total > 0) {
        // ---- many: stage the window, the own cells from the registers
#pragma unroll
        for (int n = 0; n < NV; ++n) {
            const int v = threadIdx.x + n * kPkThreads, jl = v / kRowVec, q = v % kRowVec;
            if (jl < nj && q * VEC < ncol)
                *reinterpret_cast<uint4 *>(sw + (kJB + 2 + jl + 1) * kSW + kOff + q * VEC) = u[n];
        }
        // Absent rows and bins read as 0: a peak has v >= threshold >= 1, so a 0
        // neighbour never decides a comparison (as no neighbour at all).
        const int nvec = ncol / VEC;
        for (int v = threadIdx.x; v < kSlices * nvec; v += kPkThreads) {
            const int sl = v / nvec, q = v - sl * nvec;
            const int r = sl / (kJB + 2), jj = j0 - 1 + sl % (kJB + 2), ii = i - 1 + r;
            if (r == 1 && jj >= j0 && jj < j1) continue;
            uint4 w = make_uint4(0, 0, 0, 0);
            if (ii >= 0 && ii < NR && jj >= 0 && jj < ND)
                w = *reinterpret_cast<const uint4 *>(acc + ((size_t)ii * ND + jj) * NP + k0 +
                                                     q * VEC);
            *reinterpret_cast<uint4 *>(sw + sl * kSW + kOff + q * VEC) = w;
        }
        // the two wrapped neighbour columns of every slice
        for (int v = threadIdx.x; v < 2 * kSlices; v += kPkThreads) {
            const int sl = v >> 1, side = v & 1;
            const int ii = i - 1 + sl / (kJB + 2), jj = j0 - 1 + sl % (kJB + 2);
            const int kk = side ? (k0 + ncol) % NP : (k0 + NP - 1) % NP;
            const bool ok = ii >= 0 && ii < NR && jj >= 0 && jj < ND;
            sw[sl * kSW + (side ? kOff + ncol : kOff - 1)] =
                ok ? acc[((size_t)ii * ND + jj) * NP + kk] : (T)0;
        }
        __syncthreads();

        // ---- walk the bins.  cm[r][s]: largest of columns k-1, k, k+1 in row
        // i-1+r at bin j-1+s; c1/n1: the three columns of row i at bins j and
        // j+1.  A cell is a peak when v >= T, v exceeds every neighbour that
        // precedes it in l (row i-1, bin j-1 of row i, column k-1 of its own
        // bin) and is at least every neighbour that follows it (row i+1, bin j+1,
        // column k+1) -- the two maxima below; across the phi0 wrap the order of
        // the column neighbours flips.
        const int c = threadIdx.x;
        const bool cok = c < ncol;
        const int k = k0 + c;
        const int cc = cok ? c : 0;                           // stays inside the staged row
        // q[-1], q[0], q[1]: columns k - 1, k, k + 1 of slice (r, jj)
        auto S = [&](int r, int jj) -> const T * {
            return sw + (r * (kJB + 2) + jj) * kSW + kOff + cc;
        };
        int cm[3][3], c1[3], n1[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int sl = 0; sl < 2; ++sl) {
                const T *q = S(r, sl);
                const int a = (int)q[-1], b = (int)q[0], d = (int)q[1];
                cm[r][sl] = __vimax3_s32(a, b, d);
                if (r == 1 && sl == 1) { c1[0] = a; c1[1] = b; c1[2] = d; }
            }
        const bool wrap_lo = k == 0, wrap_hi = k == NP - 1;
#pragma unroll
        for (int jl = 0; jl < kJB; ++jl) {
            if (jl < nj) {   // uniform over the CTA
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const T *q = S(r, jl + 2);
                    const int a = (int)q[-1], b = (int)q[0], d = (int)q[1];
                    cm[r][2] = __vimax3_s32(a, b, d);
                    if (r == 1) { n1[0] = a; n1[1] = b; n1[2] = d; }
                }
                const int v = c1[1];
                const int before = max(__vimax3_s32(cm[0][0], cm[0][1], cm[0][2]),
                                       __vimax3_s32(cm[1][0], wrap_lo ? 0 : c1[0],
                                                    wrap_hi ? c1[2] : 0));
                const int after = max(__vimax3_s32(cm[2][0], cm[2][1], cm[2][2]),
                                      __vimax3_s32(cm[1][2], wrap_lo ? c1[0] : 0,
                                                   wrap_hi ? 0 : c1[2]));
                const bool pk = cok && v >= thr && v > before && v >= after &&
                                (!MASKED || ((inside >> region_block(j0 + jl, ND)) & 1u));
                const unsigned bal = __ballot_sync(0xffffffffu, pk);
                if (lane == 0) s_flag[jl][warp] = bal;
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    cm[r][0] = cm[r][1];
                    cm[r][1] = cm[r][2];
                }
                c1[0] = n1[0]; c1[1] = n1[1]; c1[2] = n1[2];
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < nj * kFlagWords) {   // whole groups of kFlagWords lanes
        const int jl = threadIdx.x / kFlagWords, w = threadIdx.x % kFlagWords;
        const size_t seg = ((size_t)i * ND + j0 + jl) * nkb + kb;
        const uint32_t f = s_flag[jl][w];
        const unsigned grp = 0xffu << (lane & ~7);
        int incl = __popc(f);
#pragma unroll
        for (int o = 1; o < kFlagWords; o <<= 1) {
            const int below = __shfl_up_sync(grp, incl, o, kFlagWords);
            if (w >= o) incl += below;
        }
        if (WRITE) {
            const int j = j0 + jl;
            int pos = segs[seg] + incl - __popc(f);
            for (uint32_t b = f; b; b &= b - 1u, ++pos) {
                const int k = k0 + 32 * w + __ffs(b) - 1;
                if (pos < cap)
                    out[(size_t)e * cap + pos] =
                        ht_peak{i, j, k, (int)acc[((size_t)i * ND + j) * NP + k]};
            }
        } else {
            if (flags) flags[seg * kFlagWords + w] = f;
            if (w == kFlagWords - 1) segs[seg] = incl;
        }
    }
}
static_assert(kFlagWords == 8, "the groups of eight lanes above");

// Write pass from the bits: a thread per half segment.
template <typename T>
__global__ void __launch_bounds__(kPkThreads)
k_peaks_write(DevGeom G, const T *__restrict__ acc, size_t acc_stride,
              const int *__restrict__ segoff, const uint32_t *__restrict__ flags,
              size_t ws_stride, int nseg, ht_peak *__restrict__ out, int cap)
{
    const int e = blockIdx.y, t = blockIdx.x * kPkThreads + threadIdx.x;
    const int seg = t >> 1, half = t & 1;
    acc += e * acc_stride;
    segoff = reinterpret_cast<const int *>(reinterpret_cast<const char *>(segoff) + e * ws_stride);
    flags = reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(flags) + e * ws_stride);
    out += (size_t)e * cap;
    uint4 f = make_uint4(0, 0, 0, 0);
    if (seg < nseg) f = reinterpret_cast<const uint4 *>(flags)[t];
    const int mine = __popc(f.x) + __popc(f.y) + __popc(f.z) + __popc(f.w);
    const int other = __shfl_xor_sync(0xffffffffu, mine, 1);
    if (!mine) return;
    int pos = segoff[seg] + (half ? other : 0);
    const int nkb = (G.n_phi0 + kPkThreads - 1) / kPkThreads;
    const int r = seg / nkb, i = r / G.n_d0, j = r - i * G.n_d0;
    const int k0 = (seg - r * nkb) * kPkThreads + half * 128;
    const uint32_t w[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
        for (uint32_t b = w[q]; b; b &= b - 1u, ++pos) {
            const int k = k0 + 32 * q + __ffs(b) - 1;
            if (pos < cap) out[pos] = ht_peak{i, j, k, (int)acc[(size_t)r * G.n_phi0 + k]};
        }
}

template <typename T, bool MASKED>
cudaError_t run_peaks(const DevGeom &G, const T *acc, size_t acc_stride, int n_ev, ht_peak *peaks,
                      int cap, int *d_count, void *ws, size_t ws_stride, bool with_flags,
                      const unsigned long long *masks, cudaStream_t st)
{
    const int nkb = (G.n_phi0 + kPkThreads - 1) / kPkThreads;
    const int njb = (G.n_d0 + kJB - 1) / kJB;
    const int nseg = G.n_rho * G.n_d0 * nkb;
    char *p = reinterpret_cast<char *>(ws);
    int *segcnt = reinterpret_cast<int *>(p);
    p += align256(((size_t)nseg + 1) * 4);
    int *segoff = reinterpret_cast<int *>(p);
    p += align256(((size_t)nseg + 1) * 4);
    void *const tmp = p;
    uint32_t *flags =
        with_flags ? reinterpret_cast<uint32_t *>(p + scan_tmp_bytes(nseg)) : nullptr;
    const dim3 grid(nkb * njb, G.n_rho, n_ev);
    k_peaks_tile<T, MASKED, false><<<grid, kPkThreads, Stage<T>::kBytes, st>>>(
        G, acc, acc_stride, segcnt, flags, ws_stride, masks, nullptr, 0);
    const cudaError_t e = scan_exclusive_batch(segcnt, ws_stride, segoff, ws_stride, nullptr, nseg,
                                               n_ev, d_count, tmp, ws_stride, st);
    if (e != cudaSuccess) return e;
    if (flags) {
        const dim3 wgrid((2 * nseg + kPkThreads - 1) / kPkThreads, n_ev);
        k_peaks_write<T><<<wgrid, kPkThreads, 0, st>>>(G, acc, acc_stride, segoff, flags,
                                                       ws_stride, nseg, peaks, cap);
    } else {
        k_peaks_tile<T, MASKED, true><<<grid, kPkThreads, Stage<T>::kBytes, st>>>(
            G, acc, acc_stride, segoff, nullptr, ws_stride, masks, peaks, cap);
    }
    return cudaGetLastError();
}

}  // namespace

// The staged window needs more than the default 48 KB of dynamic shared
// memory.  Called once per device.
cudaError_t prepare_peaks_kernels()
{
#define HT_PKF(T)                                                                             \
    (const void *)k_peaks_tile<T, false, false>, (const void *)k_peaks_tile<T, true, false>,  \
        (const void *)k_peaks_tile<T, false, true>, (const void *)k_peaks_tile<T, true, true>
    const void *fns[] = {HT_PKF(uint16_t), HT_PKF(int32_t)};
#undef HT_PKF
    for (const void *f : fns) {
        const cudaError_t e =
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPkSmemMax);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static size_t peak_segments(const DevGeom &G)
{
    return (size_t)G.n_rho * G.n_d0 * ((G.n_phi0 + kPkThreads - 1) / kPkThreads);
}

size_t peaks_workspace_bytes(const DevGeom &G)
{
    const size_t nseg = peak_segments(G);
    return 2 * align256((nseg + 1) * 4) + scan_tmp_bytes((int)nseg);
}

size_t peaks_flag_bytes(const DevGeom &G) { return align256(peak_segments(G) * kFlagWords * 4); }

cudaError_t launch_peaks(const DevGeom &G, const void *acc, size_t acc_stride, int n_ev,
                         ht_peak *peaks, int cap, int *d_count, void *ws, size_t ws_stride,
                         size_t ws_bytes, cudaStream_t st, const unsigned long long *masks)
{
    const bool flags = ws_bytes >= peaks_workspace_bytes(G) + peaks_flag_bytes(G);
    const uint16_t *a16 = reinterpret_cast<const uint16_t *>(acc);
    const int32_t *a32 = reinterpret_cast<const int32_t *>(acc);
#define HT_PK(T, M, a)                                                                        \
    run_peaks<T, M>(G, a, acc_stride, n_ev, peaks, cap, d_count, ws, ws_stride, flags, masks, st)
    if (G.count_bits == 16)
        return masks ? HT_PK(uint16_t, true, a16) : HT_PK(uint16_t, false, a16);
    return masks ? HT_PK(int32_t, true, a32) : HT_PK(int32_t, false, a32);
#undef HT_PK
}

}  // namespace ht

// ---------------------------------------------------------------------------
// Peak finding without any allocation (ht_find_peaks_noalloc in ht.h).
//
// The scratch that ht_find_peaks takes from the caller's workspace -- one
// count and one offset per (rho row, d0 bin, phi0 block of 256) segment plus
// the scan's block sums -- lives here in a file-scope device array, sized
// for at most kNoallocMaxSegments segments.  Every GPU that loads the library
// holds it until the process exits.  The array's name is only a host-side
// stand-in in host code, so its device address is looked up per device with
// cudaGetSymbolAddress (on the first successful call made with that device
// current; a failed lookup is not cached, so the next call tries again) and
// passed to the kernels.  Nothing in it needs clearing between calls: each
// word a call reads was written earlier in the same call.
#include <mutex>

namespace {

constexpr int kNoallocMaxSegments = 1 << 19;
constexpr size_t kNoallocSegBytes = ht::align256(((size_t)kNoallocMaxSegments + 1) * 4);
constexpr size_t kNoallocScratchBytes =
    2 * kNoallocSegBytes + ht::align256(((size_t)kNoallocMaxSegments / 4096 + 2) * 4);
constexpr int kNoallocMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

std::mutex g_noalloc_mutex;
void *g_noalloc_ptr[kNoallocMaxDevices];   // null until a lookup on that device succeeds

}  // namespace

extern "C" ht_status ht_find_peaks_noalloc(const ht_geometry *g, const void *acc, ht_peak *peaks,
                                           int32_t cap, int32_t *d_count, ht_stream stream)
{
    if (!g || !acc || !d_count || (cap > 0 && !peaks))
        return ht::set_error(HT_ERR_ARG, "ht_find_peaks_noalloc: null argument");
    if (cap < 0) return ht::set_error(HT_ERR_ARG, "ht_find_peaks_noalloc: cap < 0");
    if (reinterpret_cast<uintptr_t>(acc) % 16 != 0)
        return ht::set_error(HT_ERR_ARG, "ht_find_peaks_noalloc: accumulator not 16-byte aligned");
    const size_t nkb = (g->G.n_phi0 + ht::kPkThreads - 1) / ht::kPkThreads;
    const size_t nseg = (size_t)g->G.n_rho * g->G.n_d0 * nkb;
    if (nseg > (size_t)kNoallocMaxSegments)
        return ht::set_error(HT_ERR_CAPACITY,
                             "ht_find_peaks_noalloc: geometry has more than 524288 segments "
                             "(n_rho * n_d0 * ceil(n_phi0 / 256)); use ht_find_peaks");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return ht::set_error(HT_ERR_CUDA, "ht_find_peaks_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= kNoallocMaxDevices)
        return ht::set_error(HT_ERR_ARG, "ht_find_peaks_noalloc: device index above 63");
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
                cudaGetLastError();   // clear it: the next call looks the address up again
                return ht::set_error(HT_ERR_CUDA, "ht_find_peaks_noalloc: cudaGetSymbolAddress "
                                                  "of the scratch failed (retried next call)");
            }
            g_noalloc_ptr[dev] = p;
        }
        scratch = g_noalloc_ptr[dev];
    }
    e = ht::launch_peaks(g->G, acc, 0, 1, peaks, cap, d_count, scratch, 0, 0,
                         reinterpret_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return ht::set_error(HT_ERR_CUDA, cudaGetErrorString(e));
    return HT_OK;
}
