// k_votez.cu -- per-candidate (z0, cot theta) vote.
//
// The paper works in the transverse plane only (Section 5's detector model);
// this second vote completes each candidate along z.  Reading: at the
// candidate's cell centres the arc length to a hit is L = theta / rho with
// theta = atan2(rho c, 1 + rho (s + d0)); each hit votes z0 = z - L t_q for
// every cot-theta centre t_q; the result is the histogram's maximum cell,
// ties to the smallest n n_cot + q.
//
// Design (GB300):
//  * Hits are grouped by candidate in device memory, so every candidate
//    reads only its own hits.  Their order and place do not matter, so a
//    candidate with hits takes its range from one running total (a warp's
//    candidates together) instead of a scan over every candidate slot, and
//    candidates without hits are settled there.  Single events and batches
//    share the kernels (global candidate id e * cap + m).
//  * Candidates with at most 32 hits (nearly all): one warp per candidate.
//    Lane = hit computes the arc length; then lane = cot column: a lane bins
//    all the candidate's hits in its columns and counts equal bins by
//    comparing them pairwise (45 comparisons for ten hits), so the 128
//    columns are four independent rounds instead of 128 warp-wide matches in
//    a row.  The float64 arc lengths, where any bin needs them, are computed
//    for all hits at once (lane = hit); a bin's float64 quotient is a product
//    unless that lies within 1e-9 of an integer.
//  * Latency-bound.  Stage on GB300, 25 events of 2k-60k hits: 337 -> 84 us
//    (most of it was the scan and a warp per empty candidate slot); 25 of 10k
//    hits: 538 -> 150 us.
//  * Larger candidates: one CTA per candidate with an n_z0 x n_cot uint32
//    histogram in shared memory and a block argmax.
//  * Arithmetic: float32 with a proven error bound per (hit, q); any bin
//    coordinate within its bound of an edge is redone in float64 in the
//    definition's order with the basic-operation atan2, so every vote
//    matches the float64 definition bit for bit.
#include <cuda_runtime.h>
#include <stdint.h>

#include "ht_internal.cuh"

namespace ht {

size_t z_big_smem(const DevGeom &G) { return (size_t)G.n_z0 * G.n_cot * 4; }

namespace {

constexpr int kBigThreads = 256;

struct ZCand {
    float rho, invrho, sn, cs, d0c;
    double rho64, sn64, cs64, d0c64;
    bool rho0;
};

__device__ __forceinline__ ZCand z_cand(const DevGeom &G, const ht_peak &p)
{
    ZCand c;
    c.rho = G.rho32[p.i_rho];
    c.invrho = G.invrho32[p.i_rho];
    c.sn = G.sn32[p.k_phi0];
    c.cs = G.cs32[p.k_phi0];
    c.rho64 = G.rho64[p.i_rho];
    c.sn64 = G.sn64[p.k_phi0];
    c.cs64 = G.cs64[p.k_phi0];
    c.d0c64 = __dmul_rn(__dsub_rn((double)p.j_d0, __dmul_rn(0.5, (double)G.n_d0)), G.delta);
    c.d0c = (float)c.d0c64;
    c.rho0 = c.rho64 == 0.0;
    return c;
}

// Arc length in float32 and a bound on its error (turning angle from atan2f,
// taken as <= 4 ulp, plus the propagated rounding of its arguments).
__device__ __forceinline__ void arc32(const ZCand &C, float x, float y, float &L, float &eL)
{
    const float s = fmaf(x, C.sn, -(y * C.cs));
    const float c = fmaf(x, C.cs, y * C.sn);
    const float R1 = fabsf(x) + fabsf(y);
    const float Es = 3.0f * kEps * R1;
    if (C.rho0) {
        L = c;
        eL = kSafe * Es;
        return;
    }
    const float a = C.rho * c;
    const float w = s + C.d0c;
    const float bb = fmaf(C.rho, w, 1.0f);
    const float th = atan2f(a, bb);
    L = th * C.invrho;
    const float ar = fabsf(C.rho);
    const float da = fmaf(ar, Es, 2.0f * kEps * fabsf(a));
    const float dbb = fmaf(ar, Es + kEps * (fabsf(w) + fabsf(C.d0c)), kEps * (fabsf(C.rho * w) + fabsf(bb)));
    const float den = fmaf(a, a, bb * bb);
    const float dth = 8.0f * kEps * fabsf(th) + __fdividef(fmaf(fabsf(bb), da, fabsf(a) * dbb), den);
    eL = kSafe * fmaf(fabsf(C.invrho), dth, 2.0f * kEps * fabsf(L));
    if (!(den > 1e-6f)) eL = 3.4e38f;   // hit at the circle's centre: exact path
}

// Arc length in float64, in the definition's operation order.
__device__ __forceinline__ double arc64(const ZCand &C, float xf, float yf)
{
    const double x = xf, y = yf;
    const double s = __dsub_rn(__dmul_rn(x, C.sn64), __dmul_rn(y, C.cs64));
    const double c = __dadd_rn(__dmul_rn(x, C.cs64), __dmul_rn(y, C.sn64));
    if (C.rho64 == 0.0) return c;
    const double th = atan2_basic64(__dmul_rn(C.rho64, c),
                                    __dadd_rn(1.0, __dmul_rn(C.rho64, __dadd_rn(s, C.d0c64))));
    return __ddiv_rn(th, C.rho64);
}

// z0 bin of one (hit, q) by float32: -1 outside the axis, -2 too close to an
// edge to be decided.
__device__ __forceinline__ int z_bin32(const DevGeom &G, float z, float L, float eL, int q)
{
    const float t = G.cstep_f * (float)(2 * q + 1 - G.n_cot);
    const float zz = z + G.z0_max_f;
    const float v = fmaf(-L, t, zz);
    const float u = v * G.inv_dz_f;
    const float err = fmaf(fmaf(fabsf(t), eL, kSafe * kEps * (2.0f * fabsf(L * t) + fabsf(zz) + fabsf(v))),
                           G.inv_dz_f, kSafe * kEps * fabsf(u));
    const float nz = (float)G.n_z0;
    if (u + err < 0.0f || u - err >= nz) return -1;
    const float f = floorf(u);
    const float fr = u - f;
    // u + 1 (u in (-1, 0)) is rounded: only f >= 0 is decided here
    return f >= 0.0f && fminf(fr, 1.0f - fr) > err ? (int)f : -2;
}

// The same by the float64 definition, from the hit's arc length L64.
__device__ __forceinline__ int z_bin64(const DevGeom &G, float z, double L64, int q)
{
    const double t64 = __dmul_rn((double)(2 * q + 1 - G.n_cot), G.cstep);
    const double z0 = __dsub_rn((double)z, __dmul_rn(L64, t64));
    const double v = __dadd_rn(z0, G.z0_max);
    // a product settles all but the quotients within 1e-9 of an integer
    const double w = v * G.inv_dz, f = floor(w);
    if (fabs(w) < 1e6 && w - f > 1e-9 && w - f < 1.0 - 1e-9)
        return f >= 0.0 && f < (double)G.n_z0 ? (int)f : -1;
    const double u64 = __ddiv_rn(v, G.dz);
    if (u64 >= 0.0 && u64 < (double)G.n_z0) return (int)floor(u64);
    return -1;
}

constexpr int kZWarps = 4, kZThreads = 32 * kZWarps;

// One warp's state: a candidate's hits and one round's bins (lane = column).
struct ZWarp {
    double L64[32];
    float z[32], L[32], eL[32];
    short bin[32][32];   // [hit][lane]
};

// (z0, cot theta) result of one candidate with 1..32 hits list[o .. o + nh),
// one warp.  Every lane returns the result.
__device__ __forceinline__ ht_zres z_small_cand(const DevGeom &G, const float *__restrict__ x,
                                                const float *__restrict__ y,
                                                const float *__restrict__ z, const ht_peak &pk,
                                                const int *__restrict__ list, int o, int nh,
                                                int lane, ZWarp &W)
{
    const ZCand C = z_cand(G, pk);
    __syncwarp();   // the previous candidate's readers are done
    float xf = 0.0f, yf = 0.0f;
    if (lane < nh) {
        const int h = list[o + lane];
        xf = x[h];
        yf = y[h];
        W.z[lane] = z[h];
        arc32(C, xf, yf, W.L[lane], W.eL[lane]);
    }
    __syncwarp();
    bool have64 = false;   // uniform
    // the lane's best cell: key = count, then smallest index n n_cot + q
    int best_c = 0, best_idx = 0x7fffffff;
    for (int q0 = 0; q0 < G.n_cot; q0 += 32) {   // uniform
        const int q = q0 + lane;
        const bool col = q < G.n_cot;
        bool open = false;
        for (int h = 0; h < nh; ++h) {
            const int b = col ? z_bin32(G, W.z[h], W.L[h], W.eL[h], q) : -1;
            W.bin[h][lane] = (short)b;
            open |= b == -2;
        }
        if (__any_sync(0xffffffffu, open)) {
            // the float64 arc lengths, of all hits at once (lane = hit)
            if (!have64) {
                if (lane < nh) W.L64[lane] = arc64(C, xf, yf);
                have64 = true;
                __syncwarp();
            }
            if (open)
                for (int h = 0; h < nh; ++h)
                    if (W.bin[h][lane] == -2) W.bin[h][lane] = (short)z_bin64(G, W.z[h], W.L64[h], q);
            __syncwarp();
        }
        for (int h = 0; h < nh; ++h) {   // (each lane reads what it wrote)
            const int b = W.bin[h][lane];
            if (b < 0 || nh - h < best_c) continue;
            int c = 1;
            for (int g = h + 1; g < nh; ++g) c += W.bin[g][lane] == b;
            const int idx = b * G.n_cot + q;
            if (c > best_c || (c == best_c && idx < best_idx)) {
                best_c = c;
                best_idx = idx;
            }
        }
    }
    const int top = __reduce_max_sync(0xffffffffu, best_c);
    const int idx = __reduce_min_sync(0xffffffffu, best_c == top ? best_idx : 0x7fffffff);
    return top > 0 ? ht_zres{idx / G.n_cot, idx % G.n_cot, top} : ht_zres{-1, -1, 0};
}

// (z0, cot theta) result of one candidate with any number of hits, one CTA:
// n_z0 x n_cot uint32 histogram in shared memory and a block argmax.
// Thread 0 returns the result.  All threads must call.
__device__ __forceinline__ ht_zres z_big_cand(const DevGeom &G, const float *__restrict__ x,
                                              const float *__restrict__ y,
                                              const float *__restrict__ z, const ht_peak &pk,
                                              const int *__restrict__ list, int o, int nh)
{
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned *hist = reinterpret_cast<unsigned *>(smem);
    __shared__ float sL[kBigThreads], seL[kBigThreads], sx[kBigThreads], sy[kBigThreads],
        sz[kBigThreads];
    __shared__ unsigned long long red[kBigThreads / 32];
    const int NC = G.n_cot, NZ = G.n_z0, ncell = NZ * NC;
    const ZCand C = z_cand(G, pk);
    for (int t = threadIdx.x; t < ncell; t += kBigThreads) hist[t] = 0u;
    for (int c0 = 0; c0 < nh; c0 += kBigThreads) {
        __syncthreads();
        const int hc = min(kBigThreads, nh - c0);
        if (threadIdx.x < hc) {
            const int h = list[o + c0 + threadIdx.x];
            sx[threadIdx.x] = x[h];
            sy[threadIdx.x] = y[h];
            sz[threadIdx.x] = z[h];
            arc32(C, sx[threadIdx.x], sy[threadIdx.x], sL[threadIdx.x], seL[threadIdx.x]);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < hc * NC; t += kBigThreads) {
            const int hl = t / NC, q = t - hl * NC;
            int nbin = z_bin32(G, sz[hl], sL[hl], seL[hl], q);
            if (nbin == -2) nbin = z_bin64(G, sz[hl], arc64(C, sx[hl], sy[hl]), q);
            if (nbin >= 0) atomicAdd(&hist[nbin * NC + q], 1u);
        }
    }
    __syncthreads();
    // argmax: key = count << 32 | ~index (largest count, then smallest index)
    unsigned long long bk = 0ull;
    for (int t = threadIdx.x; t < ncell; t += kBigThreads) {
        const unsigned c = hist[t];
        const unsigned long long k = ((unsigned long long)c << 32) | (0xffffffffull - (unsigned)t);
        if (c && k > bk) bk = k;
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) bk = max(bk, __shfl_xor_sync(0xffffffffu, bk, s));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = bk;
    __syncthreads();
    ht_zres r{-1, -1, 0};
    if (threadIdx.x == 0) {
        unsigned long long b = 0ull;
        for (int w = 0; w < kBigThreads / 32; ++w) b = max(b, red[w]);
        if (b) {
            const int idx = (int)(0xffffffffu - (unsigned)(b & 0xffffffffull));
            r = ht_zres{idx / NC, idx % NC, (int)(b >> 32)};
        }
    }
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------- launches
// Candidates of event slot e: ids e * cap + m, m < min(counts[e], cap); hits
// carry batch-wide indices, off[0 .. n_ev] are the events' hit offsets (null:
// one event of n hits).  tot[0]: grouped hits, tot[1]: candidates of up to
// 32 hits (listed from the front of todo), tot[2]: larger ones (from its back).
__device__ __forceinline__ int event_of(const int *__restrict__ off, int n_ev, int h)
{
    int lo = 0, hi = n_ev;          // off[lo] <= h < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= h) lo = mid; else hi = mid;
    }
    return lo;
}

struct ZGroup {
    const int *off, *d_nev, *counts;   // off, d_nev null: one event
    int n, cap;

    __device__ __forceinline__ int hits(int &n_ev) const
    {
        n_ev = d_nev ? *d_nev : 1;
        return off ? off[n_ev] : n;
    }
    // global id of hit h's candidate, -1 for none
    __device__ __forceinline__ long long cand(const int *__restrict__ assign, int h, int n_ev) const
    {
        const int a = assign[h];
        if (a < 0) return -1;
        const int e = off ? event_of(off, n_ev, h) : 0;
        return a < min(counts[e], cap) ? (long long)e * cap + a : -1;
    }
};

// cnt = 0 for every kept candidate; grid.y = event slot.
__global__ void k_z_zero(ZGroup Z, int *__restrict__ cnt, int *__restrict__ tot)
{
    const int e = blockIdx.y;
    if (e >= (Z.d_nev ? *Z.d_nev : 1)) return;
    if (e == 0 && blockIdx.x == 0 && threadIdx.x < 3) tot[threadIdx.x] = 0;
    const int nc = min(Z.counts[e], Z.cap);
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < nc; m += gridDim.x * blockDim.x)
        cnt[(size_t)e * Z.cap + m] = 0;
}

__global__ void k_z_count(ZGroup Z, const int *__restrict__ assign, int *__restrict__ cnt)
{
    int n_ev;
    const int n = Z.hits(n_ev);
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < n; h += gridDim.x * blockDim.x) {
        const long long g = Z.cand(assign, h, n_ev);
        if (g >= 0) atomicAdd(&cnt[g], 1);
    }
}

// A candidate with hits takes its range of the grouped list and its place in
// todo (one atomic per warp and counter); one without gets its result.
__global__ void __launch_bounds__(256)
k_z_alloc(ZGroup Z, const int *__restrict__ cnt, int *__restrict__ start, int *__restrict__ cur,
          int *__restrict__ todo, int ns, int *__restrict__ tot, ht_zres *__restrict__ out)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int e = blockIdx.y, lane = threadIdx.x & 31;
    if (e >= (Z.d_nev ? *Z.d_nev : 1)) return;
    const int nc = min(Z.counts[e], Z.cap);
    const unsigned lt = (1u << lane) - 1u;
    for (int m0 = blockIdx.x * blockDim.x + threadIdx.x - lane; m0 < nc;
         m0 += gridDim.x * blockDim.x) {   // uniform over the warp
        const int m = m0 + lane;
        const size_t g = (size_t)e * Z.cap + m;
        const int nh = m < nc ? cnt[g] : 0;
        const unsigned any = __ballot_sync(kAll, nh > 0);
        if (m < nc && nh == 0) out[g] = ht_zres{-1, -1, 0};
        if (!any) continue;
        int incl = nh;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kAll, incl, o);
            if (lane >= o) incl += v;
        }
        const unsigned ms = __ballot_sync(kAll, nh > 0 && nh <= 32);
        const unsigned mb = __ballot_sync(kAll, nh > 32);
        int at = 0;
        if (lane == 31) at = atomicAdd(&tot[0], incl);
        if (lane == 0 && ms) at = atomicAdd(&tot[1], __popc(ms));
        if (lane == 1 && mb) at = atomicAdd(&tot[2], __popc(mb));
        const int base = __shfl_sync(kAll, at, 31), as = __shfl_sync(kAll, at, 0),
                  ab = __shfl_sync(kAll, at, 1);
        if (nh == 0) continue;
        start[g] = cur[g] = base + incl - nh;
        if (nh <= 32) todo[as + __popc(ms & lt)] = (int)g;
        else todo[ns - 1 - (ab + __popc(mb & lt))] = (int)g;
    }
}

__global__ void k_z_scatter(ZGroup Z, const int *__restrict__ assign, int *__restrict__ cur,
                            int *__restrict__ list)
{
    int n_ev;
    const int n = Z.hits(n_ev);
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < n; h += gridDim.x * blockDim.x) {
        const long long g = Z.cand(assign, h, n_ev);
        if (g >= 0) list[atomicAdd(&cur[g], 1)] = h;
    }
}

__global__ void __launch_bounds__(kZThreads)
k_z_small(DevGeom G, const float *__restrict__ x, const float *__restrict__ y,
          const float *__restrict__ z, const ht_peak *__restrict__ peaks,
          const int *__restrict__ cnt, const int *__restrict__ start,
          const int *__restrict__ list, const int *__restrict__ todo,
          const int *__restrict__ tot, ht_zres *__restrict__ out)
{
    __shared__ ZWarp s_w[kZWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = tot[1];
    for (int t = blockIdx.x * kZWarps + warp; t < n; t += gridDim.x * kZWarps) {
        const int g = todo[t];
        const ht_zres r = z_small_cand(G, x, y, z, peaks[g], list, start[g], cnt[g], lane, s_w[warp]);
        if (lane == 0) out[g] = r;
    }
}

__global__ void __launch_bounds__(kBigThreads)
k_z_big(DevGeom G, const float *__restrict__ x, const float *__restrict__ y,
        const float *__restrict__ z, const ht_peak *__restrict__ peaks,
        const int *__restrict__ cnt, const int *__restrict__ start,
        const int *__restrict__ list, const int *__restrict__ todo, int ns,
        const int *__restrict__ tot, ht_zres *__restrict__ out)
{
    const int n = tot[2];
    for (int t = blockIdx.x; t < n; t += gridDim.x) {
        const int g = todo[ns - 1 - t];
        const ht_zres r = z_big_cand(G, x, y, z, peaks[g], list, start[g], cnt[g]);
        if (threadIdx.x == 0) out[g] = r;
    }
}

size_t z_bytes(size_t ng, int n)
{
    return 4 * align256((ng + 1) * 4) + 256 + align256((size_t)(n > 0 ? n : 1) * 4);
}

cudaError_t run_z(const DevGeom &G, const ZGroup &Z, int n_ev, int max_hits, const float *x,
                  const float *y, const float *z, const int *assign, const ht_peak *peaks,
                  ht_zres *out, void *ws, cudaStream_t st)
{
    const size_t ng = (size_t)n_ev * Z.cap;
    char *p = reinterpret_cast<char *>(ws);
    int *cnt = reinterpret_cast<int *>(p); p += align256((ng + 1) * 4);
    int *start = reinterpret_cast<int *>(p); p += align256((ng + 1) * 4);
    int *cur = reinterpret_cast<int *>(p); p += align256((ng + 1) * 4);
    int *todo = reinterpret_cast<int *>(p); p += align256((ng + 1) * 4);
    int *tot = reinterpret_cast<int *>(p); p += 256;
    int *list = reinterpret_cast<int *>(p);
    const int sms = device_sms();
    const int nb = max(1, min(sms * 8, (max_hits + 255) / 256));
    const dim3 gc(max(1, min((Z.cap + 255) / 256, sms * 8 / n_ev + 1)), n_ev);
    k_z_zero<<<gc, 256, 0, st>>>(Z, cnt, tot);
    k_z_count<<<nb, 256, 0, st>>>(Z, assign, cnt);
    k_z_alloc<<<gc, 256, 0, st>>>(Z, cnt, start, cur, todo, (int)ng, tot, out);
    k_z_scatter<<<nb, 256, 0, st>>>(Z, assign, cur, list);
    k_z_small<<<sms * 8, kZThreads, 0, st>>>(G, x, y, z, peaks, cnt, start, list, todo, tot, out);
    k_z_big<<<sms * 2, kBigThreads, z_big_smem(G), st>>>(G, x, y, z, peaks, cnt, start, list, todo,
                                                         (int)ng, tot, out);
    return cudaGetLastError();
}

}  // namespace

size_t vote_z_workspace_bytes(const DevGeom &, int n, int cap)
{
    return z_bytes((size_t)(cap > 0 ? cap : 0), n);
}

cudaError_t prepare_z_kernels(int max_smem)
{
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, (const void *)k_z_big);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute((const void *)k_z_big, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                max_smem - (int)fa.sharedSizeBytes);
}

// Batch z vote: candidates of all n_ev event slots at once.
size_t vote_z_batch_workspace_bytes(int n_ev, int cap, int max_hits)
{
    return z_bytes((size_t)n_ev * cap, max_hits);
}

cudaError_t launch_vote_z_batch(const DevGeom &G, const float *x, const float *y, const float *z,
                                const int *assign, const int *off, const int *d_nev,
                                const ht_peak *peaks, const int *counts, int cap, int n_ev,
                                ht_zres *out, void *ws, int max_hits, cudaStream_t st)
{
    return run_z(G, ZGroup{off, d_nev, counts, 0, cap}, n_ev, max_hits, x, y, z, assign, peaks, out,
                 ws, st);
}

cudaError_t launch_vote_z(const DevGeom &G, const float *x, const float *y, const float *z,
                          int n, const int *assign, const ht_peak *peaks, const int *d_count,
                          int cap, ht_zres *out, void *ws, cudaStream_t st)
{
    if (cap == 0) return cudaSuccess;
    return run_z(G, ZGroup{nullptr, nullptr, d_count, n, cap}, 1, n, x, y, z, assign, peaks, out,
                 ws, st);
}

}  // namespace ht
