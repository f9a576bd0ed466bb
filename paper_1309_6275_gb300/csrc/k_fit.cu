// k_fit.cu -- refinement of the candidates (ht_fit_tracks in include/ht.h):
// a least-squares circle fit of each candidate to its assigned hits.
// Section 5 has costlier computations confirm the candidates and Section 6
// names a Kalman filter for it (run on the CPU there, with a GPU version
// suggested); without material or process noise a Kalman filter over
// the hits computes the weighted least-squares estimate, fitted here
// directly.
//
// Reading: p = (rho, d0, phi0) starts at the candidate's cell centre; the
// residual of hit (x, y) is F / 2 with F = rho d0^2 + 2 (1 + rho s) d0 +
// rho r^2 + 2 s (the signed distance to the circle to first order); `iters`
// Gauss-Newton steps solve (J^T J) dp = -J^T r by Cholesky (a non-positive
// pivot stops with status -1); chi2 and sigma^2 (J^T J)^-1 at the final p.
// Optional hit selection: only hits within `road` of the cell-centre circle
// are fitted; then the hits within `cut` sigma of the fitted circle are
// fitted again with `iters2` steps (the outlier rejection of a track fit).
//
// Design (GB300): candidates' hit lists by counting sort (count, scan,
// scatter), then a pass that settles the candidates with too few hits and
// lists the others.  The float64 pipe bounds the fit: a warp's float64
// instruction takes about 16 cycles of an SM however few of its lanes work, so
// a warp per candidate (ten hits on 32 lanes, and every lane repeating the
// sine, the Cholesky factor and the substitutions) spends most of it on idle
// or repeated lanes.  A candidate of up to kFitSmall hits is fitted by one
// thread, its hits in turn, its hit selection kept as a bit mask, the sine
// and cosine computed once per parameter vector; by eight lanes where the
// candidates would not fill the GPU one to a thread (64 threads per SM: two
// warps keep its float64 pipe busy), by sixteen where not even sixteen each do.
// Larger candidates take a warp each.
// GB300, 21,855 candidates of 7 to 10 hits, road, cut and eight steps: 3.67 ->
// 0.265 ms.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "ht_internal.cuh"

namespace ht {
namespace {

__device__ __forceinline__ int event_of(const int *off, int n_ev, int h)
{
    int lo = 0, hi = n_ev;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= h) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Count (list null) or scatter the hits of every candidate: candidate m of
// event e is slot e * cap + m.
__global__ void k_fit_lists(const int *__restrict__ off, int n_ev,
                            const int *__restrict__ assign, const int *__restrict__ counts,
                            int cap, int *__restrict__ cnt, int *__restrict__ cur,
                            int *__restrict__ list)
{
    const int total = off[n_ev];
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < total; h += gridDim.x * blockDim.x) {
        const int m = assign[h];
        if (m < 0) continue;
        const int e = event_of(off, n_ev, h);
        if (m >= min(counts[e], cap)) continue;
        const size_t slot = (size_t)e * cap + m;
        if (list) list[atomicAdd(&cur[slot], 1)] = h;
        else atomicAdd(&cnt[slot], 1);
    }
}

__device__ __forceinline__ double half_f(double rho, double d0, double s, double r2)
{
    return 0.5 * (rho * d0 * d0 + 2.0 * (1.0 + rho * s) * d0 + rho * r2 + 2.0 * s);
}

// Cholesky of the symmetric 3 x 3 matrix {A0 A1 A2; . A3 A4; . . A5}:
// L = {l0; l1 l2; l3 l4 l5}; false if a pivot is not positive.
__device__ __forceinline__ bool chol3(const double A[6], double L[6])
{
    if (!(A[0] > 0.0)) return false;
    L[0] = sqrt(A[0]);
    L[1] = A[1] / L[0];
    const double d1 = A[3] - L[1] * L[1];
    if (!(d1 > 0.0)) return false;
    L[2] = sqrt(d1);
    L[3] = A[2] / L[0];
    L[4] = (A[4] - L[3] * L[1]) / L[2];
    const double d2 = A[5] - L[3] * L[3] - L[4] * L[4];
    if (!(d2 > 0.0)) return false;
    L[5] = sqrt(d2);
    return true;
}

struct FitArgs {
    double delta, half_nd, pi_over_np, sigma, road, cut;
    const double *rho64;
    int n_phi0, min_hits, iters, iters2;
};

constexpr int kFitSmall = 32;       // hits of a candidate fitted by one thread or some lanes
constexpr int kFitThreads = 64;     // small blocks spread few candidates over the SMs

// One candidate's hits as W consecutive lanes of a warp see them: lane sub
// takes hits sub, sub + W, ... of list[b .. b + nh).  keep: bit i selects the
// lane's i-th hit (up to kFitSmall per lane); with more hits than that the
// selection is evaluated at each use (q, w).
template <int W>
struct Fitter {
    const float *x, *y;
    const int *list;
    int nh, sub;
    double p[3], sn, cs;   // parameters, sine and cosine of phi0
    double q[5], w;        // selection: residual at q (with its sine, cosine) at most w
    unsigned keep;

    __device__ __forceinline__ double sum(double v) const
    {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, W);
        return v;
    }

    __device__ __forceinline__ int sum(int v) const
    {
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, W);
        return v;
    }

    __device__ __forceinline__ bool selected(double xh, double yh) const
    {
        if (!(w < 1e300)) return true;
        return fabs(half_f(q[0], q[1], xh * q[3] - yh * q[4], xh * xh + yh * yh)) <= w;
    }

    __device__ __forceinline__ void set_p()
    {
        sincos(p[2], &sn, &cs);
    }

    // Selects the hits within width of the circle p; returns their number.
    __device__ __forceinline__ int select(double width)
    {
        q[0] = p[0]; q[1] = p[1]; q[2] = p[2]; q[3] = sn; q[4] = cs;
        w = width;
        keep = 0u;
        int k = 0;
        for (int t = sub, i = 0; t < nh; t += W, ++i) {
            const int h = list[t];
            if (!selected((double)x[h], (double)y[h])) continue;
            ++k;
            if (i < 32) keep |= 1u << i;
        }
        return sum(k);
    }

    // Normal equations of the selected hits at p: A (6 unique entries), J^T r
    // and sum r^2; every lane gets them.
    __device__ __forceinline__ void normal_eq(double A[6], double g[3], double &rr) const
    {
        double a[6] = {0, 0, 0, 0, 0, 0}, gg[3] = {0, 0, 0}, s2 = 0;
        const double rho = p[0], d0 = p[1];
        for (int t = sub, i = 0; t < nh; t += W, ++i) {
            if (i < 32 && !((keep >> i) & 1u)) continue;
            const int h = list[t];
            const double xh = (double)x[h], yh = (double)y[h];
            if (i >= 32 && !selected(xh, yh)) continue;
            const double s = xh * sn - yh * cs, c = xh * cs + yh * sn;
            const double r2 = xh * xh + yh * yh;
            const double r = half_f(rho, d0, s, r2);
            const double j0 = 0.5 * (d0 * d0 + 2.0 * s * d0 + r2);
            const double j1 = rho * d0 + 1.0 + rho * s;
            const double j2 = (1.0 + rho * d0) * c;
            a[0] += j0 * j0; a[1] += j0 * j1; a[2] += j0 * j2;
            a[3] += j1 * j1; a[4] += j1 * j2; a[5] += j2 * j2;
            gg[0] += j0 * r; gg[1] += j1 * r; gg[2] += j2 * r;
            s2 += r * r;
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) A[i] = sum(a[i]);
#pragma unroll
        for (int i = 0; i < 3; ++i) g[i] = sum(gg[i]);
        rr = sum(s2);
    }

    // Gauss-Newton steps on the selected hits; false (and p kept) when the
    // normal matrix is not positive definite.  All W lanes hold the same sums,
    // so they leave together; lanes of other candidates may go on (active:
    // this one still steps).
    __device__ __forceinline__ bool steps(int iters, bool active)
    {
        for (int it = 0; it < iters && __any_sync(0xffffffffu, active); ++it) {
            double A[6], g[3], rr, L[6];
            normal_eq(A, g, rr);
            if (active && !chol3(A, L)) active = false;
            if (active) {
                // forward then backward substitution: L z = g, L^T dp = z
                const double z0 = g[0] / L[0];
                const double z1 = (g[1] - L[1] * z0) / L[2];
                const double z2 = (g[2] - L[3] * z0 - L[4] * z1) / L[5];
                const double d2 = z2 / L[5];
                const double d1 = (z1 - L[4] * d2) / L[2];
                const double d0 = (z0 - L[1] * d1 - L[3] * d2) / L[0];
                p[0] -= d0;
                p[1] -= d1;
                p[2] -= d2;
                set_p();
            }
        }
        return active;
    }

    // The whole fit of the candidate at peak pk (nh >= min_hits hits; nh = 0
    // for lanes without a candidate, whose result is not used).
    __device__ __forceinline__ ht_track fit(const FitArgs &F, const ht_peak pk)
    {
        ht_track T;
        T.reserved = 0;
        p[0] = F.rho64[pk.i_rho];
        p[1] = ((double)pk.j_d0 - F.half_nd) * F.delta;
        p[2] = (double)(2 * pk.k_phi0 + 1 - F.n_phi0) * F.pi_over_np;
        set_p();
        // the road: hits near the cell-centre circle
        int nk = select(F.road > 0.0 ? F.road : 1e308);
        bool few = nk < F.min_hits;
        bool ok = steps(F.iters, !few);
        if (F.cut > 0.0) {
            // the outlier cut: hits near the fitted circle, fitted again
            const bool again = ok;
            const unsigned keep0 = keep;
            const double q0[5] = {q[0], q[1], q[2], q[3], q[4]}, w0 = w;
            const int nk2 = select(F.cut * F.sigma);
            if (again) {
                nk = nk2;
                few = nk < F.min_hits;
            } else {   // the road's selection stays
                keep = keep0;
                w = w0;
#pragma unroll
                for (int i = 0; i < 5; ++i) q[i] = q0[i];
            }
            ok = steps(F.iters2, again && !few);
        }
        T.rho = p[0]; T.d0 = p[1]; T.phi0 = p[2];
        T.n_hits = nk;
        double A[6], g[3], rr, L[6];
        normal_eq(A, g, rr);
        T.sig_rho = T.sig_d0 = T.sig_phi0 = nan("");
        if (few) {
            T.chi2 = nanf("");
            T.status = 0;
            return T;
        }
        T.chi2 = (float)(rr / (F.sigma * F.sigma));
        T.status = ok ? 1 : -1;
        if (chol3(A, L)) {
            // diagonal of (L L^T)^-1 = columns of L^-1 squared and summed
            const double i0 = 1.0 / L[0], i2 = 1.0 / L[2], i5 = 1.0 / L[5];
            const double i1 = -L[1] * i0 * i2;                       // (L^-1)[1][0]
            const double i4 = -L[4] * i2 * i5;                       // (L^-1)[2][1]
            const double i3 = -(L[3] * i0 + L[4] * i1) * i5;         // (L^-1)[2][0]
            const double s2 = F.sigma * F.sigma;
            T.sig_rho = sqrt(s2 * (i0 * i0 + i1 * i1 + i3 * i3));
            T.sig_d0 = sqrt(s2 * (i2 * i2 + i4 * i4));
            T.sig_phi0 = sqrt(s2 * (i5 * i5));
        } else {
            T.status = -1;
        }
        return T;
    }
};

// Settles the candidates with too few hits and lists the others' slots: those
// of up to kFitSmall hits from the front of todo (n[0] of them), larger ones
// from its back (n[1]).  grid.y = event.
__global__ void __launch_bounds__(256)
k_fit_split(FitArgs F, const ht_peak *__restrict__ peaks, const int *__restrict__ counts, int cap,
            const int *__restrict__ start, int ns, ht_track *__restrict__ out,
            int *__restrict__ todo, int *__restrict__ n)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int e = blockIdx.y, nc = min(counts[e], cap), lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (int m0 = blockIdx.x * blockDim.x + threadIdx.x - lane; m0 < nc;
         m0 += gridDim.x * blockDim.x) {   // uniform over the warp
        const int m = m0 + lane;
        const size_t slot = (size_t)e * cap + m;
        const int nh = m < nc ? start[slot + 1] - start[slot] : -1;
        const bool fit = nh >= F.min_hits;   // min_hits >= 3
        const unsigned ms = __ballot_sync(kAll, fit && nh <= kFitSmall);
        const unsigned mb = __ballot_sync(kAll, fit && nh > kFitSmall);
        int at = 0;   // one counter per warp and list
        if (lane == 0 && ms) at = atomicAdd(&n[0], __popc(ms));
        if (lane == 1 && mb) at = atomicAdd(&n[1], __popc(mb));
        const int as = __shfl_sync(kAll, at, 0), ab = __shfl_sync(kAll, at, 1);
        if (fit) {
            if (nh <= kFitSmall) todo[as + __popc(ms & lt)] = (int)slot;
            else todo[ns - 1 - (ab + __popc(mb & lt))] = (int)slot;
        }
        if (fit || m >= nc) continue;
        const ht_peak pk = peaks[slot];
        ht_track T;
        T.rho = F.rho64[pk.i_rho];
        T.d0 = ((double)pk.j_d0 - F.half_nd) * F.delta;
        T.phi0 = (double)(2 * pk.k_phi0 + 1 - F.n_phi0) * F.pi_over_np;
        T.sig_rho = T.sig_d0 = T.sig_phi0 = nan("");
        T.chi2 = nanf("");
        T.n_hits = nh;
        T.status = 0;
        T.reserved = 0;
        out[slot] = T;
    }
}

// W lanes per candidate over the list todo[0 .. n) (step 1) or backwards
// from todo (step -1).
template <int W>
__device__ __forceinline__ void fit_list(const FitArgs &F, const float *__restrict__ x,
                                         const float *__restrict__ y,
                                         const ht_peak *__restrict__ peaks,
                                         const int *__restrict__ start,
                                         const int *__restrict__ list, const int *todo, int step,
                                         int n, ht_track *__restrict__ out)
{
    const int per = (gridDim.x * kFitThreads) / W;
    const int g0 = (blockIdx.x * kFitThreads + threadIdx.x) / W;
    const int wfirst = (blockIdx.x * kFitThreads + (threadIdx.x & ~31)) / W;   // the warp's first
    for (int at = 0; wfirst + at < n; at += per) {   // uniform over the warp
        const int i = g0 + at;
        const bool act = i < n;
        const size_t slot = (size_t)todo[step * (act ? i : wfirst + at)];
        const int b = start[slot];
        Fitter<W> f;
        f.x = x;
        f.y = y;
        f.list = list + b;
        f.nh = act ? start[slot + 1] - b : 0;
        f.sub = threadIdx.x % W;
        const ht_track T = f.fit(F, peaks[slot]);
        if (act && f.sub == 0) out[slot] = T;
    }
}

__global__ void __launch_bounds__(kFitThreads)
k_fit_tracks(FitArgs F, const float *__restrict__ x, const float *__restrict__ y,
             const ht_peak *__restrict__ peaks, const int *__restrict__ start,
             const int *__restrict__ list, const int *__restrict__ todo, int ns,
             const int *__restrict__ n, int dense, ht_track *__restrict__ out)
{
    const int small = n[0], big = n[1];
    // a thread each where the candidates fill `dense` threads, else eight lanes,
    // or sixteen where those fill no more: with so few a candidate's own latency
    // counts (50 of 10, 20 and 32 hits 109, 120 and 132 -> 104, 114 and 115 us; a
    // warp each 107, 107 and 108, but 3 and 6 hits 113 and 107 against 109 and 104)
    if (small >= dense) fit_list<1>(F, x, y, peaks, start, list, todo, 1, small, out);
    else if (small > dense / 16) fit_list<8>(F, x, y, peaks, start, list, todo, 1, small, out);
    else fit_list<16>(F, x, y, peaks, start, list, todo, 1, small, out);
    fit_list<32>(F, x, y, peaks, start, list, todo + ns - 1, -1, big, out);
}

}  // namespace
}  // namespace ht

extern "C" {

size_t ht_fit_workspace_size(int32_t n_events, int32_t cap, int32_t n_hits)
{
    const size_t ns = (size_t)(n_events > 0 ? n_events : 1) * (size_t)(cap > 0 ? cap : 1);
    return 3 * ht::align256((ns + 1) * 4) + ht::align256((size_t)(n_hits > 0 ? n_hits : 1) * 4) +
           ht::scan_tmp_bytes((int)ns);
}

ht_status ht_fit_tracks(const ht_geometry *g, const float *x, const float *y, const int32_t *d_off,
                        int32_t n_events, int32_t n_hits, const int32_t *assign,
                        const ht_peak *peaks, const int32_t *d_count, int32_t cap,
                        int32_t min_hits, int32_t iters, double sigma, double road, double cut,
                        int32_t iters2, ht_track *out, void *workspace, size_t workspace_bytes,
                        ht_stream stream)
{
    if (!g || !d_off || !d_count || !out || !workspace || n_events < 1 || n_hits < 0 || cap < 1 ||
        min_hits < 3 || iters < 0 || iters > 64 || iters2 < 0 || iters2 > 64 ||
        !(sigma > 0.0) || road != road || cut != cut ||
        (n_hits > 0 && (!x || !y || !assign)) || !peaks)
        return ht::set_error(HT_ERR_ARG, "ht_fit_tracks: bad argument");
    if ((int64_t)n_events * cap > 0x7fffffffLL)
        return ht::set_error(HT_ERR_CAPACITY, "ht_fit_tracks: n_events * cap above 2^31");
    if (workspace_bytes < ht_fit_workspace_size(n_events, cap, n_hits) ||
        reinterpret_cast<uintptr_t>(workspace) % 256 != 0)
        return ht::set_error(HT_ERR_ARG, "ht_fit_tracks: workspace size or alignment");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int ns = n_events * cap;
    char *w = reinterpret_cast<char *>(workspace);
    int *cnt = reinterpret_cast<int *>(w);
    int *start = reinterpret_cast<int *>(w + ht::align256(((size_t)ns + 1) * 4));
    int *cur = reinterpret_cast<int *>(w + 2 * ht::align256(((size_t)ns + 1) * 4));
    int *list = reinterpret_cast<int *>(w + 3 * ht::align256(((size_t)ns + 1) * 4));
    void *tmp = w + 3 * ht::align256(((size_t)ns + 1) * 4) +
                ht::align256((size_t)(n_hits > 0 ? n_hits : 1) * 4);
    cudaError_t e = cudaMemsetAsync(cnt, 0, (size_t)ns * 4, st);
    const int gb = n_hits > 0 ? min((n_hits + 255) / 256, 4096) : 1;
    if (e == cudaSuccess) {
        ht::k_fit_lists<<<gb, 256, 0, st>>>(d_off, n_events, assign, d_count, cap, cnt, nullptr,
                                            nullptr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = ht::scan_exclusive(cnt, start, cur, ns, nullptr, nullptr, tmp, st);
    if (e == cudaSuccess) {
        ht::k_fit_lists<<<gb, 256, 0, st>>>(d_off, n_events, assign, d_count, cap, nullptr, cur,
                                            list);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        ht::FitArgs F;
        F.delta = g->G.delta;
        F.half_nd = 0.5 * (double)g->G.n_d0;
        F.pi_over_np = ht::kPi / (double)g->G.n_phi0;
        F.sigma = sigma;
        F.road = road;
        F.cut = cut;
        F.iters2 = iters2;
        F.rho64 = g->G.rho64;
        F.n_phi0 = g->G.n_phi0;
        F.min_hits = min_hits;
        F.iters = iters;
        // the cursors are spent: they hold the list of candidates to fit; the
        // scan's scratch holds its two counts
        int *n = reinterpret_cast<int *>(tmp);
        e = cudaMemsetAsync(n, 0, 8, st);
        if (e == cudaSuccess) {
            const int sms = ht::device_sms();
            const int gx = max(1, min((cap + 255) / 256, sms * 8 / min(n_events, sms) + 1));
            ht::k_fit_split<<<dim3(gx, n_events), 256, 0, st>>>(F, peaks, d_count, cap, start, ns,
                                                                out, cur, n);
            ht::k_fit_tracks<<<sms * 8, ht::kFitThreads, 0, st>>>(F, x, y, peaks, start, list, cur,
                                                                  ns, n, sms * 64, out);
            e = cudaGetLastError();
        }
    }
    return e == cudaSuccess ? HT_OK : ht::set_error(HT_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"
