// k_confirm.cu -- confirmation of Hough candidates and the final hit
// assignment (ht_confirm, and the confirmation stage of ht_batch_run_tracks).
//
// Section 5 of arXiv:1309.6275: local maxima of the vote space are
// candidates, which costlier computations then confirm; Fig. 5 refines the
// candidates by a fit.  Reading, for candidate m = (i, j, k) and every hit h
// of its event, with b the bins of h's roots in column (rho_i, phi0_k)
// exactly as the vote casts them:
//   own(h)   some b == j,   pool(h)   some |b - j| <= pool;
//   seed layers: the layers with exactly one own hit (at least three); the
//   first, the last, and the one between them nearest their middle index;
//   seed circle: through those three own hits;
//   inliers: per layer, the pool hit closest to the circle (smaller hit
//   index on a tie) if its distance is below tol;
//   confirmed iff the inlier layers number at least min_layers.
// Then each hit goes to the confirmed candidate that lists it with the most
// inlier layers, ties to the smallest candidate index.
//
// A warp per candidate, persistent over the batch's candidates, on the hit
// index by layer and azimuth (k_hitindex.cu).  Nearly every candidate fails,
// so the work goes in the order that lets it fail early:
//  1. the own hits: only the azimuth cells whose hits can have a root in the
//     candidate's one bin (about a quarter of its pool's); own(h) from the
//     signs of the circle equation at the bin's two edges;
//  2. the seed circle's float32 frame, for up to 32 candidates at once, a
//     lane each (its float64 products would otherwise take the float64 pipe
//     a warp at a time);
//  3. the cells that circle crosses on every layer, and the float32 distance
//     of their hits with an error bound: hits on fewer than min_layers
//     layers end the candidate;
//  4. only then pool(h), per-layer contenders, and the float64 distance of
//     the definition where the bound cannot settle a layer.
// Every decision that float32 cannot prove is the vote's exact bin decision
// (double-float, then float64 in the definition's operation order) or the
// definition's float64 distance, so the results are bit-identical to the
// float64 plain definition.
//
// Bound by latency and issue (60% of slots; index loads and fixed latencies
// lead the stalls): 1350 warp instructions per candidate, where scanning and
// binning the whole pool (435 hits) with a frame per warp took 6800.  Stage on
// GB300: 25 events of 2k-60k hits (1.25 M candidates) 11.7 -> 2.1 ms, 25 of 10k
// hits (2.7 M) 16.7 -> 4.2, two of 50k (512 x 256 x 1024) 8.7 -> 1.5.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tiles.cuh"

namespace ht {


namespace {

// Per-candidate constants of its column (rho_i, phi0_k) for column_bins.
struct ColumnCtx {
    int i, k;
    float sk, ck, rho, invrho, invrho_es, rt;
    bool has_b;

    __device__ __forceinline__ void init(const DevGeom &G, int i_, int k_)
    {
        i = i_;
        k = k_;
        sk = G.sn32[k];
        ck = G.cs32[k];
        rho = G.rho32[i];
        invrho = G.invrho32[i];
        invrho_es = fabsf(invrho) * G.err_scale;
        rt = fabsf(rho) * 1.0001f;
        has_b = G.rho64[i] != 0.0;
    }
};

// The bins of hit (xf, yf) in the candidate's column, exactly as the vote
// casts them (guarded float32, then the vote's double-float and float64
// tiers for what float32 cannot prove); returns their number (0 to 2) and
// writes them to j[].
__device__ __forceinline__ int column_bins(const DevGeom &G, const ColumnCtx &C, float xf,
                                           float yf, int j[2])
{
    const float c = fmaf(xf, C.ck, yf * C.sk);
    const float R1 = fabsf(xf) + fabsf(yf);
    const float Ec = (kSafe * 3.0f * kEps) * R1;
    if (c < -Ec) return 0;   // c <= 0 proven: the hit is not on a first half turn here
    if (c <= Ec) return redo_bins(G, xf, yf, C.i, C.k, j);
    const float s = fmaf(xf, C.sk, -(yf * C.ck));
    const float r2 = fmaf(xf, xf, yf * yf);
    const Item it = make_item(G, s, c, r2, R1, C.rt);
    int jA, jB, r;
    if (C.has_b)
        r = eval32<true>(G, C.rho, C.invrho_es, C.invrho, it, jA, jB);
    else
        r = eval32<false>(G, C.rho, 0.0f, C.invrho, it, jA, jB);
    if (r == kRedo) return redo_bins(G, xf, yf, C.i, C.k, j);
    int nv = 0;
    if (jA >= 0) j[nv++] = jA;
    if (jB >= 0) j[nv++] = jB;
    return nv;
}

// circle3 and seed_frame are calls: inlined, their code and registers stand in
// the loop that nearly every candidate leaves before (stage of 25 events of 10k
// hits 4.65 ms, called 4.2).
//
// Circle through three points: centre = P1 + ((b_y |a|^2 - a_y |b|^2) / d,
// (a_x |b|^2 - b_x |a|^2) / d) with a = P2 - P1, b = P3 - P1,
// d = 2 (a_x b_y - a_y b_x); false when d == 0 (collinear).
static __device__ __noinline__ bool circle3(double x1, double y1, double x2, double y2, double x3,
                                        double y3, double &xc, double &yc, double &R)
{
    const double ax = __dsub_rn(x2, x1), ay = __dsub_rn(y2, y1);
    const double bx = __dsub_rn(x3, x1), by = __dsub_rn(y3, y1);
    const double d = __dmul_rn(2.0, __dsub_rn(__dmul_rn(ax, by), __dmul_rn(ay, bx)));
    if (d == 0.0) return false;
    const double a2 = __dadd_rn(__dmul_rn(ax, ax), __dmul_rn(ay, ay));
    const double b2 = __dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by));
    const double ux = __ddiv_rn(__dsub_rn(__dmul_rn(by, a2), __dmul_rn(ay, b2)), d);
    const double uy = __ddiv_rn(__dsub_rn(__dmul_rn(ax, b2), __dmul_rn(bx, a2)), d);
    xc = __dadd_rn(x1, ux);
    yc = __dadd_rn(y1, uy);
    R = __dsqrt_rn(__dadd_rn(__dmul_rn(ux, ux), __dmul_rn(uy, uy)));
    return true;
}

// |sqrt((x - xc)^2 + (y - yc)^2) - R|
__device__ __forceinline__ double circle_dist(float xf, float yf, double xc, double yc, double R)
{
    const double dx = __dsub_rn((double)xf, xc), dy = __dsub_rn((double)yf, yc);
    return fabs(__dsub_rn(__dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy))), R));
}

// Float32 frame of the seed circle at its first point P1, for the distance
// estimate t(w) = (k |w|^2 - 2 w.n) / (|k w - n| + 1), w = P - P1 (exact for
// a unit n towards the centre and k = 1 / R), and the coefficients of a
// bound e(w) = B2 |w|^2 + B1 (|w_x| + |w_y|) + B0 on |t(w)| minus the
// float64 distance of the definition (circle3, then circle_dist).  With
// a = P2 - P1, b = P3 - P1 (exact in float64), c = a_x b_y - a_y b_x and
// v = (b_y |a|^2 - a_y |b|^2, a_x |b|^2 - b_x |a|^2), the centre is
// P1 + v / (2 c) and |v| = |a| |b| |b - a|, so n = sign(c) v / |v| and
// k = 2 |c| / |v|: v and c take float64 products and sums only (no division
// or square root), the rest is float32.  The terms of the bound, u = 2^-24,
// r = (|a| + |b|) / |b - a|, S = |a| |b| / |c| (one over the sine of the
// angle at P1):
//  - turning n by an angle moves t by at most |w| times it (a rotation
//    about P1), a norm 1 + eta by at most 3 |eta| |w|: 13 u |w| for float32,
//    2^-53 (6 sqrt2 r + 1) |w| for the float64 error of v;
//  - |dt/dk| <= 2 |w|^2 (a circle through P1 is within |w| of P), times
//    k's relative error 5.5 u + 2^-53 (S + 8.5 r + 2);
//  - the float64 definition is within 2^-53 R (17 r + 2 S + 13) (+1e-12 cm)
//    of the exact circle through the three points (R = 1 / k);
//  - the float32 evaluation of t: 6e-7 (k |w|^2 + 2 (|w_x| + |w_y|)) + 1e-6
//    cm;
// each first-order and taken with a margin.  Returns false exactly when
// circle3 does (c == 0 in its operation order).  A degenerate frame (an
// underflow, r or S huge) gets B0 = +inf, which sends every distance to the
// float64 definition.
struct SeedFrame {
    float x1, y1, nx, ny, kap, B0, B1, B2;
};

static __device__ __noinline__ bool seed_frame(float x1, float y1, float x2, float y2, float x3,
                                           float y3, SeedFrame &F)
{
    const double ax = __dsub_rn((double)x2, (double)x1), ay = __dsub_rn((double)y2, (double)y1);
    const double bx = __dsub_rn((double)x3, (double)x1), by = __dsub_rn((double)y3, (double)y1);
    const double c = __dsub_rn(__dmul_rn(ax, by), __dmul_rn(ay, bx));
    if (c == 0.0) return false;
    const double a2 = __fma_rn(ax, ax, __dmul_rn(ay, ay));
    const double b2 = __fma_rn(bx, bx, __dmul_rn(by, by));
    const float vx = (float)__fma_rn(by, a2, -__dmul_rn(ay, b2));
    const float vy = (float)__fma_rn(ax, b2, -__dmul_rn(bx, a2));
    const float cf = fabsf((float)c);
    const float vn = sqrtf(fmaf(vx, vx, vy * vy));
    const float ex = (float)__dsub_rn((double)x3, (double)x2);
    const float ey = (float)__dsub_rn((double)y3, (double)y2);
    const float la = sqrtf((float)a2), lb = sqrtf((float)b2);
    const float r = 1.001f * (la + lb) / sqrtf(fmaf(ex, ex, ey * ey));
    const float S = 1.001f * (la * lb) / cf;
    F.x1 = x1;
    F.y1 = y1;
    if (!(vn > 0.0f && vn < 3.0e38f && cf > 0.0f && r < 1.0e6f && S < 1.0e9f)) {
        F.nx = 1.0f;
        F.ny = 0.0f;
        F.kap = 0.0f;
        F.B2 = F.B1 = 0.0f;
        F.B0 = __int_as_float(0x7f800000);
        return true;
    }
    const float sg = c > 0.0 ? 1.0f : -1.0f;
    F.nx = sg * (vx / vn);
    F.ny = sg * (vy / vn);
    F.kap = 2.0f * cf / vn;
    const float R = vn / (2.0f * cf);
    F.B2 = F.kap * (1.3e-6f + 2.5e-16f * S + 2.2e-15f * r + 5e-16f);
    F.B1 = 2.0e-6f + 1.2e-15f * r;
    F.B0 = 1.0e-6f + 1.0e-12f + 1.22e-16f * R * (17.0f * r + 2.0f * S + 13.0f);
    return true;
}

constexpr int kCfThreads = 128, kCfWarps = kCfThreads / 32;
// Hits near the circle held per pass (more: further passes).  128, 160 and 192,
// 10k hits, pool 4: tol 0.01 cm 277, 276 and 285 us, 1.5 cm 1043, 947 and 950.
constexpr int kCfCap = 160;
constexpr int kCfChunk = 32;       // candidates of a warp's chunk, at most

// A candidate's seeds and, once computed, its float32 seed frame with the
// circle's implicit form |P|^2 kap - 2 P.g + h = 0, g = kap P1 + n (towards
// the centre from the origin), h = kap |P1|^2 + 2 P1.n.
struct CfSeed {
    int pa, pb, pc, ev;     // index positions (pa < 0: none), event
    SeedFrame F;
    float psi, gn, h;       // azimuth and length of g
};

struct CfWarp {
    int own_pos[16];
    int best_h[16];
    double best_d[16];
    // per layer, over the pool hits of the pass: least lower and upper bound
    // of a distance (float bits), contenders (count, one of them) and the
    // pass's positions [qs, qe) (the pool is in layer order)
    unsigned lbmin[16], ubmin[16];
    int ncont[16], cq[16], qs[16], qe[16];
    int2 rr[32];            // non-empty runs scanned: start less the positions before it, layer
    int pool_p[kCfCap + 1], pool_h[kCfCap + 1];   // index position and event-local hit index
    float pool_lo[kCfCap + 1], pool_hi[kCfCap + 1];   // bounds on the hit's float64 distance
    unsigned char pool_l[kCfCap + 1];
    double xc, yc, R;       // the float64 seed circle, once computed
    CfSeed seed[kCfChunk];
};

// The warps' state of k_confirm (at namespace scope, so that the functions
// that take a warp's index address it as shared memory).
__shared__ CfWarp g_cfw[kCfWarps];

// The hits a candidate scans: runs of positions of the event's hit index
// (k_hitindex.cu), lane r's run being [start, start + len).  Position t of
// the sequence belongs to the run that covers it; at(base) gives every
// lane its position base + lane (p) and layer (l), or false past the end.
struct Runs {
    int excl, len, n;
    int wid;

    __device__ __forceinline__ void set(int start, int len_, int layer, int wid_, int lane)
    {
        constexpr unsigned kAll = 0xffffffffu;
        wid = wid_;
        len = len_;
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kAll, incl, o);
            if (lane >= o) incl += v;
        }
        excl = incl - len;
        n = __shfl_sync(kAll, incl, 31);
        const unsigned ne = __ballot_sync(kAll, len > 0);
        __syncwarp();   // the previous runs' readers are done
        if (len > 0)
            g_cfw[wid].rr[__popc(ne & ((1u << lane) - 1u))] = make_int2(start - excl, layer);
        __syncwarp();
    }

    // The place of index position p, which is in one of the runs (every lane).
    __device__ __forceinline__ int place(int p, int lane) const
    {
        constexpr unsigned kAll = 0xffffffffu;
        const unsigned ne = __ballot_sync(kAll, len > 0);
        const int t = len > 0 ? p - g_cfw[wid].rr[__popc(ne & ((1u << lane) - 1u))].x : -1;
        const unsigned m = __ballot_sync(kAll, len > 0 && t >= excl && t < excl + len);
        return __shfl_sync(kAll, t, __ffs(m) - 1);
    }

    __device__ __forceinline__ bool at(int base, int lane, int &p, int &l) const
    {
        constexpr unsigned kAll = 0xffffffffu;
        const int d = excl - base;
        const unsigned m = __reduce_or_sync(kAll, len > 0 && d > 0 && d < 32 ? 1u << d : 0u);
        const int c0 = __popc(__ballot_sync(kAll, len > 0 && d <= 0)) - 1;
        const bool ok = base + lane < n;
        if (ok) {
            const int2 r = g_cfw[wid].rr[c0 + __popc(m & (kAll >> (31 - lane)))];
            p = r.x + base + lane;
            l = r.y;
        }
        return ok;
    }
};

// Event of flattened candidate f: the last e with cpre[e] <= f (cpre is the
// exclusive prefix of the per-event kept-candidate counts, n_ev + 1 entries).
__device__ __forceinline__ int event_of(const int *cpre, int n_ev, int f)
{
    int lo = 0, hi = n_ev - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cpre[mid] <= f) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Azimuth window [w0, w1] (radians, near phik) of the hits of one layer that
// can have a root within d0 in [lo, hi] (cm) in column (rho, phi0_k); full:
// any hit of the layer, empty: none.  A root d0 of the circle equation gives
//   s = -(2 d0 + rho (d0^2 + r^2)) / (2 u),   u = 1 + rho d0,
// with ds/dd0 = -(u^2 + 1 - rho^2 r^2) / (2 u^2) and ds/d(r^2) = -rho / (2 u):
// for u > 0, s is monotone in r^2 (sign -rho), and in d0 (decreasing) while
// u^2 + 1 > rho^2 r^2; otherwise |ds/dd0| <= (1 + (1 + rho^2 r^2) / u^2) / 2
// bounds it around the middle of [lo, hi].  So over the window and the
// layer's radius range [rmin, rmax] s lies in an interval given by two
// corners (or the middle and that bound); with c > 0 the hit's azimuth is
// phi0_k - asin(s / r).  A layer beyond the circles' reach (the farthest
// point of a circle with perigee d0 is |d0 + 1/rho| + 1/|rho| from the
// origin) is empty.  Margins (1e-3 cm plus 1e-5 relative on s and on the
// reach, 2e-3 rad on the azimuth) cover float32 rounding; where u > 0 is not
// proven the whole layer is scanned.
__device__ __forceinline__ void layer_window(float rho, float phik, float lo, float hi,
                                             float rmin, float rmax, bool &full, bool &empty,
                                             float &w0, float &w1)
{
    full = false;
    empty = !(rmin <= rmax);
    w0 = w1 = 0.0f;
    if (empty) return;
    const float tl = fmaf(rho, lo, 1.0f), th = fmaf(rho, hi, 1.0f);
    const float tmin = fminf(tl, th);
    if (!(tmin >= 0.05f) || !(rmin >= 1e-3f)) {
        full = true;
        return;
    }
    const float ir = 1.0f / rho;   // +-inf for rho = 0: no reach limit
    const float reach = fmaxf(fabsf(lo + ir), fabsf(hi + ir)) + fabsf(ir);
    if (rmin > fmaf(reach, 1.0f + 1e-5f, 1e-3f)) {
        empty = true;
        return;
    }
    const float rA = rho > 0.0f ? rmin : rmax, rB = rho > 0.0f ? rmax : rmin;
    float s_hi, s_lo;
    if (fmaf(rho * rho * 1.001f, rmax * rmax, 1e-3f) < fmaf(tmin, tmin, 1.0f)) {
        s_hi = -fmaf(rho, fmaf(lo, lo, rA * rA), 2.0f * lo) / (2.0f * tl);
        s_lo = -fmaf(rho, fmaf(hi, hi, rB * rB), 2.0f * hi) / (2.0f * th);
    } else {
        const float mid = 0.5f * (lo + hi), tm = fmaf(rho, mid, 1.0f);
        const float L = 0.5f * (1.0f + fmaf(rho * rho, rmax * rmax, 1.0f) / (tmin * tmin));
        const float ds = 1.001f * L * 0.5f * (hi - lo);
        s_hi = -fmaf(rho, fmaf(mid, mid, rA * rA), 2.0f * mid) / (2.0f * tm) + ds;
        s_lo = -fmaf(rho, fmaf(mid, mid, rB * rB), 2.0f * mid) / (2.0f * tm) - ds;
    }
    const float ms = fmaf(1e-5f, fabsf(s_hi) + fabsf(s_lo), 1e-3f);
    s_hi += ms;
    s_lo -= ms;
    const float a_hi = s_hi / (s_hi > 0.0f ? rmin : rmax);
    const float a_lo = s_lo / (s_lo < 0.0f ? rmin : rmax);
    if (a_lo > 1.0f || a_hi < -1.0f) {
        empty = true;
        return;
    }
    w0 = phik - asinf(fminf(a_hi, 1.0f)) - 2e-3f;
    w1 = phik - asinf(fmaxf(a_lo, -1.0f)) + 2e-3f;
}

// Azimuth window [w0, w1] of the hits of one layer (radii in [rmin, rmax])
// with c > 0 in the column at phik whose distance from the seed circle is
// below tolw.  On the circle's implicit form a point at signed distance t
// gives kap |P|^2 - 2 P.g + h = t (2 + kap t), so with q = cos(psi_hit - psi)
//   |kap r^2 + h - 2 r |g| q| <= T,   T = tolw (2 + kap tolw):
// q lies between (kap r + (h -+ T) / r) / (2 |g|) at the ends of the radius
// range, or at the interior minimum sqrt(kap h) / |g| of kap r + h / r, and
// the hit on either side of psi.  Each side is kept where it meets the
// half-plane c > 0, their hull is the window.  Margins: 4e-6 of the terms'
// sizes and 1e-5 cm on T (float32 rounding of g and h and of the sums), and
// 2e-3 rad on the azimuth (acos near 1 for argument errors below 2e-6).
__device__ __forceinline__ void circle_window(const CfSeed &C, float phik, float tolw, float rmin,
                                              float rmax, bool &full, bool &empty, float &w0,
                                              float &w1)
{
    constexpr float kHalf = 1.57079633f + 4e-3f;   // c > 0, with a margin
    full = false;
    empty = !(rmin <= rmax);
    w0 = phik - kHalf;
    w1 = phik + kHalf;
    if (empty) return;
    const float k = C.F.kap, x1 = C.F.x1, y1 = C.F.y1;
    if (!(rmin >= 1e-3f) || !(C.gn >= 1e-3f) || !(C.F.B0 < 1e30f)) {
        full = true;
        return;
    }
    const float p1 = fabsf(x1) + fabsf(y1), W = rmax + p1;
    const float tw = tolw + fmaf(C.F.B2, W * W, fmaf(2.0f * C.F.B1, W, C.F.B0));
    const float T = fmaf(tw, fmaf(k, tw, 2.0f), 1e-5f) +
                    4e-6f * (k * fmaf(rmax, rmax, p1 * p1) + 2.0f * p1 + 2.0f * rmax * C.gn);
    const float ig = 0.5f / C.gn;
    const float ia = 1.0f / rmin, ib = 1.0f / rmax;
    const float qa = fmaf(k, rmin, C.h * ia), qb = fmaf(k, rmax, C.h * ib);
    float lo = fminf(qa, qb);
    if (C.h > k * rmin * rmin && C.h < k * rmax * rmax) lo = fminf(lo, 1.9999f * sqrtf(k * C.h));
    const float qlo = fmaf(-T, ia, lo) * ig - 2e-6f;
    const float qhi = fmaf(T, ia, fmaxf(qa, qb)) * ig + 2e-6f;
    if (qlo > 1.0f || qhi < -1.0f) {
        empty = true;
        return;
    }
    const float a1 = acosf(fminf(qhi, 1.0f)), a2 = acosf(fmaxf(qlo, -1.0f));
    if (!(a2 - a1 <= 1.0f)) return;   // wide: every hit with c > 0
    const float mid = 0.5f * (a1 + a2), hw = 0.5f * (a2 - a1) + 2e-3f;
    float l0 = 1e9f, h0 = -1e9f;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        float d = (side ? C.psi - mid : C.psi + mid) - phik;   // to [-pi, pi]
        d = fmaf(-6.28318531f, rintf(d * 0.159154943f), d);
        const float a = fmaxf(d - hw, -kHalf), b = fminf(d + hw, kHalf);
        if (a <= b) {
            l0 = fminf(l0, a);
            h0 = fmaxf(h0, b);
        }
    }
    empty = !(l0 <= h0);
    w0 = phik + l0;
    w1 = phik + h0;
}

// Lane (layer l, part) of a layer's window as a run of index positions: the
// window's cells, in two parts when they wrap.
__device__ __forceinline__ void window_run(const int *__restrict__ offs, int cell0, int part,
                                           bool full, bool empty, float w0, float w1, int &start,
                                           int &len)
{
    start = len = 0;
    if (empty) return;
    const float k = kIdxAz / 6.28318531f;
    const int b0 = (int)floorf((w0 + 3.14159265f) * k), b1 = (int)floorf((w1 + 3.14159265f) * k);
    const int nb = b1 - b0 + 1;
    const int *o = offs + cell0;
    int a = 0, b = kIdxAz;   // cells [a, b)
    if (full || nb >= kIdxAz) {
        if (part) return;
    } else {
        const int b0m = b0 & (kIdxAz - 1);
        const bool wrap = b0m + nb > kIdxAz;
        if (part && !wrap) return;
        a = part ? 0 : b0m;
        b = part ? b0m + nb - kIdxAz : wrap ? kIdxAz : b0m + nb;
    }
    start = o[a];
    len = o[b] - start;
}

// The run (window_run) of layer l's hits that can have a root in the bins
// [j0, j1) of column (rho, phi0_k): the bins' edges, a hundredth of a bin and
// 1e-4 cm beyond.
__device__ __forceinline__ void bin_run(const DevGeom &G, const HitIndex &I, int e, int l, int part,
                                        float rho, float phik, int j0, int j1, int &start, int &len)
{
    const float lo = fmaf((float)j0 - G.off_f - 0.01f, G.delta_f, -1e-4f);
    const float hi = fmaf((float)j1 - G.off_f + 0.01f, G.delta_f, 1e-4f);
    const float rmin = __uint_as_float(I.rmm[2 * (e * 16 + l)]);
    const float rmax = __uint_as_float(I.rmm[2 * (e * 16 + l) + 1]);
    bool full, empty;
    float w0, w1;
    layer_window(rho, phik, lo, hi, rmin, rmax, full, empty, w0, w1);
    window_run(I.offs, (e * 16 + l) * kIdxAz, part, full, empty, w0, w1, start, len);
}

// Whether the root of a hit in column (rho, phi0) that grows through F = 0 is
// between da and db (cm): F(d) = rho d^2 + 2 (1 + rho s) d + rho r^2 + 2 s of
// the circle equation is linear in s and r^2, so its signs at the two ends
// decide, without a square root.  dF/dd = 2 (1 + rho (s + d)), and where that
// is positive at both ends F is monotone between them: one root there when
// F(da) < 0 < F(db), else none (the other root, if any, is outside).
// Returns 0 (no root), 1 (a root), or 2: too close to an end for float32,
// or dF/dd or the sign of c not proven.  The bound is first order (u = 2^-24,
// taken four times): s is within 3u R1, r^2 within 2u, the tables' rho within
// u, da and db within 2u of themselves:
//   u (11 R1 + 6 |rho| R1^2 + 12 dmax).
struct EdgePair {
    float ka, la, kb, lb, ma, mb, ce, rho;

    __device__ __forceinline__ void init(const DevGeom &G, float rho_, int j0, int j1)
    {
        rho = rho_;
        const float da = ((float)j0 - G.off_f) * G.delta_f, db = ((float)j1 - G.off_f) * G.delta_f;
        ka = fmaf(rho * da, da, 2.0f * da);
        kb = fmaf(rho * db, db, 2.0f * db);
        la = fmaf(2.0f * rho, da, 2.0f);
        lb = fmaf(2.0f * rho, db, 2.0f);
        ma = fmaf(rho, da, 1.0f);
        mb = fmaf(rho, db, 1.0f);
        ce = 12.0f * G.dext_f;
    }

    __device__ __forceinline__ int root(float x, float y, float sk, float ck) const
    {
        const float s = fmaf(x, sk, -(y * ck)), c = fmaf(x, ck, y * sk);
        const float R1 = fabsf(x) + fabsf(y);
        const float Ec = (kSafe * 3.0f * kEps) * R1;
        const float base = rho * fmaf(x, x, y * y);
        const float Fa = fmaf(la, s, ka + base), Fb = fmaf(lb, s, kb + base);
        const float e = (kSafe * kEps) * fmaf(fmaf(6.0f * fabsf(rho), R1, 11.0f), R1, ce);
        const float m = fminf(fmaf(rho, s, ma), fmaf(rho, s, mb));
        if (c < -Ec) return 0;
        if (!(c > Ec && m > 0.05f)) return 2;
        if (Fa > e || Fb < -e) return 0;
        return Fa < -e && Fb > e ? 1 : 2;
    }
};

// The same by the vote's exact bin decision: a bin in [j0, j1).
static __device__ __noinline__ bool exact_root(const DevGeom &G, int i, int k, float x, float y,
                                               int j0, int j1)
{
    ColumnCtx C;
    C.init(G, i, k);
    int jj[2];
    const int nv = column_bins(G, C, x, y, jj);
    bool in = false;
    for (int v = 0; v < nv; ++v) in |= jj[v] >= j0 && jj[v] < j1;
    return in;
}

// The seeds of one candidate of event e: scans, per layer, the hits whose
// azimuth can give a root in its bin, and takes the layers with one own hit.
__device__ __forceinline__ void find_seeds(const DevGeom &G, const ConfirmDev &P,
                                           const HitIndex &I, int e, const ht_peak pk, CfSeed &out,
                                           int wid, int lane)
{
    constexpr unsigned kAll = 0xffffffffu;
    CfWarp &W = g_cfw[wid];
    const float rho = G.rho32[pk.i_rho], phik = G.phi32[pk.k_phi0];
    Runs R;
    {
        const int l = lane >> 1;
        int start = 0, len = 0;
        if (l < P.n_layers)
            bin_run(G, I, e, l, lane & 1, rho, phik, pk.j_d0, pk.j_d0 + 1, start, len);
        R.set(start, len, l, wid, lane);
    }
    const float sk = G.sn32[pk.k_phi0], ck = G.cs32[pk.k_phi0];
    EdgePair E;
    E.init(G, rho, pk.j_d0, pk.j_d0 + 1);
    unsigned once = 0u, twice = 0u;   // layers with an own hit, with more
    for (int base = 0; base < R.n; base += 32) {
        int p = 0, l = 0;
        int st = 0;
        if (R.at(base, lane, p, l)) {
            const float x = I.x[p], y = I.y[p];
            st = E.root(x, y, sk, ck);
            if (st == 2)
                st = exact_root(G, pk.i_rho, pk.k_phi0, x, y, pk.j_d0, pk.j_d0 + 1) ? 1 : 0;
        }
        const bool own = st == 1;
        const unsigned bo = __ballot_sync(kAll, own);
        if (bo) {
            const unsigned m = __reduce_or_sync(kAll, own ? 1u << l : 0u);
            if (__popc(bo) != __popc(m)) {   // a layer twice in this step
                const unsigned peers = __match_any_sync(kAll, own ? l : 32 + lane);
                twice |= __reduce_or_sync(kAll, own && __popc(peers) > 1 ? 1u << l : 0u);
            }
            twice |= once & m;
            once |= m;
            if (own) W.own_pos[l] = p;   // read only where the layer holds exactly one own hit
        }
    }
    __syncwarp();
    // the first, the last, and the layer between them nearest their middle
    // (the smaller on a tie)
    const unsigned seeds = once & ~twice;
    int pa = -1, pb = -1, pc = -1;
    if (__popc(seeds) >= 3) {
        const int la = __ffs(seeds) - 1, lc = 31 - __clz(seeds), t2 = la + lc;
        const unsigned inner = seeds & ~(1u << la) & ~(1u << lc);
        const unsigned low = inner & ((2u << (t2 >> 1)) - 1u), high = inner & ~low;
        const int l1 = 31 - __clz(low), l2 = __ffs(high) - 1;   // -1: none
        const int lb = !high ? l1 : !low ? l2 : t2 - 2 * l1 <= 2 * l2 - t2 ? l1 : l2;
        pa = W.own_pos[la];
        pb = W.own_pos[lb];
        pc = W.own_pos[lc];
    }
    if (lane == 0) {
        out.pa = pa;
        out.pb = pb;
        out.pc = pc;
        out.ev = e;
    }
    __syncwarp();   // own_pos is reused
}

// The seed frame of one candidate (a lane per candidate: the float64
// products of up to 32 candidates at once).
__device__ __forceinline__ void make_frame(const HitIndex &I, CfSeed &C)
{
    if (C.pa < 0) return;
    SeedFrame F;
    if (!seed_frame(I.x[C.pa], I.y[C.pa], I.x[C.pb], I.y[C.pb], I.x[C.pc], I.y[C.pc], F)) {
        C.pa = -1;
        return;
    }
    const float gx = fmaf(F.kap, F.x1, F.nx), gy = fmaf(F.kap, F.y1, F.ny);
    C.F = F;
    C.psi = atan2f(gy, gx);
    C.gn = sqrtf(fmaf(gx, gx, gy * gy));
    C.h = fmaf(F.kap, fmaf(F.x1, F.x1, F.y1 * F.y1), 2.0f * fmaf(F.x1, F.nx, F.y1 * F.ny));
}

// Confirmation of one candidate with a seed frame, by one warp.  Returns the
// number of inlier layers when it is confirmed (W.best_h[l] of lanes with
// in_l: the inlier hits), else 0.
//
// Distances: the float32 estimate of seed_frame and its bound give a hit an
// interval [lo, hi] holding its float64 distance.  Only hits with lo below
// tol can be inliers: the scan, over the azimuth cells the circle crosses,
// keeps those, and where they lie on fewer than min_layers layers the
// candidate is not confirmed.  Otherwise the pool's hits among them are
// found, and per layer the contenders: the hits with lo at most the layer's
// least hi; the layer's nearest hit is one of them.  A layer without a
// contender has no inlier, a single contender certainly below tol is the
// inlier, and otherwise the float64 distances of the contenders decide (the
// definition's seed circle is computed then, once per candidate).  More than
// kCfCap hits go in passes of as many whole layers as fit, each scan going on
// where the pass before it ended; of a layer with more hits than that, every
// contender goes by its float64 distance.
//
// WIDE: the tolerance is of the size of the pool, so the circle's cells can
// hold more hits than the pool's, and most pool hits are near it.  Each layer
// then scans whichever cells hold fewer, the pool test comes first, and only
// the pool's hits are kept.  10k hits, bins of 0.31 cm: pool 4, tol 1.5 and 100
// cm 1.66 -> 0.95 and 80 -> 0.99 ms; pool 0 1.52 -> 0.47 and 80 -> 0.47.
template <bool WIDE>
__device__ __forceinline__ int confirm_one(const DevGeom &G, const ConfirmDev &P,
                                           const HitIndex &I, const ht_peak pk, const CfSeed &C,
                                           float tol_lo, float tol_hi, int wid, int lane,
                                           bool &in_l)
{
    CfWarp &W = g_cfw[wid];
    constexpr unsigned kAll = 0xffffffffu;
    const float kInf = __int_as_float(0x7f800000);
    const int e = C.ev;
    const float rho = G.rho32[pk.i_rho], phik = G.phi32[pk.k_phi0];
    const int pool = min(P.pool, G.n_d0);   // (any int32 is accepted)
    const int jp0 = max(pk.j_d0 - pool, 0), jp1 = min(pk.j_d0 + pool + 1, G.n_d0);
    Runs R;
    {
        const int l = lane >> 1;
        int start = 0, len = 0;
        if (l < P.n_layers) {
            const float rmin = __uint_as_float(I.rmm[2 * (e * 16 + l)]);
            const float rmax = __uint_as_float(I.rmm[2 * (e * 16 + l) + 1]);
            bool full, empty;
            float w0, w1;
            circle_window(C, phik, tol_hi, rmin, rmax, full, empty, w0, w1);
            window_run(I.offs, (e * 16 + l) * kIdxAz, lane & 1, full, empty, w0, w1, start, len);
        }
        if (WIDE) {
            int ps = 0, pl = 0;
            if (l < P.n_layers) bin_run(G, I, e, l, lane & 1, rho, phik, jp0, jp1, ps, pl);
            if (pl + __shfl_xor_sync(kAll, pl, 1) < len + __shfl_xor_sync(kAll, len, 1)) {
                start = ps;
                len = pl;
            }
        }
        R.set(start, len, l, wid, lane);
    }
    in_l = false;
    const SeedFrame F = C.F;
    EdgePair E;   // the pool's edges (where most candidates end before: not yet)
    float sk, ck;
    auto pool_init = [&]() {
        E.init(G, rho, jp0, jp1);
        sk = G.sn32[pk.k_phi0];
        ck = G.cs32[pk.k_phi0];
    };
    auto in_pool = [&](float x, float y) -> bool {
        const int st = E.root(x, y, sk, ck);
        return st == 2 ? exact_root(G, pk.i_rho, pk.k_phi0, x, y, jp0, jp1) : st == 1;
    };
    if (WIDE) pool_init();
    int total = 0;
    // hits of rank [r0, r0 + kCfCap) near the circle (WIDE: and in the pool), in
    // layer order, and the one behind them, the first at place t0 of the sequence;
    // the first scan (r0 = 0) goes through all hits, sets total and returns their
    // layers
    auto scan = [&](int r0, int t0) {
        unsigned lm = 0u;
        int rank = r0;
        for (int base = t0; base < R.n && (r0 == 0 || rank <= r0 + kCfCap); base += 32) {
            int p = 0, l = 0;
            float lo = kInf, hi = kInf;
            if (R.at(base, lane, p, l)) {
                const float x = I.x[p], y = I.y[p];
                if (!WIDE || in_pool(x, y)) {
                    const float wx = x - F.x1, wy = y - F.y1;
                    const float w2 = fmaf(wx, wx, wy * wy);
                    const float wn = fmaf(wx, F.nx, wy * F.ny);
                    const float num = fmaf(F.kap, w2, -2.0f * wn);
                    const float qx = fmaf(F.kap, wx, -F.nx), qy = fmaf(F.kap, wy, -F.ny);
                    const float d = fabsf(num / (sqrtf(fmaf(qx, qx, qy * qy)) + 1.0f));
                    const float er = fmaf(F.B2, w2, fmaf(F.B1, fabsf(wx) + fabsf(wy), F.B0));
                    const float dl = __fsub_rd(d, er);
                    lo = dl > 0.0f ? dl : 0.0f;   // +0 (the bits order as the values)
                    hi = __fadd_ru(d, er);
                }
            }
            const bool near = lo < tol_hi;
            const unsigned bal = __ballot_sync(kAll, near);
            if (!bal) continue;
            const int r = rank + __popc(bal & ((1u << lane) - 1u)) - r0;
            if (near && r <= kCfCap) {
                W.pool_p[r] = p;
                W.pool_l[r] = (unsigned char)l;
                W.pool_lo[r] = lo;
                W.pool_hi[r] = hi;
            }
            lm |= __reduce_or_sync(kAll, near ? 1u << l : 0u);
            rank += __popc(bal);
        }
        if (r0 == 0) total = rank;
        return lm;
    };
    if (__popc(scan(0, 0)) < P.min_layers) return 0;
    if (lane < 16) {
        W.best_h[lane] = -1;
        W.best_d[lane] = 0.0;
    }
    const long long tol_bits = __double_as_longlong(P.tol);
    const bool single = total <= kCfCap;
    if (!WIDE) pool_init();
    bool exact = false;
    unsigned split = 0u;   // layers that one pass does not hold
    for (int r0 = 0, t0 = 0, next = 0; r0 < total; r0 = next) {
        if (r0 > 0) scan(r0, t0);
        int nq = min(total - r0, kCfCap);
        __syncwarp();
        if (r0 + nq < total) {   // the layer that the pass ends in waits for the next one
            const int first = W.pool_l[0], last = W.pool_l[nq - 1];
            if (first != last) {
                int n = 0;
                for (int q0 = 0; q0 < nq; q0 += 32)
                    n += __popc(__ballot_sync(kAll, q0 + lane < nq && W.pool_l[q0 + lane] != last));
                nq = n;
            } else {
                split |= 1u << last;
            }
            t0 = R.place(W.pool_p[nq], lane);
        }
        next = r0 + nq;
        __syncwarp();
        // the pool's hits among them, kept in order
        int kept = 0;
        for (int q0 = 0; q0 < nq; q0 += 32) {
            const int q = q0 + lane;
            int p = 0;
            bool in = false;
            unsigned char l = 0;
            float lo = 0.0f, hi = 0.0f;
            if (q < nq) {
                p = W.pool_p[q];
                l = W.pool_l[q];
                lo = W.pool_lo[q];
                hi = W.pool_hi[q];
                in = WIDE || in_pool(I.x[p], I.y[p]);
            }
            const unsigned bal = __ballot_sync(kAll, in);
            if (in) {
                const int r = kept + __popc(bal & ((1u << lane) - 1u));
                W.pool_p[r] = p;   // r <= q: read before
                W.pool_l[r] = l;
                W.pool_lo[r] = lo;
                W.pool_hi[r] = hi;
                W.pool_h[r] = I.h[p];
            }
            kept += __popc(bal);
            __syncwarp();
        }
        nq = kept;
        if (lane < 16) {
            W.lbmin[lane] = W.ubmin[lane] = 0x7f800000u;   // +inf
            W.ncont[lane] = 0;
            W.qs[lane] = kCfCap;
            W.qe[lane] = 0;
        }
        __syncwarp();
        // the least bounds per layer (each layer is one run of positions)
        for (int q0 = 0; q0 < nq; q0 += 32) {
            const int q = q0 + lane;
            const int l = q < nq ? W.pool_l[q] : 16;
            float slo = q < nq ? W.pool_lo[q] : kInf, shi = q < nq ? W.pool_hi[q] : kInf;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float olo = __shfl_down_sync(kAll, slo, o);
                const float ohi = __shfl_down_sync(kAll, shi, o);
                const int ol = __shfl_down_sync(kAll, l, o);
                if (lane + o < 32 && ol == l) {
                    slo = fminf(slo, olo);
                    shi = fminf(shi, ohi);
                }
            }
            const int lp = __shfl_up_sync(kAll, l, 1), ln = __shfl_down_sync(kAll, l, 1);
            if (q < nq && (lane == 0 || lp != l)) {
                atomicMin(&W.lbmin[l], __float_as_uint(slo));
                atomicMin(&W.ubmin[l], __float_as_uint(shi));
                atomicMin(&W.qs[l], q);
            }
            if (q < nq && (lane == 31 || ln != l)) atomicMax(&W.qe[l], q + 1);
        }
        __syncwarp();
        if (single) {
            // layers that can hold an inlier at all: too few, not confirmed
            const bool can = lane < P.n_layers && __uint_as_float(W.lbmin[lane]) < tol_hi;
            if (__popc(__ballot_sync(kAll, can)) < P.min_layers) return 0;
        }
        for (int q = lane; q < nq; q += 32) {
            const int l = W.pool_l[q];
            if (W.pool_lo[q] <= __uint_as_float(W.ubmin[l])) {
                atomicAdd(&W.ncont[l], 1);
                W.cq[l] = q;   // read only where the layer has one contender
            }
        }
        __syncwarp();
        bool need = false;
        if (lane < P.n_layers) {
            const int nc = W.ncont[lane];
            if (!((split >> lane) & 1u) && nc == 1 && W.pool_hi[W.cq[lane]] < tol_lo) {
                W.best_h[lane] = W.pool_h[W.cq[lane]];   // certainly the inlier
                W.best_d[lane] = 0.0;                     // (below tol)
            } else {
                need = nc > 0;
            }
        }
        const unsigned need_m = __ballot_sync(kAll, need);
        if (need_m != 0u && !exact) {
            if (lane == 0)
                circle3((double)I.x[C.pa], (double)I.y[C.pa], (double)I.x[C.pb], (double)I.y[C.pb],
                        (double)I.x[C.pc], (double)I.y[C.pc], W.xc, W.yc, W.R);
            __syncwarp();
            exact = true;
        }
        for (unsigned m = need_m; m != 0u; m &= m - 1u) {
            const int l = __ffs(m) - 1;
            const float ub = __uint_as_float(W.ubmin[l]);
            long long bk = 0x7fffffffffffffffll;   // none: above every distance's bits
            int bh = -1;
            for (int q = W.qs[l] + lane; q < W.qe[l]; q += 32) {
                if (!(W.pool_lo[q] <= ub)) continue;
                const int p = W.pool_p[q], h = W.pool_h[q];
                const long long key = __double_as_longlong(circle_dist(I.x[p], I.y[p], W.xc, W.yc, W.R));
                if (key < bk || (key == bk && h < bh)) {
                    bk = key;
                    bh = h;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const long long ok2 = __shfl_xor_sync(kAll, bk, o);
                const int oh = __shfl_xor_sync(kAll, bh, o);
                if (ok2 < bk || (ok2 == bk && oh < bh)) {
                    bk = ok2;
                    bh = oh;
                }
            }
            if (lane == 0 && bh >= 0) {
                const long long cur = __double_as_longlong(W.best_d[l]);
                if (W.best_h[l] < 0 || bk < cur || (bk == cur && bh < W.best_h[l])) {
                    W.best_d[l] = __longlong_as_double(bk);
                    W.best_h[l] = bh;
                }
            }
        }
        __syncwarp();
    }
    in_l = lane < P.n_layers && W.best_h[lane] >= 0 &&
           __double_as_longlong(W.best_d[lane]) < tol_bits;
    const int sc = __popc(__ballot_sync(kAll, in_l));
    return sc >= P.min_layers ? sc : 0;
}

// Confirmation of every kept candidate of a batch (cpre: exclusive prefix of
// the events' kept counts), persistent: each warp takes chunks of consecutive
// candidates from a device counter (*head, zero at launch; as many as keep
// every warp busy, at most kCfChunk).  Of a chunk it finds the seeds
// candidate by candidate, the seed frames all at once (a lane each), then
// confirms candidate by candidate.  A confirmed candidate's inliers offer
// the key score << 32 | (2^32 - 1 - m) to their hits: the largest wins (most
// inlier layers, then the smallest candidate index); gbest (batch hit index)
// must be zero, k_assoc_final_batch decodes it.  score per slot (0 = not
// confirmed); inl (may be null): 16 inlier hits per slot, -1 none.  I: the
// batch's hit index (k_hitindex.cu).
template <bool WIDE>
__global__ void __launch_bounds__(kCfThreads, 8)
k_confirm(DevGeom G, ConfirmDev P, HitIndex I, const int *__restrict__ off,
          const int *__restrict__ d_nev, const ht_peak *__restrict__ peaks, int cap,
          const int *__restrict__ cpre, int *__restrict__ score, int *__restrict__ inl,
          unsigned long long *__restrict__ gbest, int *__restrict__ head)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    CfWarp &W = g_cfw[wid];
    const int n_ev = *d_nev;
    const int total = cpre[n_ev];
    const int chunk = min(max(total / (int)(gridDim.x * kCfWarps * 2), 1), kCfChunk);
    float tol_hi = (float)P.tol;   // tol rounded up to float32
    if ((double)tol_hi < P.tol) tol_hi = nextafterf(tol_hi, 3.0e38f);
    float tol_lo = (float)P.tol;   // and down
    if ((double)tol_lo > P.tol) tol_lo = nextafterf(tol_lo, 0.0f);
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(head, 1);
        const long long t64 = (long long)__shfl_sync(0xffffffffu, c, 0) * chunk;
        if (t64 >= total) break;
        const int t0 = (int)t64, n = min(chunk, total - t0);
        int e = event_of(cpre, n_ev, t0);
        for (int q = 0; q < n; ++q) {
            while (t0 + q >= cpre[e + 1]) ++e;   // t < cpre[n_ev]
            find_seeds(G, P, I, e, peaks[(size_t)e * cap + (t0 + q - cpre[e])], W.seed[q], wid, lane);
        }
        if (lane < n) make_frame(I, W.seed[lane]);
        __syncwarp();
        for (int q = 0; q < n; ++q) {
            const CfSeed &C = W.seed[q];
            const int m = t0 + q - cpre[C.ev];
            const size_t slot = (size_t)C.ev * cap + m;
            bool in_l = false;
            int sc = 0;
            if (C.pa >= 0)
                sc = confirm_one<WIDE>(G, P, I, peaks[slot], C, tol_lo, tol_hi, wid, lane, in_l);
            if (lane == 0) score[slot] = sc;
            if (inl && lane < 16) inl[slot * 16 + lane] = sc > 0 && in_l ? W.best_h[lane] : -1;
            if (sc > 0 && in_l)
                atomicMax(&gbest[off[C.ev] + W.best_h[lane]],
                          ((unsigned long long)sc << 32) | (0xffffffffull - (unsigned)m));
            __syncwarp();
        }
    }
}

// cpre[e] = sum over events before e of min(counts[e], cap); cpre[n_ev] is
// the total.  One block; n_ev <= 4096.
__global__ void __launch_bounds__(1024)
k_cand_prefix(const int *__restrict__ counts, const int *__restrict__ d_nev, int cap,
              int *__restrict__ cpre)
{
    __shared__ int part[1024];
    const int n_ev = *d_nev;
    const int per = (n_ev + 1023) / 1024;
    const int e0 = threadIdx.x * per;
    int sum = 0;
    for (int e = e0; e < min(e0 + per, n_ev); ++e) sum += min(counts[e], cap);
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {   // inclusive scan (Hillis-Steele)
        const int v = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = threadIdx.x ? part[threadIdx.x - 1] : 0;
    for (int e = e0; e < min(e0 + per, n_ev); ++e) {
        cpre[e] = run;
        run += min(counts[e], cap);
    }
    if (threadIdx.x == 1023) cpre[n_ev] = part[1023];
}

__global__ void k_single_offsets(int *__restrict__ off, int *__restrict__ nev, int n)
{
    off[0] = 0;
    off[1] = n;
    nev[0] = 1;
}

}  // namespace

cudaError_t launch_assoc_final_batch(const unsigned long long *gbest, const int *off,
                                     const int *d_nev, int *assign, int max_hits, cudaStream_t st);

namespace {

struct CfWs {
    int *cpre, *head;
    unsigned long long *gbest;
};

// Carves (p non-null) or sizes the confirmation workspace.
size_t cf_layout(int max_events, int max_hits, char *p, CfWs *w)
{
    const size_t parts[] = {(size_t)(max_events + 1) * 4, 64,
                            (size_t)(max_hits > 0 ? max_hits : 1) * 8};
    size_t at = 0;
    char *q[3];
    for (int i = 0; i < 3; ++i) {
        q[i] = p ? p + at : nullptr;
        at += align256(parts[i]);
    }
    if (w) {
        w->cpre = reinterpret_cast<int *>(q[0]);
        w->head = reinterpret_cast<int *>(q[1]);
        w->gbest = reinterpret_cast<unsigned long long *>(q[2]);
    }
    return at;
}

}  // namespace

cudaError_t prepare_confirm_kernels() { return cudaSuccess; }

// Confirmation and final assignment of a batch (device offsets and event
// count; idx: its hit index; inl may be null).  ws: confirm_workspace_bytes(
// max_events, max_hits).
size_t confirm_workspace_bytes(int max_events, int max_hits)
{
    return cf_layout(max_events, max_hits, nullptr, nullptr);
}

cudaError_t launch_confirm_batch(const DevGeom &G, const ConfirmDev &P, const int *off,
                                 const int *d_nev, int max_events, int max_hits,
                                 const ht_peak *peaks, const int *counts, int cap, int *score,
                                 int *inl, int *assign, void *ws, const HitIndex &idx, int sms,
                                 cudaStream_t st)
{
    CfWs w;
    cf_layout(max_events, max_hits, reinterpret_cast<char *>(ws), &w);
    cudaError_t e = cudaMemsetAsync(w.head, 0, 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(w.gbest, 0, (size_t)max_hits * 8, st);
    if (e != cudaSuccess) return e;
    k_cand_prefix<<<1, 1024, 0, st>>>(counts, d_nev, cap, w.cpre);
    // Half the pool's width: below it the circle's cells are the fewer.  10k hits,
    // narrow and wide kernel: pool 0 (0.31 cm) tol 0.1 364 and 397 us, 0.4 485 and
    // 452; pool 4 (2.8 cm) 0.8 629 and 648, 1.5 1006 and 897; pool 20 (12.8 cm)
    // 3 1461 and 1509, 6 2260 and 2208.
    const bool wide = P.tol > 0.5 * (2.0 * (double)P.pool + 1.0) * G.delta;
    const auto kernel = wide ? k_confirm<true> : k_confirm<false>;
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kCfThreads, 0);
    kernel<<<sms * (occ > 0 ? occ : 1), kCfThreads, 0, st>>>(
        G, P, idx, off, d_nev, peaks, cap, w.cpre, score, inl, w.gbest, w.head);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_assoc_final_batch(w.gbest, off, d_nev, assign, max_hits, st);
}

// One event (host hit count n, device candidate count d_count).
size_t confirm_workspace_bytes_single(int n)
{
    return align256(16) + hit_index_bytes(1, n) + confirm_workspace_bytes(1, n);
}

cudaError_t launch_confirm(const DevGeom &G, const ConfirmDev &P, const float *x, const float *y,
                           const uint8_t *layer, int n, const ht_peak *peaks, const int *d_count,
                           int cap, int *score, int *inl, int *assign, void *ws, cudaStream_t st)
{
    int *meta = reinterpret_cast<int *>(ws);   // off[2], n_ev
    k_single_offsets<<<1, 1, 0, st>>>(meta, meta + 2, n);
    char *p = reinterpret_cast<char *>(ws) + align256(16);
    const HitIndex idx = carve_hit_index(1, n, p);
    const int sms = device_sms();
    const cudaError_t e = launch_hit_index(x, y, layer, meta, meta + 2, 1, n, idx, sms, st);
    if (e != cudaSuccess) return e;
    return launch_confirm_batch(G, P, meta, meta + 2, 1, n, peaks, d_count, cap,
                                score, inl, assign, p + hit_index_bytes(1, n), idx, sms, st);
}


// ------------------------------------------------------------ compaction
// The confirmed candidates (score > 0) of every event, in candidate order,
// as a compact list of found tracks, and each hit's assignment as an index
// into its event's tracks (ht_batch_run_tracks_host).
namespace {

__global__ void k_track_flags(const int *__restrict__ d_nev, const int *__restrict__ cpre,
                              int cap, const int *__restrict__ score, int *__restrict__ flag)
{
    const int n_ev = *d_nev, total = cpre[n_ev];
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < total; f += gridDim.x * blockDim.x) {
        const int e = event_of(cpre, n_ev, f);
        flag[f] = score[(size_t)e * cap + (f - cpre[e])] > 0 ? 1 : 0;
    }
}

// tfirst[e] = the compact index of event e's first track (e <= n_ev)
__global__ void k_track_first(const int *__restrict__ d_nev, const int *__restrict__ cpre,
                              const int *__restrict__ pos, const int *__restrict__ ntot,
                              int *__restrict__ tfirst)
{
    const int n_ev = *d_nev, total = cpre[n_ev];
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e <= n_ev; e += gridDim.x * blockDim.x)
        tfirst[e] = cpre[e] < total ? pos[cpre[e]] : *ntot;
}

__global__ void k_track_write(const int *__restrict__ d_nev, const int *__restrict__ cpre,
                              int cap, const int *__restrict__ flag, const int *__restrict__ pos,
                              const int *__restrict__ tfirst, const ht_peak *__restrict__ peaks,
                              const int *__restrict__ score, const ht_zres *__restrict__ zres,
                              ht_track_out *__restrict__ tracks, int tcap, int *__restrict__ map)
{
    const int n_ev = *d_nev, total = cpre[n_ev];
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < total; f += gridDim.x * blockDim.x) {
        if (!flag[f]) continue;
        const int e = event_of(cpre, n_ev, f);
        const size_t slot = (size_t)e * cap + (f - cpre[e]);
        const int t = pos[f];
        map[slot] = t - tfirst[e];
        if (t < tcap) {
            const ht_peak pk = peaks[slot];
            const ht_zres zr = zres[slot];
            tracks[t] = ht_track_out{pk.i_rho, pk.j_d0, pk.k_phi0, pk.count, score[slot],
                                     zr.n_z0, zr.m_cot, zr.count};
        }
    }
}

__global__ void k_track_assign(const int *__restrict__ off, const int *__restrict__ d_nev,
                               int cap, const int *__restrict__ assign,
                               const int *__restrict__ map, int *__restrict__ out)
{
    const int n_ev = *d_nev, n = off[n_ev];
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < n; h += gridDim.x * blockDim.x) {
        int lo = 0, hi = n_ev - 1;   // the hit's event
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= h) lo = mid;
            else hi = mid - 1;
        }
        const int a = assign[h];
        out[h] = a >= 0 ? map[(size_t)lo * cap + a] : -1;
    }
}

}  // namespace

size_t track_compact_bytes(int max_events, int cap)
{
    const size_t nk = (size_t)max_events * (cap > 0 ? cap : 1);
    return align256((size_t)(max_events + 1) * 4) + 2 * align256((size_t)(max_events + 1) * 4) +
           3 * align256(nk * 4) + align256(16) + scan_tmp_bytes((int)nk);
}

cudaError_t launch_track_compact(const int *off, const int *d_nev, int max_events, int max_hits,
                                 const ht_peak *peaks, const int *counts, int cap,
                                 const int *score, const ht_zres *zres, const int *assign,
                                 ht_track_out *tracks, int tcap, int *tfirst, int *ntot,
                                 int *assign_out, void *ws, int sms, cudaStream_t st)
{
    const size_t nk = (size_t)max_events * (cap > 0 ? cap : 1);
    char *p = reinterpret_cast<char *>(ws);
    int *cpre = reinterpret_cast<int *>(p);
    p += align256((size_t)(max_events + 1) * 4);
    p += 2 * align256((size_t)(max_events + 1) * 4);
    int *flag = reinterpret_cast<int *>(p);
    p += align256(nk * 4);
    int *pos = reinterpret_cast<int *>(p);
    p += align256(nk * 4);
    int *map = reinterpret_cast<int *>(p);
    p += align256(nk * 4);
    p += align256(16);
    void *tmp = p;
    k_cand_prefix<<<1, 1024, 0, st>>>(counts, d_nev, cap, cpre);
    k_track_flags<<<sms * 4, 256, 0, st>>>(d_nev, cpre, cap, score, flag);
    cudaError_t e = scan_exclusive(flag, pos, nullptr, (int)nk, nullptr, ntot, tmp, st);
    if (e != cudaSuccess) return e;
    k_track_first<<<(max_events + 256) / 256, 256, 0, st>>>(d_nev, cpre, pos, ntot, tfirst);
    k_track_write<<<sms * 4, 256, 0, st>>>(d_nev, cpre, cap, flag, pos, tfirst, peaks, score, zres,
                                            tracks, tcap, map);
    k_track_assign<<<sms * 4, 256, 0, st>>>(off, d_nev, cap, assign, map, assign_out);
    (void)max_hits;
    return cudaGetLastError();
}

}  // namespace ht
