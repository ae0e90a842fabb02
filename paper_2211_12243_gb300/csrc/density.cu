// Smoothing length and particle volume (§2.3.2 Eqs. 5-6, §2.3.5 Eq. 18):
// per particle, solve g(h) = (4 pi/3) h^3 sum_j W(r_ij, h) - N_NGB = 0 by
// safeguarded Newton over the particle's neighbour list, then
// omega = 1 / sum_j W(r_ij, h) (self term included).
//
// g is non-decreasing in h (h^3 W(r, h) is a function of r/h that grows as
// r/h falls), so [lo, hi] brackets the root; a Newton proposal outside the
// bracket (or beyond the list's search radius) is replaced by bisection or
// clamped.  The list covers every j with r < h_search, so g is exact for
// any h <= h_search; a root beyond h_search is reported for a re-search.
//
// Both paths iterate in float on the fixed-point separations.  FP64 path: the iteration is then
// finished in double by a third-order (Halley) step -- g and g' summed in
// double, g'', which only scales the square of the step, in float -- so that
// one pass over the list in double is enough.  Mixed path: one Newton step
// evaluated in double-float (pairs of floats, Dekker/Knuth error-free
// transformations) on the exact 64-bit separations refines h to double-class
// accuracy without the GPU's scarce FP64 pipe; omega is taken from that
// evaluation.
//
// Tight lists (hydro_step only): once an upper bracket hi of the root is
// known, no later iterate exceeds it, so the particle's list is compacted in
// place to the entries within hi (plus a relative slack that covers the
// float separation's error) and the last pass compacts it to the final h.
// The search radius hs is lowered to the radius the compacted list is
// complete for; the gradient and flux kernels, which test r_ij < h_i
// exactly on every entry, then walk only the members.  Compaction keeps the
// order of the entries, so the members are summed in the same order as in
// the full list.
#include "fp64.cuh"
#include "hydro_internal.cuh"
#include "row.cuh"
#include "tile_rank.cuh"

namespace hyd {

namespace {

struct DensArgs {
    int64_t n;
    const int64_t *nbr_off;
    int32_t *nbr_cnt;         // rewritten when lists are compacted
    int32_t *nbr_idx;
    double *hs;               // lowered to the compacted lists' radius
    const double *xs, *ys, *zs;
    const uint32_t *qx, *qy, *qz;
    const int32_t *pbox;
    const Box *boxes;
    uint8_t *active;          // bit0: solve this particle; bit1: search failed
    const double *nngb;       // per particle N_NGB (NULL: n_ngb)
    double n_ngb;
    int kernel;
    double tol;
    int max_iter;
    bool only_active;
    bool compact;             // compact the lists to the root (see above)
    double *h;                // sorted, in: guess, out: solution
    double *om;               // sorted out
    DevCounters *cnt;
    bool rank;                // full solve: rank the CTA's 128 particles by list length
    const int32_t *list;      // the guard round's particles, their count on the device
    const int *nlist;         // (k_density_list; NULL: every particle)
    const int32_t *buckets;   // a sparse sub-step's buckets (k_density_list; NULL: every particle)
    int nbuckets;
    const int32_t *node_first, *node_cnt;
    const uint4 *pos, *low;   // mixed path: high and low words of the 64-bit fixed-point x y z
};

// Growth of the search radius hs after a failed solve.  First failure
// (hs within 1.3 of the particle's h guess): the weighted count at the
// radius, kf = N_enc(hs), grows about as hs^3 in a locally uniform
// distribution, so the root lies near hs (N / kf)^(1/3): take 10% beyond
// that, at least 5% and at most a doubling.  A radius grown before: double.
__device__ __forceinline__ double search_growth(double N, double kf, double hs, double h) {
    if (!(hs <= 1.3 * h)) return 2.0;
    double g = kf > 0.0 ? 1.1 * cbrt(N / kf) : 2.0;
    return fmin(fmax(g, 1.05), 2.0);
}

// ------------------------------------------------------- double-float tools
// value = hi + lo, |lo| <= ulp(hi)/2
struct df {
    float hi, lo;
};
__device__ __forceinline__ df two_sum(float a, float b) {
    float s = a + b;
    float bb = s - a;
    float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
__device__ __forceinline__ df quick_two_sum(float a, float b) {
    float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ df two_prod(float a, float b) {
    float p = a * b;
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ df df_add(df a, df b) {
    df s = two_sum(a.hi, b.hi);
    df t = two_sum(a.lo, b.lo);
    s.lo += t.hi;
    s = quick_two_sum(s.hi, s.lo);
    s.lo += t.lo;
    return quick_two_sum(s.hi, s.lo);
}
// df_add of a single float: the same bits with half the operations
__device__ __forceinline__ df df_addf(df a, float b) {
    df s = two_sum(a.hi, b);
    s.lo += a.lo;
    return quick_two_sum(s.hi, s.lo);
}
// 1 - q, 0 <= q <= 1
__device__ __forceinline__ df df_one_minus(df q) {
    df s = quick_two_sum(1.f, -q.hi);
    s.lo -= q.lo;
    return quick_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ df df_mul(df a, df b) {
    df p = two_prod(a.hi, b.hi);
    p.lo += a.hi * b.lo + a.lo * b.hi;
    return quick_two_sum(p.hi, p.lo);
}
__device__ __forceinline__ df df_mulf(df a, float b) {
    df p = two_prod(a.hi, b);
    p.lo += a.lo * b;
    return quick_two_sum(p.hi, p.lo);
}
__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, {-b.hi, -b.lo}); }
// square root by one Newton correction of the float root
__device__ __forceinline__ df df_sqrt(df a) {
    if (a.hi <= 0.f) return {0.f, 0.f};
    float x = sqrtf(a.hi);
    df xx = two_prod(x, x);
    df r = df_sub(a, xx);
    float corr = __fdividef(r.hi, 2.f * x);
    return quick_two_sum(x, corr);
}
__device__ __forceinline__ df df_div(df a, df b) {
    float q1 = a.hi / b.hi;
    df r = df_sub(a, df_mulf(b, q1));
    float q2 = r.hi / b.hi;
    return quick_two_sum(q1, q2);
}
// difference of two 64-bit fixed-point coordinates given as their words
__device__ __forceinline__ long long fixed_diff(uint32_t hj, uint32_t lj, uint32_t hi, uint32_t li) {
    return (long long)((((uint64_t)hj << 32) | lj) - (((uint64_t)hi << 32) | li));
}
// float-float of a 64-bit integer |v| < 2^62 from three 21-bit pieces,
// each converted exactly without a conversion instruction
__device__ __forceinline__ df from_i64(long long v) {
    int32_t hi = (int32_t)(v >> 42);                                   // |hi| < 2^20
    int32_t mid = (int32_t)(((unsigned long long)v >> 21) & 0x1FFFFFull);
    int32_t lo = (int32_t)((unsigned long long)v & 0x1FFFFFull);
    float fh = i2f_small(hi) * 4398046511104.0f;                       // 2^42
    float fm = i2f_small(mid) * 2097152.0f;                            // 2^21
    // (each term is at least as large as what is added to it, or zero)
    const df s = quick_two_sum(fh, fm);
    df t = quick_two_sum(s.hi, i2f_small(lo));
    t.lo += s.lo;
    return quick_two_sum(t.hi, t.lo);
}

// ------------------------------------------------- the iteration in float
constexpr int DENS_THREADS = 128;
static_assert(DENS_THREADS == RANK_THREADS, "the ranked tiles take 128 threads a round");
// particles that a warp each solves faster than a thread each (4,096: 78 -> 47 us,
// 8,000: 84 -> 67 us, 17,576: 82 -> 108 us)
constexpr int64_t DENS_WARP_MAX = 8192;

// separations a warp that walks one list keeps in shared memory
constexpr int DENS_CACHE = 1536;

// float separations of a particle from its list's entries, from the fixed-point
// positions: side by side (mixed path) or the coordinate arrays (FP64 path, in units
// of the box's longest side, so that their squares stay in the float range whatever
// the caller's unit of length).  Within 4e-7 r + 4e-10 L of the exact ones.
template <typename R>
struct Separation;
template <>
struct Separation<float> {
    const uint4 *pos;
    uint32_t qx, qy, qz;
    float sx, sy, sz;
    __device__ __forceinline__ Separation(const DensArgs &a, int64_t s, const Box &bx)
        : pos(a.pos), sx(bx.s[0]), sy(bx.s[1]), sz(bx.s[2]) {
        const uint4 pi = pos[s];
        qx = pi.x; qy = pi.y; qz = pi.z;
    }
    __device__ __forceinline__ float operator()(int j) const {
        const uint4 pj = pos[j];
        float dx = qdiff(qx, pj.x, sx);
        float dy = qdiff(qy, pj.y, sy);
        float dz = qdiff(qz, pj.z, sz);
        float r2 = dx * dx + dy * dy + dz * dz;
        return r2 > 0.f ? r2 * rsqrtf(r2) : 0.f;
    }
};
template <>
struct Separation<double> {
    const uint32_t *px, *py, *pz;
    uint32_t qx, qy, qz;
    float sx, sy, sz;
    __device__ __forceinline__ Separation(const DensArgs &a, int64_t s, const Box &bx)
        : px(a.qx), py(a.qy), pz(a.qz) {
        const double u = bx.rLmax * (1.0 / 4294967296.0);
        sx = (float)(bx.L[0] * u); sy = (float)(bx.L[1] * u); sz = (float)(bx.L[2] * u);
        qx = px[s]; qy = py[s]; qz = pz[s];
    }
    __device__ __forceinline__ float operator()(int j) const {
        float dx = qdiff(qx, px[j], sx);
        float dy = qdiff(qy, py[j], sy);
        float dz = qdiff(qz, pz[j], sz);
        float r2 = dx * dx + dy * dy + dz * dz;
        return r2 > 0.f ? r2 * rsqrtf(r2) : 0.f;
    }
};

struct NewtonF {
    float h;       // root (or where the iteration stopped)
    float comp;    // radius the compacted list is complete for (-1: not compacted)
    int c;         // entries of the list
    int it;        // evaluations
    bool conv, fail;
    bool flat;     // the sum hardly grows with h at the last evaluation (see FLAT)
    float kf;      // N_enc(hsi) = Kn sum f at a failure
};

// A particle's list walked by one lane (W = 1) or by the 32 of a warp (a guard
// round's few particles, whose lists at the doubled radius are long).  A warp
// gathers the separations in parallel, once, into shared memory (the first
// CACHE), and evaluates the refinement's entries in parallel.  The float
// iteration and the mixed path's refinement take their sums in the list's order
// in both forms, so a mixed root does not depend on which form solves it; the
// FP64 finish of a warp sums every 32nd entry per lane and folds, which rounds
// differently from a lane's serial sum.  A lane on its own gathers the
// separations again in every pass (a running step's h takes one or two passes;
// keeping 16 to 64 of a thread's separations in shared memory took its L1 and
// was between 7 % faster and 50 % slower).
template <int W>
struct Walk {
    static constexpr int CACHE = W == 1 ? 0 : DENS_CACHE;
    float *rs;     // the warp's cache
    int lane;      // 0 for W = 1
    template <typename T>
    __device__ __forceinline__ T sum(T v) const {
        if (W > 1)
            for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    // entry (j, r) of this lane, kept or not, moves behind the w kept before it
    __device__ __forceinline__ void keep(bool on, int32_t *idx, int j, float r, int &w) const {
        if (W == 1) {
            if (on) {
                idx[w] = j;
                w++;
            }
        } else {
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if (on) {
                const int t = w + __popc(m & ((1u << lane) - 1u));
                idx[t] = j;
                if (t < CACHE) rs[t] = r;
            }
            w += __popc(m);
            __syncwarp();
        }
    }
};

// A sum f whose logarithmic slope in h is below this fixes its float root too
// coarsely for the margin of a compacted list (f is good to about 1e-6, the margin
// is 5e-5): N_NGB within a few parts in a hundred of the particle's own term, where
// the slope of an ordinary N_NGB is about three.
constexpr float FLAT = 0.1f;

// the safeguarded Newton iteration of one particle over its list idx
template <int W, typename Sep>
__device__ __forceinline__ NewtonF newton_float(const DensArgs &a, const Sep &sep, int32_t *idx, int c,
                                                float h, float hsi, float N, float xmin,
                                                int max_iter, const Walk<W> &wk) {
    NewtonF o;
    o.comp = -1.f;
    o.conv = o.fail = false;
    o.flat = true;
    o.kf = 0.f;
    o.it = 0;
    const float Kn = kernel_Kn<float>(a.kernel);
    const float ftol = 2e-6f;
    float lo = 0.f, hi = -1.f;
    bool hi_flat = true;   // the bracket hi is that of a flat sum
    const int c0 = min(c, Walk<W>::CACHE);
    if (W > 1) {
#pragma unroll 4
        for (int k = wk.lane; k < c0; k += W) wk.rs[k] = sep(idx[k]);
        __syncwarp();
    }
    for (int it = 1; it <= max_iter; it++) {
        o.it = it;
        float f = 0.f, mq = 0.f, ih = 1.f / h;
        // an upper bracket well inside the list radius: drop the entries
        // beyond it (no later iterate exceeds hi).  Keeping the entries with
        // float r < X (1 + 1e-4) leaves the list complete for every
        // r < X (1 + 5e-5) when X > L / 65536, L the longest side, which sets the
        // separation's error (compaction is skipped below that)
        const bool shrink = a.compact && hi > xmin && hi < 0.8f * hsi && !hi_flat;
        const float keep = hi * 1.0001f;
        int w = 0;
        for (int k = 0; k < c; k++) {   // (every lane of a warp: the sums are in order)
            float r;
            if (W == 1) {
                const int j = idx[k];
                r = sep(j);
                if (shrink && r < keep) idx[w++] = j;
            } else {
                r = k < Walk<W>::CACHE ? wk.rs[k] : sep(idx[k]);
            }
            float fv, mv;
            kernel_f<float>(a.kernel, r * ih, fv, mv);
            f += fv;
            mq += mv;
        }
        if (shrink) {
            if (W > 1)
                for (int k0 = 0; k0 < c; k0 += W) {
                    const int k = k0 + wk.lane;
                    const int j = k < c ? idx[k] : 0;
                    const float r = k >= c ? INFINITY : k < Walk<W>::CACHE ? wk.rs[k] : sep(j);
                    wk.keep(r < keep, idx, j, r, w);
                }
            c = w;
            o.comp = hi * 1.00005f;
            hsi = o.comp;
        }
        float g = Kn * f - N;
        float dg = Kn * mq * ih;
        o.flat = !(mq > FLAT * f);
        if (g == 0.f) { o.conv = true; break; }
        if (g < 0.f) {
            if (h >= hsi) { o.fail = true; o.kf = Kn * f; break; }
            lo = fmaxf(lo, h);
        } else if (hi < 0.f || h < hi) {
            hi = h;
            hi_flat = o.flat;
        }
        float hn = dg > 0.f ? h - g / dg : -1.f;
        if (hn > 0.f && fabsf(hn - h) <= ftol * h && hn <= hsi) { h = hn; o.conv = true; break; }
        if (hi < 0.f) {
            if (!(hn > lo) || hn > 2.f * h) hn = 2.f * h;
            if (hn > hsi) hn = hsi;
        } else if (!(hn > lo && hn < hi)) {
            hn = 0.5f * (lo + hi);
        }
        h = hn;
    }
    o.h = h;
    o.c = c;
    return o;
}

// the root left the list radius: the radius grows, the particle is searched again
__device__ __forceinline__ void dens_fail(const DensArgs &a, int64_t s) {
    a.active[s] = (a.active[s] & ACT_GUARD) | 3;
    atomicAdd(&a.cnt->search_fail, 1);
    set_flag(a.cnt, ST_SEARCH);
}

// ---------------------------------------------------------------- FP64 path
// float evaluations before the iteration starts again in double
constexpr int FLOAT_ITER = 12;

// h^2 d^2f/dh^2 of f(r/h) in float
__device__ __forceinline__ float kernel_curv(int kernel, float q) {
    const float t = 1.f - q, q2 = q * q;
    if (kernel == 0) return -60.f * q2 * t * t * (1.f - 2.f * q);
    return q <= 0.5f ? -36.f * q2 + 72.f * q2 * q : 12.f * q * t * (q - t);
}

// Bound by the FP64 pipe: 23 FP64 instructions per neighbour in one pass,
// where five passes of Newton's iteration and one for omega, with a square
// root rounded correctly per neighbour, took about 220 (1.07 M tube 11.1 ->
// 2.95 ms, 300k log-normal box 4.7 -> 0.88 ms).
template <int W>
__device__ __forceinline__ void dens_one(const DensArgs &a, double *__restrict__ rec,
                                         const Walk<W> &wk, int64_t s) {
    if (s >= a.n) return;
    if (a.only_active && !(a.active[s] & 1)) return;
    const Box bx = a.boxes[a.pbox[s]];
    const double hsi_d = a.hs[s], hguess = a.h[s];
    const double N = a.nngb ? a.nngb[s] : a.n_ngb;
    int32_t *idx = a.nbr_idx + a.nbr_off[s];
    // (the float iteration's lengths are in units of the longest side)
    const double Lmax = bx.Lmax, rLmax = bx.rLmax;
    const float xmin = 1.f / 65536.f;
    const Separation<double> sep(a, s, bx);
    const float hsf = (float)(hsi_d * rLmax);
    float hf = (float)(hguess * rLmax);
    if (!(hf > 0.f) || hf > hsf) hf = hsf;
    // (a radius below 1e-4 of the box leaves the float separations less than
    // 4e-6 accurate: everything in double then)
    const NewtonF o = newton_float<W>(a, sep, idx, a.nbr_cnt[s], hf, hsf, (float)N, xmin,
                                      hsi_d > 1e-4 * Lmax ? min(a.max_iter, FLOAT_ITER) : 0, wk);
    const float slack = 1e-9f;   // (bounds the error of a float r)
    int c = o.c;
    // The same iteration in double from the float root (from the list radius
    // where it lies beyond, from the guess where the float iteration did not
    // settle): a step below 2e-6 h, taken to
    // third order, leaves an error below 1e-16 h.
    const double comp = (double)o.comp * Lmax;
    const double hsi = o.comp > 0.f ? comp : hsi_d;
    const double Kn = kernel_Kn<double>(a.kernel), iKn = a.kernel == 0 ? 1.0 / 14.0 : 3.0 / 32.0;
    const double M = N * iKn;   // sum f at the root
    double h = o.fail ? hsi_d : o.conv ? (double)o.h * Lmax : hguess;
    if (!(h > 0.0) || h > hsi) h = hsi;
    const double xi = a.xs[s], yi = a.ys[s], zi = a.zs[s];
    double lo = 0.0, hi = -1.0, F = 0.0;
    bool conv = false, fail = false;
    double crad = o.comp > 0.f ? comp : 0.0;
    const int left = a.max_iter - (o.conv || o.fail ? o.it : 0);   // evaluations left
    for (int it = 1; it <= (left > 1 ? left : 1); it++) {
        const double ih = 1.0 / h;   // (rounded correctly: its error is common to every q)
        double f = 0.0, f1 = 0.0, mq = 0.0;
        float s2 = 0.f;
        const float hh = narrow(h * rLmax);
        const float cut = hh * (1.f + 1e-5f) + slack, keep = hh * 1.0001f;
        // (the first pass of a converged float root compacts the list)
        const bool shrink = a.compact && it == 1 && o.conv && !o.flat && hh > xmin;
        int w = 0;
        for (int k0 = 0; k0 < c; k0 += W) {
            const int k = k0 + wk.lane;
            const bool in = W == 1 || k < c;
            const int j = in ? idx[k] : 0;
            const float rf = !in ? INFINITY : k < Walk<W>::CACHE ? wk.rs[k] : sep(j);
            if (shrink) wk.keep(rf < keep, idx, j, rf, w);
            if (rf >= cut) continue;   // W = 0
            const double dx = fold64(a.xs[j] - xi, bx.L[0]);
            const double dy = fold64(a.ys[j] - yi, bx.L[1]);
            const double dz = fold64(a.zs[j] - zi, bx.L[2]);
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            const double q = dnormal(r2) ? r2 * rsqrt64(r2) * ih : 0.0;   // (closer than 1e-154: r = 0)
            if (!dlt_pos(q, 1.0)) continue;
            const double t = 1.0 - q, t2 = t * t;
            double fn;
            if (a.kernel == 0) {
                const double t3 = t2 * t;
                fn = fma(t3 * t, fma(4.0, q, 1.0), f);
                mq = fma(20.0 * (q * q), t3, mq);
            } else if (!dlt_pos(0.5, q)) {
                const double q2 = q * q;
                fn = f + fma(6.0 * q2, q - 1.0, 1.0);
                mq = fma(q2, fma(-18.0, q, 12.0), mq);
            } else {
                fn = fma(2.0 * t2, t, f);
                mq = fma(6.0 * q, t2, mq);
            }
            f = f1;   // (two sums by turns: their rounding is most of h's error)
            f1 = fn;
            s2 += kernel_curv(a.kernel, narrow(q));
        }
        f = wk.sum(f + f1);
        mq = wk.sum(mq);
        s2 = wk.sum(s2);
        if (shrink) { c = w; crad = (double)hh * Lmax * (1.0 + 5e-5); }
        const double g = f - M;   // (g / Kn)
        F = f;
        if (g == 0.0) { conv = true; break; }
        if (g < 0.0) {
            if (h >= hsi) {
                fail = true;
                F = Kn * f;
                break;
            }
            lo = fmax(lo, h);
        } else {
            hi = (hi < 0.0 || h < hi) ? h : hi;
        }
        const double x = mq > 0.0 ? -g * (h / mq) : -2.0 * h;   // Newton step
        // Halley: x - x^2 g'' / (2 g'), g'' / g' = s2 / (h mq)
        const double y = x * ih, u = 0.5 * (double)s2 / mq;
        const double d = x * (1.0 - y * u);
        if (fabs(x) <= 2e-6 * h && h + d <= hsi && (it <= left || fabs(x) <= a.tol * h)) {
            // sum f at h + d: f + f' d + f'' d^2 / 2
            F = f + mq * (d * ih) * (1.0 + u * (d * ih));
            h += d;
            conv = true;
            break;
        }
        double hn = mq > 0.0 ? h + x : -1.0;
        if (hi < 0.0) {
            if (!(hn > lo) || hn > 2.0 * h) hn = 2.0 * h;
            if (hn > hsi) hn = hsi;
        } else if (!(hn > lo && hn < hi)) {
            hn = 0.5 * (lo + hi);
        }
        h = hn;
    }
    const bool lead = wk.lane == 0;
    if (fail) {
        if (lead) {
            a.hs[s] = hsi * search_growth(N, F, hsi, hguess);
            dens_fail(a, s);
        }
        return;
    }
    if (!conv) {
        if (lead) set_flag(a.cnt, ST_NOCONV_H);
        // sum f at the last h
        F = 0.0;
        for (int k = wk.lane; k < c; k += W) {
            const int j = idx[k];
            const double dx = fold64(a.xs[j] - xi, bx.L[0]);
            const double dy = fold64(a.ys[j] - yi, bx.L[1]);
            const double dz = fold64(a.zs[j] - zi, bx.L[2]);
            F += kernel_shape<double>(a.kernel, sqrt(dx * dx + dy * dy + dz * dz) / h);
        }
        F = wk.sum(F);
    }
    if (!lead) return;
    if (crad > 0.0) {
        a.nbr_cnt[s] = c;
        a.hs[s] = crad;
        if (!(h < crad)) {   // the root left the compacted radius: search again
            dens_fail(a, s);
            return;
        }
    }
    const double om = 1.0 / (kernel_norm<double>(a.kernel, h) * F);
    a.h[s] = h;
    a.om[s] = om;
    const Row<double> rr(rec, s);
    rr[R_H] = h;
    rr[R_OM] = om;
}

// ---------------------------------------------------------------- mixed path
// one particle's float Newton solve, then the double-float refinement
template <int W>
__device__ __forceinline__ void dens_one(const DensArgs &a, float *__restrict__ rec,
                                         const Walk<W> &wk, int64_t s) {
    if (s >= a.n) return;
    if (a.only_active && !(a.active[s] & 1)) return;
    const Box bx = a.boxes[a.pbox[s]];
    const Separation<float> sep(a, s, bx);
    const double hsi_d = a.hs[s];
    float hsi = (float)hsi_d;
    const float N = (float)(a.nngb ? a.nngb[s] : a.n_ngb);
    const int64_t o = a.nbr_off[s];
    int32_t *idx = a.nbr_idx + o;
    float h = (float)a.h[s];
    if (!(h > 0.f) || h > hsi) h = hsi;
    const float xmin = (float)(bx.Lmax * (1.0 / 65536.0));
    const NewtonF nf = newton_float<W>(a, sep, idx, a.nbr_cnt[s], h, hsi, N, xmin, a.max_iter, wk);
    const bool lead = wk.lane == 0;
    if (nf.fail) {   // (no compaction happened: failing needs h >= hsi, below any bracket)
        if (lead) {
            a.hs[s] = hsi_d * search_growth((double)N, (double)nf.kf, hsi_d, a.h[s]);
            dens_fail(a, s);
        }
        return;
    }
    if (!nf.conv && lead) set_flag(a.cnt, ST_NOCONV_H);
    h = nf.h;
    const float comp = nf.comp;
    const int c = nf.c;
    // one Newton step in double-float on exact 64-bit fixed-point separations
    const uint4 li = a.low[s];
    const float sx = (float)(bx.L[0] * 5.421010862427522e-20);  // L / 2^64
    const float sy = (float)(bx.L[1] * 5.421010862427522e-20);
    const float sz = (float)(bx.L[2] * 5.421010862427522e-20);
    df hd = {h, 0.f};
    df ih = df_div({1.f, 0.f}, hd);
    df F = {0.f, 0.f}, MQ = {0.f, 0.f};
    const float hcut = h * (1.f + 1e-5f);   // W = 0 beyond h: skip those (float r is good to 1e-7)
    const bool fin = a.compact && h > xmin && !nf.flat;
    const float keep = h * 1.0001f;
    int w = 0;
    for (int k0 = 0; k0 < c; k0 += W) {
        const int k = k0 + wk.lane;
        const bool in = W == 1 || k < c;
        const int j = in ? idx[k] : 0;
        const float rf = !in ? INFINITY : k < Walk<W>::CACHE ? wk.rs[k] : sep(j);
        if (fin) wk.keep(rf < keep, idx, j, rf, w);
        df fv = {0.f, 0.f}, mv = {0.f, 0.f};
        bool on = rf < hcut;
        if (on) {
            const uint4 pj = a.pos[j], lj = a.low[j];
            const long long ix = fixed_diff(pj.x, lj.x, sep.qx, li.x);
            const long long iy = fixed_diff(pj.y, lj.y, sep.qy, li.y);
            const long long iz = fixed_diff(pj.z, lj.z, sep.qz, li.z);
            df dx = df_mulf(from_i64(ix), sx);
            df dy = df_mulf(from_i64(iy), sy);
            df dz = df_mulf(from_i64(iz), sz);
            df r2 = df_add(df_add(df_mul(dx, dx), df_mul(dy, dy)), df_mul(dz, dz));
            df q = df_mul(df_sqrt(r2), ih);
            on = q.hi < 1.f;
            if (on) {
                df t = df_one_minus(q);
                df t2 = df_mul(t, t);
                if (a.kernel == 0) {
                    df t3 = df_mul(t2, t);
                    fv = df_mul(df_mul(t3, t), df_addf({4.f * q.hi, 4.f * q.lo}, 1.f));
                    mv = df_mulf(df_mul(df_mul(q, q), t3), 20.f);
                } else {
                    df q2 = df_mul(q, q);
                    if (q.hi <= 0.5f) {
                        fv = df_add(df_sub({1.f, 0.f}, df_mulf(q2, 6.f)), df_mulf(df_mul(q2, q), 6.f));
                        mv = df_sub(df_mulf(q2, 12.f), df_mulf(df_mul(q2, q), 18.f));
                    } else {
                        fv = df_mulf(df_mul(t2, t), 2.f);
                        mv = df_mulf(df_mul(q, t2), 6.f);
                    }
                }
            }
        }
        if (W == 1) {
            if (on) {
                F = df_add(F, fv);
                MQ = df_add(MQ, mv);
            }
        } else {
            // in the list's order
            for (unsigned m = __ballot_sync(0xffffffffu, on); m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                F = df_add(F, {__shfl_sync(0xffffffffu, fv.hi, l), __shfl_sync(0xffffffffu, fv.lo, l)});
                MQ = df_add(MQ, {__shfl_sync(0xffffffffu, mv.hi, l), __shfl_sync(0xffffffffu, mv.lo, l)});
            }
        }
    }
    if (!lead) return;
    // g = Kn F - N, dg = Kn MQ / h  ->  h_new = h - (F - N/Kn) h / MQ
    double Fd = (double)F.hi + (double)F.lo;
    double MQd = (double)MQ.hi + (double)MQ.lo;
    double hN = (double)h;
    double Kd = a.kernel == 0 ? 14.0 : 32.0 / 3.0;
    // (N_NGB in double: a guard round's grown 32 * 1.2^k is not a float)
    const double Nd = a.nngb ? a.nngb[s] : a.n_ngb;
    double hnew = MQd > 0.0 ? hN - (Fd - Nd / Kd) * hN / MQd : hN;
    if (fin || comp > 0.f) {
        // the compacted list is complete for r < crad
        const double crad = fin ? hN * (1.0 + 5e-5) : (double)comp;
        a.nbr_cnt[s] = fin ? w : c;
        a.hs[s] = crad;
        if (!(hnew < crad)) {
            // the refinement left the compacted radius (an unconverged float
            // root): search again from a rebuilt list
            dens_fail(a, s);
            return;
        }
    }
    // omega from the sum at h (first order in the small correction)
    // sum_j W(r, hnew) = norm(hnew) sum f(q_new); d/dh [h^3 sum W] = Kn MQ / h * 3/(4 pi)
    double normh = kernel_norm<double>(a.kernel, hnew);
    double fsum = Fd + (hnew - hN) * MQd / hN;   // first-order update of sum f(q)
    double om = 1.0 / (normh * fsum);
    a.h[s] = hnew;
    a.om[s] = om;
    const Row<float> rr(rec, s);
    rr[R_H] = (float)hnew;
    rr[R_OM] = (float)om;
}

// one thread per particle, in the sorted order (a partial solve too: its
// particles are often many and clustered, and a compacted list would scatter
// each warp's gathers over the box); the full solve ranks the CTA's 128
// particles by list length.  (Larger ranked tiles spread the repeated
// gathers of the Newton iterations over more of the Morton curve: slower.)
__device__ __forceinline__ int64_t dens_particle(const DensArgs &a) {
    if (!a.rank) return blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    __shared__ unsigned rank_key[RANK_THREADS];
    const int64_t base = blockIdx.x * (int64_t)RANK_THREADS;
    rank_tile(rank_key, 1, a.nbr_cnt, base, a.n);
    return base + rank_index(rank_key[threadIdx.x], 1);
}

__global__ void k_density_f64(DensArgs a, double *__restrict__ rec) {
    dens_one<1>(a, rec, Walk<1>{nullptr, 0}, dens_particle(a));
}

// Bound by the latency of the walk's gathers and by the L1 data stage they go
// through: 16-byte positions side by side in place of the records' first columns
// and of three 64-bit arrays, and 10 CTAs per SM (48 registers; 9: 2 % slower, 12:
// 2 % slower on the tube), took 1.95 -> 1.58 ms (2.10 M particles), 0.786 -> 0.653
// (1.07 M tube), 2.79 -> 2.23 (4 M log-normal).  Two to eight entries' loads in
// flight per thread cost more registers than they hide; so does cutting the
// list to the root before the refinement.
__global__ void __launch_bounds__(DENS_THREADS, 10) k_density_mixed(DensArgs a, float *__restrict__ rec) {
    dens_one<1>(a, rec, Walk<1>{nullptr, 0}, dens_particle(a));
}

// A guard round's re-solve: a warp per particle of the round's guard list.
// The particles are few (0.4 % of a log-normal box in the first round, fewer
// later) and their lists long, so a thread each leaves most of the GPU idle
// behind one serial walk (gradient stage of a 4 M log-normal box, which holds
// the rounds: 7.15 -> 5.79 ms; 300k in FP64 9.5 -> 6.3 ms).
template <typename R>
__global__ void __launch_bounds__(DENS_THREADS)
k_density_list(DensArgs a, R *__restrict__ rec) {
    __shared__ float rs[DENS_THREADS / 32][DENS_CACHE];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Walk<32> wk{rs[warp], lane};
    const int nl = a.list ? *a.nlist : a.buckets ? a.nbuckets * BUCKET : (int)a.n;
    for (int t = blockIdx.x * (DENS_THREADS / 32) + warp; t < nl; t += gridDim.x * (DENS_THREADS / 32)) {
        int64_t s = t;
        if (a.list) {
            s = a.list[t];
        } else if (a.buckets) {
            const int b = a.buckets[t / BUCKET], k = t % BUCKET;
            if (k >= a.node_cnt[b]) continue;
            s = a.node_first[b] + k;
        }
        __syncwarp();
        dens_one<32>(a, rec, wk, s);
    }
}

// the search radius of particles whose root lay beyond it, as the density
// kernel grew it (not below margin h); never beyond half the shortest box
// side (one periodic image)
// (list non-NULL: only its *nlist particles -- a guard round's, the only
// ones it solves; every other particle's flags are clear then)
__global__ void k_grow_search(int64_t n, uint8_t *__restrict__ active, double *__restrict__ hs,
                              const double *__restrict__ h, double margin,
                              const int32_t *__restrict__ pbox, const Box *__restrict__ boxes,
                              const int32_t *__restrict__ list, const int *__restrict__ nlist) {
    const int64_t cnt = list ? (int64_t)*nlist : n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cnt;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = list ? list[t] : t;
        const uint8_t a = active[s];
        if (a & 2) {
            const Box bx = boxes[pbox[s]];
            double half = 0.5 * fmin(bx.L[0], fmin(bx.L[1], bx.L[2]));
            hs[s] = fmin(fmax(hs[s], h[s] * margin), half);   // (grown by the density kernel)
            active[s] = (a & ACT_GUARD) | 1;
        } else {
            active[s] = a & ACT_GUARD;
        }
    }
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t run_density(hydro_ctx *c, bool only_active, bool compact, stream_t st, bool guard) {
    const int64_t n = c->plan.n;
    DensArgs a;
    a.n = n;
    a.nbr_off = c->d_nbr_off.get();
    a.nbr_cnt = c->d_nbr_cnt.get();
    a.nbr_idx = c->d_nbr_idx.get();
    a.hs = c->d_hs.get();
    a.xs = c->d_xs.get(); a.ys = c->d_ys.get(); a.zs = c->d_zs.get();
    a.qx = c->d_qx.get(); a.qy = c->d_qy.get(); a.qz = c->d_qz.get();
    a.pbox = c->d_pbox.get();
    a.boxes = c->d_boxes.get();
    a.active = c->d_active.get();
    a.nngb = c->d_nngb.get();
    a.n_ngb = c->cfg.n_ngb;
    a.kernel = c->cfg.kernel;
    a.tol = c->cfg.h_tol;
    a.max_iter = c->cfg.max_h_iter;
    a.only_active = only_active;
    a.compact = compact;
    a.h = c->d_hsorted.get();
    a.om = c->d_omsorted.get();
    a.cnt = c->d_cnt;
    // ranked when the gradient kernel ranks (the same divergence)
    a.rank = c->grad_rank && !only_active;
    a.list = c->d_guard_idx.get();
    a.nlist = &c->d_cnt->nguard;
    HYD_CUDA(cudaMemsetAsync(&c->d_cnt->search_fail, 0, sizeof(int), st));
    // a warp per particle: the guard round's list, or every particle of a set
    // so small that a thread each would leave the GPU idle, also that of the few
    // buckets of a sparse sub-step of individual timesteps, which hold all its
    // starting particles (us a sub-step with a thread for each of all particles,
    // with these warps over all particles, over the buckets: 48^3 422, 387, 381;
    // 128^3 1273, 1345, 1223; 200^3 4029, 4406, 3960)
    const bool listed = guard && only_active;
    const bool sparse = c->rung_live && only_active && c->rung_touch_n >= 0 &&
                        c->rung_touch_n * BUCKET <= DENS_WARP_MAX;
    const bool warps = listed || sparse || n <= DENS_WARP_MAX;
    if (!listed) a.list = nullptr;
    a.buckets = sparse && !listed ? c->d_touch.get() : nullptr;
    a.nbuckets = a.buckets ? (int)c->rung_touch_n : 0;
    a.node_first = c->d_node_first.get();
    a.node_cnt = c->d_node_cnt.get();
    const int64_t np = a.buckets ? (int64_t)a.nbuckets * BUCKET : n;
    const unsigned grid = !warps ? grid_for(n, DENS_THREADS)
        : listed ? 152u * 8u : std::min(152u * 8u, grid_for(np * 32, DENS_THREADS));
    if (c->cfg.precision == HYDRO_MIXED) {
        a.pos = c->d_pos.get();   // (gather_state)
        a.low = c->d_low.get();
        if (warps) k_density_list<float><<<grid, DENS_THREADS, 0, st>>>(a, c->d_recf.get());
        else k_density_mixed<<<grid, DENS_THREADS, 0, st>>>(a, c->d_recf.get());
    } else if (warps) {
        k_density_list<double><<<grid, DENS_THREADS, 0, st>>>(a, c->d_recd.get());
    } else {
        k_density_f64<<<grid, DENS_THREADS, 0, st>>>(a, c->d_recd.get());
    }
    return launch_check();
}

cudaError_t grow_search_radius(hydro_ctx *c, stream_t st, bool guard) {
    const int64_t n = c->plan.n;
    k_grow_search<<<guard ? 152 * 4 : grid_for(n, 256), 256, 0, st>>>(
        n, c->d_active.get(), c->d_hs.get(), c->d_hsorted.get(), c->cfg.search_margin,
        c->d_pbox.get(), c->d_boxes.get(), guard ? c->d_guard_idx.get() : nullptr,
        &c->d_cnt->nguard);
    return launch_check();
}

}  // namespace hyd
