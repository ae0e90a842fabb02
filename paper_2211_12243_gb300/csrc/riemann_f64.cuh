// The Riemann solvers of the FP64 flux kernel: the problems, formulae and
// accuracy of riemann.cuh (Toro 2009, ch. 4 and 10), arranged to issue few
// FP64 instructions (fp64.cuh says why those alone count).
//
// Exact solver: the star pressure is iterated in float first, which leaves a
// relative error of about 1e-6, and finished in FP64 by a third-order
// (Halley) step: the pressure function and its derivative in FP64 once per
// side, the second derivative, which only scales the square of the step, in
// float.  A step below 3e-6 relative leaves an error below 1e-16; a larger one
// is followed by another.  Before, the FP64 iteration started from Toro's
// guess and took four to five evaluations to its 1e-12 and two more.  A
// rarefaction's power (p/p_K)^z is formed from the float power t0 by
// (1 + w)^z = 1 + z w + ... with w = (p/p_K) t0^(-1/z) - 1, w small, where 1/z is
// an integer; other gammas take pow().
//
// Flux kernel of the 1.07 M tube (MFM) 56.4 -> 12.5 ms, of a 300k log-normal box
// (MFV) 27.2 -> 4.9 ms, the sums' rounding errors (add_error) included; it keeps
// the FP64 pipe busy for 68-80 % of the time, and a third CTA per SM gains nothing.
#pragma once

#include "riemann.cuh"

namespace hyd {

// the iteration of riemann.cuh for what the fast path does not settle
// (states beyond the float range, no convergence): out of line, rarely run
static __device__ __noinline__ int star_solve_plain(const GasK<double> &k, double rl, double ul,
                                                    double pl, double cl, double rr, double ur,
                                                    double pr, double cr, double tol,
                                                    int max_newton, double *ps, double *us) {
    double p, u;
    const StarOut o = star_solve<double>(k, rl, ul, pl, cl, rr, ur, pr, cr, -1.0, tol, max_newton,
                                         p, u);
    *ps = p;
    *us = u;
    return o.iters;
}

// (p/pk)^z - 1, from the float power t0f of the float ratio
__device__ __forceinline__ double pow_z_m1(const GasK<double> &k, double p, double pk, float t0f) {
    if (k.nz > 0) {
        const double t0 = widen(t0f);
        const double tp = ipow64(t0, k.nz) * pk;
        const double w = (p - tp) * rcp40(tp);
        if ((dbits(w) & 0x7fffffffffffffffll) < 0x3f1a36e2eb1c432dll) {   // |w| < 1e-4
            const double s = w * fma(w, fma(w, k.c3, k.c2), k.z);
            return fma(t0, s, t0 - 1.0);
        }
    }
    return pow(p / pk, k.z) - 1.0;
}

// f_K(p) and f_K'(p) in FP64 (ip = 1/p); in float the derivative dff, which
// weighs the sides, and the curvature kap = p f'' / f'
__device__ __forceinline__ void side_eval64(const GasK<double> &k, const GasK<float> &kf, double rk,
                                            double pk, double ck, const SideF &sf, double p,
                                            double ip, float pf, float ipf, double &f, double &df,
                                            float &dff, float &kap) {
    const double d = p - pk;
    if (dpos(d)) {
        const double rk5 = rk * k.ig5;
        const double q = rsqrt64(rk5 * fma(k.g6, pk, p));   // sqrt(A / (p + B))
        const double hd = 0.5 * d * (q * q * rk5);          // (p - p_K) / (2 (p + B))
        f = d * q;
        df = fma(-q, hd, q);
        const float rq = rsqrtf(pf + sf.B);
        const float ia = rq * rq;
        const float dia = (pf - sf.pk) * ia, h = 1.f - 0.5f * dia;
        dff = sf.sA * rq * h;
        kap = pf * ia * __fdividef(0.75f * dia - 1.f, h);
    } else {
        const float t0f = __powf(pf * sf.ipk, kf.z);
        const double tm1 = pow_z_m1(k, p, pk, t0f);
        const double cg = ck * k.inv_g;
        f = k.g4 * ck * tm1;
        df = fma(cg, tm1, cg) * ip;
        dff = t0f * sf.cg * ipf;
        kap = kf.z - 1.f;
    }
}

// p* and u* of the exact problem (vacuum set when the sides part)
__device__ __forceinline__ StarOut star_solve64(const GasK<double> &k, const GasK<float> &kf,
                                                double rl, double ul, double pl, double cl,
                                                double rr, double ur, double pr, double cr,
                                                double tol, int max_newton, double &ps, double &us) {
    StarOut o{0, 0, 0};
    const double du = ur - ul;
    // (compared in FP64: states that are not numbers are no vacuum, and zeros of
    // either sign at zero sound speeds are one)
    if (k.g4 * (cl + cr) <= du) {
        o.vacuum = 1;
        ps = us = 0.0;
        return o;
    }
    // float start
    const float rlf = narrow(rl), plf = narrow(pl), rrf = narrow(rr), prf = narrow(pr);
    const float ulf = narrow(ul), urf = narrow(ur);
    const float clf = narrow(cl), crf = narrow(cr), duf = narrow(du);
    const SideF fl_ = side_prep(kf, rlf, plf, clf), fr_ = side_prep(kf, rrf, prf, crf);
    float pf = star_guess<float>(kf, rlf, ulf, plf, clf, rrf, urf, prf, crf);
    if (!(pf > 1e-37f)) pf = 1e-37f;
    int it = 0;
    for (; it < 12; it++) {
        float a, da, b, db;
        const float ip = __fdividef(1.f, pf);
        side_eval(kf, fl_, pf, ip, a, da);
        side_eval(kf, fr_, pf, ip, b, db);
        float pn = pf - __fdividef(a + b + duf, da + db);
        if (!(pn > 1e-37f)) pn = 1e-37f;
        const bool done = fabsf(pn - pf) < 5e-4f * pn;   // (the step squares the error)
        pf = pn;
        if (done) break;
    }
    // FP64 finish (a float start out of range or not converged, and a state without
    // a sound speed, whose float root is 0 and not NaN: the plain path)
    if (pf > 1e-30f && pf < 1e30f && it < 12 && clf >= 0.f && crf >= 0.f) {
        double p = widen(pf);
        for (int n = 1; n <= 4; n++) {
            const double ip = rcp40(p);
            const float ipf = __fdividef(1.f, pf);
            double fl, dfl, fr, dfr;
            float wl, wr, kl, kr;
            side_eval64(k, kf, rl, pl, cl, fl_, p, ip, pf, ipf, fl, dfl, wl, kl);
            side_eval64(k, kf, rr, pr, cr, fr_, p, ip, pf, ipf, fr, dfr, wr, kr);
            const double D = dfl + dfr, N = -((fl + fr) + du) * rcp40(D);
            // Halley: N (1 - N f'' / (2 f')), with p f'' / f' the weighted mean
            // of the sides' curvatures
            const float iw = __fdividef(1.f, wl + wr), x = narrow(N) * ipf;
            const double step = fma(N, widen(-0.5f * x * (wl * kl + wr * kr) * iw), N);
            p += step;
            // (densities beyond the float range leave no weights for the curvatures
            // and the step is not a number or infinite: the plain path)
            if (!dnormal(p)) break;
            if (fabsf(x) < 3e-6f) {
                ps = p;
                const double h = fma(dfr - dfl, step, fr - fl) +
                                 widen(0.5f * x * (wr * kr - wl * kl) * iw) * (D * step);
                us = 0.5 * ((ul + ur) + h);
                o.iters = it + 1 + n;
                return o;
            }
            pf = narrow(p);
        }
    }
    o.iters = star_solve_plain(k, rl, ul, pl, cl, rr, ur, pr, cr, tol, max_newton, &ps, &us);
    return o;
}

// the state at x/t = 0 (star_sample of riemann.cuh, which says how the sides
// share a branch tree).  Behind a rarefaction rho* = rho_K (c* / c_K)^(2/(g-1)).
__device__ __forceinline__ void star_sample64(const GasK<double> &k, const GasK<float> &kf,
                                              double rl, double ul, double pl, double cl, double rr,
                                              double ur, double pr, double cr, double ps, double us,
                                              double &rho, double &u, double &p, int &side) {
    const bool left = dge0(us);   // (a speed that is not a number: right)
    side = left ? -1 : 1;
    const double rK = left ? rl : rr, pK = left ? pl : pr, cK = left ? cl : cr;
    const double uK = left ? ul : -ur, uS = left ? us : -us;
    double rs = rK, vs = uK, qs = pK;
    if (dlt(pK, ps)) {
        // shock: the pre-shock state beyond it (u_K >= c_K sqrt(g2 p*/p_K + z)),
        // else the star state
        const double t = ps * rcp64(pK);
        if (!dpos(uK) || dlt_pos(uK * uK, cK * cK * fma(k.g2, t, k.z))) {
            rs = rK * ((t + k.g6) * rcp64(fma(k.g6, t, 1.0)));
            vs = uS;
            qs = ps;
        }
    } else if (!dge0(uK - cK)) {   // (else beyond the rarefaction's head)
        double tz;
        if (k.nz > 0) {
            tz = 1.0 + pow_z_m1(k, ps, pK, __powf(__fdividef(narrow(ps), narrow(pK)), kf.z));
        } else {
            tz = pow(ps / pK, k.z);
        }
        const double cm = cK * tz;
        // (a right side keeps its tail point in the star region)
        const double e = uS - cm;
        const bool star = dneg(e) || (!left && dzero(e));
        if (star) {
            rs = rK * (k.n4 > 0 ? ipow64(tz, k.n4) : pow(ps / pK, k.inv_g));
            vs = uS;
            qs = ps;
        } else {
            // inside the fan
            const double cc = k.g5 + k.g6 * uK * rcp64(cK);
            const double c4 = k.n4 > 0 && dge0(cc) ? ipow64(cc, k.n4) : pow(cc, k.g4);
            rs = rK * c4;
            vs = k.g5 * (cK + 0.5 * k.gm1 * uK);
            qs = pK * (c4 * cc * cc);   // cc^(2g/(g-1)) = cc^(2/(g-1)) cc^2
        }
    }
    rho = rs;
    u = left ? vs : -vs;
    p = qs;
}

// HLLC flux along n (hllc_flux of riemann.cuh): the side that the contact
// leaves at x/t = 0 is selected first, so one path serves both
template <bool CONTACT_ONLY>
__device__ __forceinline__ void hllc_flux64(const GasK<double> &k, double rl, double ul, double pl,
                                            const double *wl, double rr, double ur, double pr,
                                            const double *wr, const double *n, double *F,
                                            double &ps, double &ss) {
    const double irl = rcp64(rl), irr = rcp64(rr);
    const double cl = sqrt64(k.g * pl * irl), cr = sqrt64(k.g * pr * irr);
    double ppv = 0.5 * (pl + pr) - 0.125 * (ur - ul) * (rl + rr) * (cl + cr);
    ppv = dpos(ppv) ? ppv : 0.0;
    const double ql = dlt_pos(dabs_(pl), ppv) ? sqrt64(1.0 + k.g2 * fma(ppv, rcp64(pl), -1.0)) : 1.0;
    const double qr = dlt_pos(dabs_(pr), ppv) ? sqrt64(1.0 + k.g2 * fma(ppv, rcp64(pr), -1.0)) : 1.0;
    const double sl = ul - cl * ql, sr = ur + cr * qr;
    const double al = rl * (sl - ul), ar = rr * (sr - ur);
    ss = (pr - pl + al * ul - ar * ur) * rcp64(al - ar);
    ps = fma(al, ss - ul, pl);
    if (CONTACT_ONLY) return;
    // (speeds that are not numbers select as in hllc_flux)
    const bool left = dge0(sl) || dge0(ss);
    const double r = left ? rl : rr, u = left ? ul : ur, p = left ? pl : pr;
    const double ir = left ? irl : irr, s = left ? sl : sr, al_ = left ? al : ar;
    const double w0 = left ? wl[0] : wr[0], w1 = left ? wl[1] : wr[1], w2 = left ? wl[2] : wr[2];
    const double E = 0.5 * fma(r, fma(u, u, fma(w0, w0, fma(w1, w1, w2 * w2))), k.g4 * p);
    double fm = r * u, fn = fma(fm, u, p), fe = u * (E + p);
    // between the outer waves (s and the contact on either side of x/t = 0)
    if (left ? !dge0(sl) : dge0(sr)) {
        const double kk = al_ * rcp64(s - ss);
        const double e2 = kk * fma(ss - u, ss + p * rcp64(al_), E * ir);
        fn = fma(s, fma(kk, ss, -fm), fn);
        fm = fma(s, kk - r, fm);
        fe = fma(s, e2 - E, fe);
    }
    F[0] = fm;
    F[1] = fma(fn, n[0], fm * w0);
    F[2] = fma(fn, n[1], fm * w1);
    F[3] = fma(fn, n[2], fm * w2);
    F[4] = fe;
}

}  // namespace hyd
