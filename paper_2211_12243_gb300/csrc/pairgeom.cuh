// Pair geometry shared by the pair kernels: separation of two particles
// from their records, and exact membership r_ij < h.
#pragma once

#include "fp64.cuh"
#include "hydro_internal.cuh"
#include "row.cuh"

namespace hyd {

// separation from the first three slots
__device__ __forceinline__ void rec_sep(const double *ri, const double *rj, const Box &bx,
                                        double d[3], double &r2) {
    d[0] = fold64(__dsub_rn(rj[0], ri[0]), bx.L[0]);
    d[1] = fold64(__dsub_rn(rj[1], ri[1]), bx.L[1]);
    d[2] = fold64(__dsub_rn(rj[2], ri[2]), bx.L[2]);
    r2 = r2_exact(d[0], d[1], d[2]);
}

__device__ __forceinline__ void rec_sep(const float *ri, const float *rj, const Box &bx,
                                        float d[3], float &r2) {
    d[0] = qdiff(__float_as_uint(ri[0]), __float_as_uint(rj[0]), bx.s[0]);
    d[1] = qdiff(__float_as_uint(ri[1]), __float_as_uint(rj[1]), bx.s[1]);
    d[2] = qdiff(__float_as_uint(ri[2]), __float_as_uint(rj[2]), bx.s[2]);
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
}

// the arrays an exact membership test reads
struct Exact {
    const double *xs, *ys, *zs, *h;
    const int32_t *pbox;
    const Box *boxes;
};

// r_ij^2 < h_k^2 as the definition states it in double (minimum image folded
// once, (dx^2 + dy^2) + dz^2, each step rounded).  Out of line and from memory:
// a float separation decides all but a few pairs, and the operands in double
// would cost the pair kernels some thirty registers.
static __device__ __noinline__ bool member_exact(Exact a, int i, int j, int k) {
    const Box *b = a.boxes + a.pbox[i];
    const double ex = fold64(__dsub_rn(a.xs[j], a.xs[i]), b->L[0]);
    const double ey = fold64(__dsub_rn(a.ys[j], a.ys[i]), b->L[1]);
    const double ez = fold64(__dsub_rn(a.zs[j], a.zs[i]), b->L[2]);
    const double h = a.h[k];
    return r2_exact(ex, ey, ez) < __dmul_rn(h, h);
}

// The smallest radius that the float band (1e-4 of its square) decides: L / 4096
// with L the longest side, from the sides' units 2^-32 L.
__device__ __forceinline__ float band_radius(const Box &b) {
    return fmaxf(b.s[0], fmaxf(b.s[1], b.s[2])) * 1048576.0f;
}

// Membership r_ij < h_i of particle i's pairs.
template <typename R>
struct Member;
template <>
struct Member<float> {
    float lo2, hi2;     // float band around h^2 (empty when h is tiny vs L)
    __device__ __forceinline__ void init(double h, const Box &b) {
        float hf = (float)h;
        lo2 = hf * hf * (1.0f - 1e-4f);
        hi2 = hf * hf * (1.0f + 1e-4f);
        // fixed-point separations are exact to L/2^32, L the longest side; below
        // h = L/4096 the float band would no longer be conservative, so decide
        // every pair in double there
        if (hf < band_radius(b)) { lo2 = -1.0f; hi2 = 3.0e38f; }
    }
    // r2 from the fixed-point separation
    __device__ __forceinline__ bool operator()(const Exact &a, float r2, int i, int j) const {
        if (r2 < lo2) return true;
        if (r2 > hi2) return false;
        return member_exact(a, i, j, i);
    }
};
// h^2 for comparisons of bits (dlt_pos): no distance is below that of a NaN
__device__ __forceinline__ double radius2(double h) {
    const double h2 = __dmul_rn(h, h);
    return dhi(h2) <= 0x7ff00000u ? h2 : 0.0;
}
template <>
struct Member<double> {
    double h2;
    __device__ __forceinline__ void init(double h, const Box &) { h2 = radius2(h); }
    // r2 is already the exact value (r2, h2 >= 0)
    __device__ __forceinline__ bool operator()(const Exact &, double r2, int, int) const {
        return dlt_pos(r2, h2);
    }
};

}  // namespace hyd
