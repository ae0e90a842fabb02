// Test build (tests/test_gpu_fp64_pieces.py): the FP64 arithmetic of fp64.cuh and
// the solvers of riemann_f64.cuh on arrays, beside CUDA's own operations and the
// general solvers of riemann.cuh.
#include "riemann_f64.cuh"

using namespace hyd;

namespace {

__global__ void k_arith(int op, int n, const double *a, const double *b, double *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = a[i], y = b[i];
    switch (op) {
    case 0: out[i] = rcp64(x); break;
    case 1: out[i] = rcp40(x); break;
    case 2: out[i] = rsqrt64(x); break;
    case 3: out[i] = sqrt64(x); break;
    case 4: out[i] = div1(x, y, rcp64(y)); break;
    case 5: out[i] = div2(x, y, rcp64(y)); break;
    case 6: out[i] = div2(x, y, 1.0 / y); break;
    case 7: out[i] = __longlong_as_double((long long)fixed64(x)); break;
    }
}

// states [6][n]: rho, u, p of either side; out [2][8][n]: fast and general p*, u*,
// vacuum, the sampled rho, u, p, and HLLC's star pressure and contact speed;
// flux [2][5][n]: HLLC's flux
__global__ void k_solve(int n, double gamma, const double *s, double *out, double *flux) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const GasK<double> K(gamma);
    const GasK<float> Kf(gamma);
    const double rl = s[i], ul = s[n + i], pl = s[2 * n + i], rr = s[3 * n + i], ur = s[4 * n + i],
                 pr = s[5 * n + i];
    const double wl[3] = {0.0, 0.1 * ul, 0.0}, wr[3] = {0.0, 0.1 * ur, 0.0}, nh[3] = {1.0, 0.0, 0.0};
    for (int v = 0; v < 2; v++) {
        double ps, us, rho = 0, u = 0, p = 0, hps, hss, F[5];
        int side;
        StarOut o;
        if (v == 0) {
            const double cl = sqrt64(K.g * pl * rcp64(rl)), cr = sqrt64(K.g * pr * rcp64(rr));
            o = star_solve64(K, Kf, rl, ul, pl, cl, rr, ur, pr, cr, 1e-12, 100, ps, us);
            if (!o.vacuum)
                star_sample64(K, Kf, rl, ul, pl, cl, rr, ur, pr, cr, ps, us, rho, u, p, side);
            hllc_flux64<false>(K, rl, ul, pl, wl, rr, ur, pr, wr, nh, F, hps, hss);
        } else {
            const double cl = sqrt(K.g * pl / rl), cr = sqrt(K.g * pr / rr);
            o = star_solve<double>(K, rl, ul, pl, cl, rr, ur, pr, cr, -1.0, 1e-12, 100, ps, us);
            if (!o.vacuum)
                star_sample<double>(K, rl, ul, pl, cl, rr, ur, pr, cr, ps, us, rho, u, p, side);
            hllc_flux<double>(K, rl, ul, pl, wl, rr, ur, pr, wr, nh, F, hps, hss);
        }
        const double r[8] = {ps, us, (double)o.vacuum, rho, u, p, hps, hss};
        for (int q = 0; q < 8; q++) out[(int64_t)(8 * v + q) * n + i] = r[q];
        for (int q = 0; q < 5; q++) flux[(int64_t)(5 * v + q) * n + i] = F[q];
    }
}

}  // namespace

extern "C" int probe_arith(int op, int n, const double *a, const double *b, double *out) {
    k_arith<<<(n + 255) / 256, 256>>>(op, n, a, b, out);
    return (int)cudaDeviceSynchronize();
}

extern "C" int probe_solve(int n, double gamma, const double *s, double *out, double *flux) {
    k_solve<<<(n + 127) / 128, 128>>>(n, gamma, s, out, flux);
    return (int)cudaDeviceSynchronize();
}
