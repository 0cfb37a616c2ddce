// Host build of the FP64 fluid collision (lbm_fixed.cuh, collide_fluid of
// lbm_device.cuh) against exact arithmetic.
#include "device_shim.h"

#include "lbm_launch.h"

#include <random>

using namespace lbmgpu;
typedef _Float128 real;

// Largest distance, in units of the last place, of the product by a constant from a
// K 2^-64 (K the stored constant), over operands across the range.
extern "C" double constant_product_error(double c, int trials, unsigned seed) {
    std::mt19937_64 rng(seed);
    const FixMul m = make_fix_mul(c);
    const unsigned long long K = (unsigned long long)m.hi << 32 | m.lo;
    double worst = 0.0;
    for (int t = 0; t < trials; ++t) {
        const long long a = (long long)rng() >> 2;  // [-2^61, 2^61)
        const __int128 d = ((__int128)fix_mul(a, m) << 64) - (__int128)a * (__int128)K;
        worst = std::max(worst, std::fabs(std::ldexp((double)d, -64)));
    }
    return worst;
}

// The same for the product of two variables, |a b 2^-64| < 2^58.
extern "C" double variable_product_error(int trials, unsigned seed) {
    std::mt19937_64 rng(seed);
    double worst = 0.0;
    for (int t = 0; t < trials; ++t) {
        const long long a = (long long)rng() >> 2, b = (long long)rng() >> 4;
        const __int128 d = ((__int128)fix_mul(fix_split(a), fix_split(b)) << 64) - (__int128)a * b;
        worst = std::max(worst, std::fabs(std::ldexp((double)d, -64)));
    }
    return worst;
}

// Collides `trials` cells: populations rho0 w_q (1 + drift 3 c_q.u) (1 + noise U(-1, 1)).
// out: cells taken by the fixed point; squared error and squared reference summed
// over those cells, for the fixed-point and the FP64 form; the largest error over the
// cell's largest population of each; cells whose fixed-point error is the larger.
extern "C" void collision_errors(double tau, double lm, double rho0, const double* fext,
                                 double noise, double drift, int trials, unsigned seed,
                                 double out[7]) {
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    const double lp = -1.0 / tau;
    const Coll<double> k = make_coll<double>(lp, lm, rho0, fext);
    for (int i = 0; i < 7; ++i) out[i] = 0.0;
    if (!k.fix.on) return;
    for (int t = 0; t < trials; ++t) {
        const double u[3] = {drift * U(rng), drift * U(rng), drift * U(rng)};
        double f[NQ], fx[NQ], fd[NQ], fmax = 0.0;
        for (int q = 0; q < NQ; ++q) {
            const double cu = cx(q) * u[0] + cy(q) * u[1] + cz(q) * u[2];
            f[q] = fx[q] = fd[q] = rho0 * wq(q) * (1.0 + 3.0 * cu) * (1.0 + noise * U(rng));
            fmax = std::max(fmax, std::fabs(f[q]));
        }
        if (!(k.has_force ? fixed_collide_t<true>(fx, k.fix) : fixed_collide_t<false>(fx, k.fix))) {
            for (int q = 0; q < NQ; ++q)
                if (fx[q] != f[q]) out[0] = -1e300;  // a refused cell comes back as it was
            continue;
        }
        collide_fluid(fd, k);
        real rho = 0, j[3] = {0, 0, 0};
        for (int q = 0; q < NQ; ++q) {
            rho += f[q];
            j[0] += (real)f[q] * cx(q);
            j[1] += (real)f[q] * cy(q);
            j[2] += (real)f[q] * cz(q);
        }
        real v[3];
        for (int a = 0; a < 3; ++a) v[a] = j[a] / (real)rho0;
        const real uu = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        const real uf = v[0] * (real)fext[0] + v[1] * (real)fext[1] + v[2] * (real)fext[2];
        real ex = 0, ed = 0;
        for (int q = 0; q < NQ; ++q) {
            const int p = opp(q);
            const real w = q == 0 ? (real)1 / 3 : (q <= 6 ? (real)1 / 18 : (real)1 / 36);
            const real cu = cx(q) * v[0] + cy(q) * v[1] + cz(q) * v[2];
            const real cf = cx(q) * (real)fext[0] + cy(q) * (real)fext[1] + cz(q) * (real)fext[2];
            const real sp = ((real)f[q] + f[p]) / 2, sm = ((real)f[q] - f[p]) / 2;
            const real ep = w * (rho + (real)rho0 * ((real)4.5 * cu * cu - (real)1.5 * uu));
            const real em = w * (real)rho0 * 3 * cu;
            const real F = w * (3 * cf + 9 * cu * cf - 3 * uf);
            const real g = (real)f[q] + (real)lp * (sp - ep) + (real)lm * (sm - em) + F;
            const real a = (real)fx[q] - g, b = (real)fd[q] - g;
            ex += a * a;
            ed += b * b;
            out[3] += (double)(g * g);
            out[4] = std::max(out[4], std::fabs((double)a) / fmax);
            out[5] = std::max(out[5], std::fabs((double)b) / fmax);
        }
        out[0] += 1.0;
        out[1] += (double)ex;
        out[2] += (double)ed;
        out[6] += ex > ed;
    }
}

// Whether a storage mode collides in fixed point at tau.
extern "C" int fixed_point_on(int storage, double tau) {
    const double fe[3] = {0.0, 0.0, 0.0};
    return make_coll_f64(storage, -1.0 / tau, -1.0 / tau, 1.0, fe).fix.on;
}
