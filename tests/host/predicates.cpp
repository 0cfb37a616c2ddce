// Host build of the geometric predicates of lbm_device.cuh: how often the
// FP32-filtered form decides differently from the FP64 definition.
#include "device_shim.h"

#include "lbm_launch.h"

#include <random>

using namespace lbmgpu;

// Cells at the faces of an n^3 periodic box, their centres within twice the
// filter's margin of the surface of a sphere across those faces.  out[0]:
// cells whose inside / outside decision differs; out[1]: cells whose count of
// 4^3 samples differs from the FP64 count.
extern "C" void filter_mismatches(int n, double D, int trials, unsigned seed, long long out[2]) {
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    Geom g{};
    g.nx = g.ny = g.nz = n;
    set_tiles(g, LBM_STORE_F64);
    out[0] = out[1] = 0;
    const double r = 0.5 * D, band = 2.0 * margin_f((float)r) / r;
    for (int t = 0; t < trials; ++t) {
        DevParticle P{};
        P.d = D;
        P.r = r;
        double v[3], len = 0.0;
        for (int a = 0; a < 3; ++a) {
            v[a] = U(rng) - 0.5;
            len += v[a] * v[a];
        }
        const double d = (r + (U(rng) - 0.5) * band) / std::sqrt(len);
        int c[3];
        for (int a = 0; a < 3; ++a) {
            c[a] = v[a] > 0 ? (int)(U(rng) * 2) : n - 1 - (int)(U(rng) * 2);
            const double x = c[a] + 0.5 - d * v[a];
            P.x[a] = x < 0 ? x + n : (x >= n ? x - n : x);
        }
        store_region(g, P);
        out[0] += cell_inside(g, P, c[0], c[1], c[2]) !=
                  point_inside(g, P, c[0] + 0.5, c[1] + 0.5, c[2] + 0.5);
        const CellOffset co = cell_offset(g, P, c[0], c[1], c[2]);
        int count = solid_count_quick(P, co, 4);
        if (count < 0) {
            count = 0;
            for (int lane = 0; lane < 32; ++lane)
                count += solid_count_warp(g, P, co, c[0], c[1], c[2], 4, lane);
        }
        out[1] += count != solid_count(g, P, c[0], c[1], c[2], 4);
    }
}
