// Fluid collision of FP64 populations on the integer pipes (sm_103a).
//
// GB300 issues 2 FP64 lane-operations per SM per cycle against 128 integer
// ones, so the ~124 FP64 operations of a cell's collision hold the FP64 sweep
// at 0.19 of the HBM bandwidth.  Populations, densities and velocities have a
// modest range, so the collision runs in 64-bit fixed point instead:
//   value    signed 64-bit integer, unit 2^-58 of 2^sh, where 2^sh is the
//            power of two nearest to rho0 (the collision is homogeneous in f,
//            rho0 and f_ext, so any rho0 is handled alike);
//   FP64 in  exact: only populations in [2^-6, 1) 2^sh take this path, and
//            their 53-bit significands fit above the unit;
//   + and -  exact;
//   *        high half of the 128-bit product from 32-bit limbs, rounded to
//            nearest, the low x low limb product replaced by its mean:
//            unbiased, within 1 unit of the product by the stored constant,
//            within 3/4 of a unit of that of two variables (below);
//   FP64 out the hardware conversion (round to nearest even), exponent moved.
// A population of a diagonal direction at rest, 1/36, has its last FP64 bit
// at 2^-58 too; every FP64 operation on rho or j (~1) rounds at 2^-53.  The
// result is therefore closer to exact arithmetic than the FP64 form's over the
// cells of a flow: collided populations against 113-bit arithmetic, tau = 0.6,
// relative 2-norm, 5.2e-17 (FP64 form 1.9e-16; the correctly rounded result has
// 4.6e-17), largest error 1.0e-16 of max f (6.8e-16), mean mass error per cell
// 1e-19 (3e-17), and likewise with a force, BGK, rho0 1.37 and 1000.  The FP64
// form's error falls as tau grows, to this one's near tau = 6 (FIX_TAU_MAX stays
// below that), and single cells may have the larger error here (0.1 % at tau =
// 0.6, 14 % at tau = 1 with BGK).  A cell with any population outside the
// range (negative, below 2^-6, more than ~2 to 4 times its rest value,
// non-finite) or |j| >= rho0/4 is left to the FP64 form (collide_cell), which
// also reports bad densities.
//
// The collision is arranged for few products, each by a constant:
//   f_q'    = f_q    - e - o,   f_qbar' = f_qbar - e + o  with
//   e = |l+| (f_q^+ - f_q^eq,+) - F_q^+ = |l+|/72 (36 s - 2 base - 9 (c.j)^2/rho0 + ..)
//   o = |l-| (f_q^- - f_q^eq,-) - F_q^- = |l-|/12 (6 d - c.j) - F_q^-
// for a diagonal pair (s, d = f_q +- f_qbar, base = rho - 3/2 j.j/rho0), half
// the integer factors and twice the constants for an axis pair: 19 constant
// products and 6 (9 for rho0 not a power of two) variable ones per cell.
//
// k_bulk on 128 x 128 x 256 cells: 990 us -> 219 us under ncu, 5.8 TB/s of the 304 B
// per cell (0.86 of the measured HBM bandwidth, which now bounds it); 1193
// instructions per warp of cells, issue 58 %, FP64 pipe (the 19 conversions
// out) 59 %.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace lbmgpu {

using ::fma;  // keep the float / double overloads visible

constexpr int FIX_BITS = 58;                      // unit 2^-58
constexpr long long FIX_BIAS = 1LL << 62;         // makes product operands non-negative

// Product by a constant c in (0, 1/2): K = round(c 2^64) = hi 2^32 + lo, a
// multiple of 4.  With A = a + 2^62 (a in (-2^62, 2^62)) the value
//   hi32(A) hi + ((hi32(A) lo + lo32(A) hi + rnd) >> 32)
// is floor((A K + rnd') / 2^64) up to the dropped low x low product, whose
// mean is in rnd together with the half unit; off = K/4 takes the bias out
// again.  No term overflows: hi32(A), hi < 2^31 and lo < 2^32.
struct FixMul {
    unsigned hi, lo;
    unsigned long long rnd;
    long long off;
};

// Constants of the fixed-point collision (make_fix, lbm_launch.h).
struct FixColl {
    int on;            // 0: constants out of range, every cell takes the FP64 form
    int unit_rho;      // rho0 is a power of two: j/rho0 needs no product
    int e0;            // biased exponent of the smallest population, 2^(sh - 6)
    unsigned lim0, lima, limd, lim_lo;  // FP64 high words: upper ends (rest, axis, diagonal), lower end
    int out_sub;       // (58 - sh) in the exponent field of an FP64 high word
    int inv_hi, inv_lo;                 // 2^sh / rho0 in units 2^-58, signed limbs
    FixMul p0, pa, pd;                  // |l+| / 12, / 36, / 72
    FixMul oa, od;                      // |l-| / 6, / 12
    // forcing: (2 / l+) f_ext / rho0 in units 2^-(58 + gs), signed limbs, and
    // the odd products' constants with F_q^- folded in, pairs q = 1, 3, ..., 17
    int gs;
    int g_hi[3], g_lo[3];
    unsigned long long o_rnd[9];
    long long o_off[9];
};

// a c for the constant of m, rounding and offset given apart.
__device__ __forceinline__ long long fix_mul(long long a, const FixMul& m, unsigned long long rnd,
                                             long long off) {
    const unsigned long long A = (unsigned long long)(a + FIX_BIAS);
    const unsigned aH = (unsigned)(A >> 32), aL = (unsigned)A;
    unsigned long long mid = (unsigned long long)aH * m.lo + rnd;
    mid += (unsigned long long)aL * m.hi;
    return (long long)((unsigned long long)aH * m.hi + (mid >> 32)) - off;
}
__device__ __forceinline__ long long fix_mul(long long a, const FixMul& m) {
    return fix_mul(a, m, m.rnd, m.off);
}

// Signed limbs: v = hi 2^32 + lo with lo in [-2^31, 2^31).
struct FixLimbs {
    int hi, lo;
};
__device__ __forceinline__ FixLimbs fix_split(long long v) {
    return FixLimbs{(int)((v + 0x80000000LL) >> 32), (int)v};
}
// a b 2^-64, rounded to nearest; the dropped lo x lo product is below 1/4 unit
// and has mean zero.
__device__ __forceinline__ long long fix_mul(FixLimbs a, FixLimbs b) {
    const long long mid = (long long)a.hi * b.lo + ((long long)a.lo * b.hi + 0x80000000LL);
    return (long long)a.hi * b.hi + (mid >> 32);
}

__device__ __forceinline__ unsigned umin3(unsigned a, unsigned b, unsigned c) {
    return min(min(a, b), c);
}
__device__ __forceinline__ unsigned umax3(unsigned a, unsigned b, unsigned c) {
    return max(max(a, b), c);
}

__device__ __forceinline__ double fix_to_double(long long v, int out_sub) {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d);
    return __hiloint2double(hi == 0 ? 0 : hi - out_sub, __double2loint(d));
}

// One opposite pair (Q, Q + 1): s, d its sum and difference, cj = c_Q . j;
// even = 2 base + 9 (c.j)^2/rho0 (with the forcing's share taken off).
template <int Q, bool AXIS, bool FORCE>
__device__ __forceinline__ void fix_pair(long long (&v)[19], long long cj, long long even,
                                         const FixColl& k) {
    const long long s = v[Q] + v[Q + 1], d = v[Q] - v[Q + 1];
    const long long e = AXIS ? fix_mul(18 * s - even, k.pa) : fix_mul(36 * s - even, k.pd);
    const FixMul& m = AXIS ? k.oa : k.od;
    const long long x = (AXIS ? 3 * d : 6 * d) - cj;
    const long long o = FORCE ? fix_mul(x, m, k.o_rnd[(Q - 1) / 2], k.o_off[(Q - 1) / 2])
                              : fix_mul(x, m);
    v[Q] = v[Q] - e - o;
    v[Q + 1] = v[Q + 1] - e + o;
}

// Collides the cell in place and returns true, or returns false with f
// unchanged when the cell is outside the range of the fixed point.
//
// Range: all f >= 2^-6, f_0 < 3/4, axis < 1/4, diagonal < 1/8, |j| < 1/4 per
// axis (in 2^sh; rho0 lies in [0.7, 1.42)), so rho < 3.75, j.j/rho0 < 0.27,
// (c.j)^2/rho0 < 0.36, and every product operand (36 s <= 9, 2 base <= 7.5,
// 12 f_0 <= 9, forcing <= 1.2) stays below 16 in magnitude: inside +-2^62.
template <bool FORCE>
__device__ __forceinline__ bool fixed_collide_t(double (&f)[19], const FixColl& k) {
    unsigned h[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) h[q] = (unsigned)__double2hiint(f[q]);
    unsigned mn = h[0], ma = 0, md = 0;
#pragma unroll
    for (int q = 1; q < 19; q += 2) mn = umin3(mn, h[q], h[q + 1]);
#pragma unroll
    for (int q = 1; q < 7; q += 2) ma = umax3(ma, h[q], h[q + 1]);
#pragma unroll
    for (int q = 7; q < 19; q += 2) md = umax3(md, h[q], h[q + 1]);
    if (!(mn >= k.lim_lo && h[0] < k.lim0 && ma < k.lima && md < k.limd)) return false;
    long long v[19];
#pragma unroll
    for (int q = 0; q < 19; ++q) {
        // significand << (exponent - e0): 0..5 places in range
        const unsigned hi = (h[q] & 0xFFFFFu) | 0x100000u, lo = (unsigned)__double2loint(f[q]);
        const int sh = (int)(h[q] >> 20) - k.e0;
        v[q] = (long long)(((unsigned long long)__funnelshift_l(lo, hi, sh) << 32) |
                           (unsigned)(lo << (sh & 31)));
    }
    const long long s1 = v[1] + v[2], s3 = v[3] + v[4], s5 = v[5] + v[6], s7 = v[7] + v[8];
    const long long s9 = v[9] + v[10], s11 = v[11] + v[12], s13 = v[13] + v[14];
    const long long s15 = v[15] + v[16], s17 = v[17] + v[18];
    const long long rho = v[0] + s1 + s3 + s5 + s7 + s9 + s11 + s13 + s15 + s17;
    const long long d7 = v[7] - v[8], d9 = v[9] - v[10], d11 = v[11] - v[12];
    const long long d13 = v[13] - v[14], d15 = v[15] - v[16], d17 = v[17] - v[18];
    const long long jx = (v[1] - v[2]) + d7 + d9 + d11 + d13;
    const long long jy = (v[3] - v[4]) + d7 - d9 + d15 + d17;
    const long long jz = (v[5] - v[6]) + d11 - d13 + d15 - d17;
    // |j| < 1/4: high words in [-2^24, 2^24)
    constexpr unsigned J = 1u << 24;
    if (!((unsigned)((int)(jx >> 32) + J) < 2 * J && (unsigned)((int)(jy >> 32) + J) < 2 * J &&
          (unsigned)((int)(jz >> 32) + J) < 2 * J)) {
        // the conversion was exact, so f need not be kept beside v
#pragma unroll
        for (int q = 0; q < 19; ++q) f[q] = fix_to_double(v[q], k.out_sub);
        return false;
    }
    // j 2^6 against u = j / rho0: products land in units 2^-58
    const FixLimbs ax = fix_split(jx * 64), ay = fix_split(jy * 64), az = fix_split(jz * 64);
    FixLimbs ux, uy, uz;
    if (k.unit_rho) {
        ux = fix_split(jx);
        uy = fix_split(jy);
        uz = fix_split(jz);
    } else {
        const FixLimbs inv{k.inv_hi, k.inv_lo};
        ux = fix_split(fix_mul(ax, inv));
        uy = fix_split(fix_mul(ay, inv));
        uz = fix_split(fix_mul(az, inv));
    }
    const long long xx = fix_mul(ax, ux), yy = fix_mul(ay, uy), zz = fix_mul(az, uz);
    const long long xy = fix_mul(ax, uy), xz = fix_mul(ax, uz), yz = fix_mul(ay, uz);
    const long long b2 = 2 * rho - 3 * (xx + yy + zz);  // 2 base
    if (!FORCE) {
        v[0] -= fix_mul(12 * v[0] - 2 * b2, k.p0);
        fix_pair<1, true, FORCE>(v, jx, b2 + 9 * xx, k);
        fix_pair<3, true, FORCE>(v, jy, b2 + 9 * yy, k);
        fix_pair<5, true, FORCE>(v, jz, b2 + 9 * zz, k);
        const long long txy = b2 + 9 * (xx + yy), txz = b2 + 9 * (xx + zz), tyz = b2 + 9 * (yy + zz);
        const long long cxy = 18 * xy, cxz = 18 * xz, cyz = 18 * yz;
        fix_pair<7, false, FORCE>(v, jx + jy, txy + cxy, k);
        fix_pair<9, false, FORCE>(v, jx - jy, txy - cxy, k);
        fix_pair<11, false, FORCE>(v, jx + jz, txz + cxz, k);
        fix_pair<13, false, FORCE>(v, jx - jz, txz - cxz, k);
        fix_pair<15, false, FORCE>(v, jy + jz, tyz + cyz, k);
        fix_pair<17, false, FORCE>(v, jy - jz, tyz - cyz, k);
    } else {
        // even part of the forcing: (2/l+) (9 (c.j)(c.f) - 3 j.f) / rho0 joins
        // the operand; the products carry gs more bits so that a weak force
        // keeps its significand
        const FixLimbs gx{k.g_hi[0], k.g_lo[0]}, gy{k.g_hi[1], k.g_lo[1]}, gz{k.g_hi[2], k.g_lo[2]};
        const long long mxx = fix_mul(ax, gx), myy = fix_mul(ay, gy), mzz = fix_mul(az, gz);
        const long long mxy = fix_mul(ax, gy) + fix_mul(ay, gx);
        const long long mxz = fix_mul(ax, gz) + fix_mul(az, gx);
        const long long myz = fix_mul(ay, gz) + fix_mul(az, gy);
        const long long half = (1LL << k.gs) >> 1;
        const long long w = mxx + myy + mzz, w3 = half - 3 * w;
        v[0] -= fix_mul(12 * v[0] - 2 * b2 - ((6 * w + half) >> k.gs), k.p0);
        const auto ev = [&](long long m) { return (9 * m + w3) >> k.gs; };
        fix_pair<1, true, FORCE>(v, jx, b2 + 9 * xx - ev(mxx), k);
        fix_pair<3, true, FORCE>(v, jy, b2 + 9 * yy - ev(myy), k);
        fix_pair<5, true, FORCE>(v, jz, b2 + 9 * zz - ev(mzz), k);
        const long long txy = b2 + 9 * (xx + yy), txz = b2 + 9 * (xx + zz), tyz = b2 + 9 * (yy + zz);
        fix_pair<7, false, FORCE>(v, jx + jy, txy + 18 * xy - ev(mxx + myy + mxy), k);
        fix_pair<9, false, FORCE>(v, jx - jy, txy - 18 * xy - ev(mxx + myy - mxy), k);
        fix_pair<11, false, FORCE>(v, jx + jz, txz + 18 * xz - ev(mxx + mzz + mxz), k);
        fix_pair<13, false, FORCE>(v, jx - jz, txz - 18 * xz - ev(mxx + mzz - mxz), k);
        fix_pair<15, false, FORCE>(v, jy + jz, tyz + 18 * yz - ev(myy + mzz + myz), k);
        fix_pair<17, false, FORCE>(v, jy - jz, tyz - 18 * yz - ev(myy + mzz - myz), k);
    }
#pragma unroll
    for (int q = 0; q < 19; ++q) f[q] = fix_to_double(v[q], k.out_sub);
    return true;
}

}  // namespace lbmgpu
