// Host-side launch interface between the C-ABI layer and the kernels.
// Internal to the library; not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include <cmath>

#include "../../include/lbm_gb300.h"
#include "lbm_device.cuh"
#include "lbm_dfloat.cuh"
#include "lbm_fixed.cuh"

namespace lbmgpu {

struct Launch {
    Geom g;
    Coll<double> kd;   // FP64 collision constants
    Coll<float> kf;    // FP32 collision constants
    Coll<dfloat> kff;  // float-float collision constants (FP64 storage)
    Coupl cp;
    DevParticle* parts;       // particle state used by this sweep
    DevParticle* parts_prev;  // state before the last rigid-body update (refill)
    double* partials;         // force/torque partials of this sweep
    int* status;
    int nostream;             // 1: stored buffer holds pre-collision f (no stream)
    int all_tiles;            // bulk kernel: process every tile (no coupling)
    int* gate;                // not null: launch_near and, right after it on the same stream,
    int gate_key;             //   launch_bulk run beside one another (see gate_open)
    long long near_nblk;      // near-kernel blocks per particle
    int refill_side;          // refill box: cube side in cells
    unsigned short* map;      // per-step geometry map (see k_map)
    int map_ext[3];           // region box extents of the map (cells)
    dim3 block;
    cudaStream_t stream;
};

// Near-kernel blocks: one warp, 32 cells of a particle's region (at most
// D + 2 NEAR_HALO + 1 cells per axis; the grid covers ceil(D) + 6).  A warp is
// one chain of ~3500 instructions (MEM CLI, D = 8: 22 us, a third of it waiting
// for instructions, a third for the latency of the one before), so full warps
// and one to an SM are what a small sphere needs; rows of 32 cells, two to a
// block, left 20 of 32 lanes idle at D = 8 and 22 of 64 at D = 36.  us per pass,
// rows / this: 32^3 FP64 PSM 1954 / 1850; four D = 16 spheres, one sweep
// 139 / 128; ensemble of 12, 3467 / 3397; 192 x 192 x 768 BF16 5712 / 5556.
constexpr int NEAR_THREADS = 32;
// threads per block of the refill kernels (whole warps: a warp rebuilds a cell)
constexpr int REFILL_THREADS = 128;
static_assert(NEAR_THREADS == 32, "a near block is one warp");
static_assert(REFILL_THREADS % 32 == 0, "refill blocks are whole warps");
// blocks of the refill kernel per particle for a box of side^3 cells
__host__ __device__ inline long long refill_blocks(int side) {
    return ((long long)side * side * side + REFILL_THREADS - 1) / REFILL_THREADS;
}

// Cells per axis of the region box that holds any particle of diameter <= maxd.
inline void region_extent(const Geom& g, double maxd, int ext[3]) {
    const int span = (int)ceil(maxd) + 2 * (int)NEAR_HALO + 2;
    ext[0] = g.nx < span ? g.nx : span;
    ext[1] = g.ny < span ? g.ny : span;
    ext[2] = g.nz < span ? g.nz : span;
}

// Map entries (unsigned short) for np particles.
inline long long map_entries(const Geom& g, double maxd, int np) {
    int ext[3];
    region_extent(g, maxd, ext);
    return (long long)(np > 0 ? np : 1) * ext[0] * ext[1] * ext[2];
}

inline long long near_blocks(const Geom& g, double maxd) {
    return (map_entries(g, maxd, 1) + NEAR_THREADS - 1) / NEAR_THREADS;
}

// Doubles of force partials one sweep needs: np regions x blocks x np x 6.
inline long long near_partial_doubles(long long nblk, int np) {
    const long long n = np > 0 ? np : 1;
    return n * nblk * n * 6;
}

// ---- batched ensemble ----------------------------------------------------------
// One independent simulation of a batch (one particle, FP64 PDFs).  Lives in
// device memory; the kernels read buf[cur] and flip cur themselves, so one
// step's launches are the same every step and can be replayed as a graph.
struct BatchCase {
    Geom g;
    double* buf[2];
    int cur;
    int kind;          // 1 PSM, 2 MEM, 0 none
    int subcycles;     // LBM sweeps per global step
    int layout;        // bulk tiling: 0 box tiles (g.tx x g.ty), 1 256-cell plane segments
    int wall_contact;
    Coupl cp;          // np = 1
    Coll<double> kd;
    DevParticle* part;
    DevParticle* prev;
    double* force;     // 6 doubles
    double* partials;  // subcycles x nblk x 6
    unsigned short* map;
    int map_ext[3];
    long long nblk;    // near-kernel blocks
    int refill_side;
    double gravity[3];
    int remap_charge;     // MEM: charge the re-mapping momentum (lbm_batch_set_remap_charge)
    double* charge;       // 6 doubles: pending amounts of the last re-mapping
    double* charge_part;  // refill_blocks(refill_side) x 6 block partials
};

static_assert(sizeof(BatchCase) % 8 == 0, "staged as 8-byte words");

// Work list of a batched launch: cases list[0..n) with prefix sums base[] of
// their work items (tiles, blocks or cells).
struct BatchList {
    const int* list;
    const long long* base;  // n + 1 entries
    int n;
};

// Collision constants of Eq. (5) / (9)-(11) with the forcing of Eq. (7)
// (computed in FP64, rounded once to C).
// MEM MR, Eq. (15): Lambda_- = 1/|lambda_-| - 1/2 of the collision (TRT:
// Lambda / (tau - 1/2), Eq. (11); BGK: tau - 1/2).  The correction term
// f^pc = -8 Lambda_- n^-_q / ((2 Lambda_- + 1)(1 + delta)^2) needs the
// pre-collision odd non-equilibrium n^-_q(x, t); the kernels rebuild it from
// the stored post-collision values, (1 - |lambda_-|) n^-_q =
// (f~_q - f~_qbar)/2 - 3 w_q c_q . j~ (the forcing drops out), so the scale
// applied to that difference is -4 Lambda_- / (Lambda_- - 1/2).  The rebuild
// loses n^- as |lambda_-| -> 1; MR is refused within 0.01 of Lambda_- = 1/2.
inline double mr_lambda_minus(const lbm_config& cfg) {
    return cfg.collision == LBM_TRT ? cfg.magic / (cfg.tau - 0.5) : cfg.tau - 0.5;
}
inline bool mr_supported(const lbm_config& cfg) {
    return std::fabs(mr_lambda_minus(cfg) - 0.5) >= 0.01;
}
inline double mr_correction_scale(const lbm_config& cfg) {
    const double Lm = mr_lambda_minus(cfg);
    return -4.0 * Lm / (Lm - 0.5);
}

// Constants of the fixed-point collision (lbm_fixed.cuh); on = 0 where they
// do not fit it (forces of a cell's weight, extreme rho0).
inline FixMul make_fix_mul(double c) {
    FixMul m{};
    const unsigned long long K = (unsigned long long)std::llround(std::ldexp(c, 62)) << 2;
    m.hi = (unsigned)(K >> 32);
    m.lo = (unsigned)K;
    m.rnd = 0x80000000ull + m.lo / 2;
    m.off = (long long)(K >> 2);
    return m;
}
inline void fix_limbs(double x, int& hi, int& lo) {
    const long long v = std::llround(x);
    hi = (int)((v + 0x80000000LL) >> 32);
    lo = (int)(unsigned)(v & 0xFFFFFFFFLL);
}
inline FixColl make_fix(double lp, double lm, double rho0, const double fe[3]) {
    FixColl k{};
    int sh = 0;
    double r = std::frexp(rho0, &sh);  // [1/2, 1)
    if (r > 0.70710678) r *= 0.5;
    else --sh;
    r *= 2.0;  // rho0 = r 2^sh, r in [0.707, 1.415)
    if (sh > 400 || sh < -400 || !(lp > -2.0 && lp < 0.0 && lm > -2.0 && lm < 0.0)) return k;
    k.unit_rho = r == 1.0;
    k.e0 = 1017 + sh;
    const unsigned es = (unsigned)(sh * (1 << 20));
    k.lim_lo = 0x3F900000u + es;  // 2^-6
    k.lim0 = 0x3FE80000u + es;    // 3/4
    k.lima = 0x3FD00000u + es;    // 1/4
    k.limd = 0x3FC00000u + es;    // 1/8
    k.out_sub = (FIX_BITS - sh) * (1 << 20);
    fix_limbs(std::ldexp(1.0 / r, FIX_BITS), k.inv_hi, k.inv_lo);
    k.p0 = make_fix_mul(-lp / 12.0);
    k.pa = make_fix_mul(-lp / 36.0);
    k.pd = make_fix_mul(-lp / 72.0);
    k.oa = make_fix_mul(-lm / 6.0);
    k.od = make_fix_mul(-lm / 12.0);
    double f[3], g[3], gmax = 0.0;
    for (int a = 0; a < 3; ++a) {
        f[a] = std::ldexp(fe[a], -sh);
        g[a] = 2.0 / lp * f[a] / r;
        gmax = std::fmax(gmax, std::fabs(g[a]));
        if (!(std::fabs(f[a]) < 0.01)) return k;
    }
    if (!(gmax < 0.125)) return k;
    // g in units 2^-(58 + gs), the largest component in [2^55, 2^57)
    while (k.gs < 62 && std::ldexp(gmax, k.gs) < 0.125) ++k.gs;
    for (int a = 0; a < 3; ++a) fix_limbs(std::ldexp(g[a], FIX_BITS + k.gs), k.g_hi[a], k.g_lo[a]);
    for (int q = 1; q < NQ; q += 2) {
        // o - F_q^-: the integer part of F_q^- joins off, the fraction rnd
        const FixMul& m = q <= 6 ? k.oa : k.od;
        const double F = std::ldexp(3.0 * wq(q) * (cx(q) * f[0] + cy(q) * f[1] + cz(q) * f[2]), FIX_BITS);
        const double up = std::ceil(F);
        k.o_off[(q - 1) / 2] = m.off + (long long)up;
        k.o_rnd[(q - 1) / 2] = m.rnd + (unsigned long long)std::ldexp(up - F, 32);
    }
    k.on = 1;
    return k;
}

template <typename C>
inline Coll<C> make_coll(double lp, double lm, double rho0, const double fe[3]) {
    Coll<C> k{};
    k.lam_p = (C)lp;
    k.lam_m = (C)lm;
    k.rho0 = (C)rho0;
    k.inv_rho0 = (C)(1.0 / rho0);
    k.fx = (C)fe[0];
    k.fy = (C)fe[1];
    k.fz = (C)fe[2];
    k.has_force = (fe[0] != 0.0 || fe[1] != 0.0 || fe[2] != 0.0);
    k.alpha = (C)(1.0 + 0.5 * (lp + lm));
    k.beta = (C)(0.5 * (lp - lm));
    k.c0 = (C)(1.0 + lp);
    k.m15r0 = (C)(-1.5 / rho0);
    const double w[3] = {1.0 / 3.0, 1.0 / 18.0, 1.0 / 36.0};
    for (int c = 0; c < 3; ++c) {
        k.lpw[c] = (C)(lp * w[c]);
        k.k1w[c] = (C)(4.5 * lp * w[c] / rho0);
        k.k2w[c] = (C)(3.0 * lm * w[c]);
        k.hw[c] = (C)(3.0 * w[c] / rho0);
    }
    for (int q = 1; q < NQ; q += 2) {
        const double cf = cx(q) * fe[0] + cy(q) * fe[1] + cz(q) * fe[2];
        k.gq[(q - 1) / 2] = (C)(9.0 * wq(q) * cf / rho0);
        k.fq[(q - 1) / 2] = (C)(3.0 * wq(q) * cf);
    }
    if constexpr (std::is_same<C, double>::value) k.fix = make_fix(lp, lm, rho0, fe);
    return k;
}

// FP64 collision constants of a storage mode.  The fixed-point form is left out in
// LBM_STORE_F64_DP, and above tau = 2 unless LBM_STORE_F64_FX asks for it: root mean
// square error over that of the FP64 form, largest of 20 flows, BGK: tau = 2 0.66, 3
// 0.91, 4 0.93, 6 1.05, 8 1.06 (TRT stays below 1).
constexpr double FIX_TAU_MAX = 2.0;
inline Coll<double> make_coll_f64(int storage, double lp, double lm, double rho0, const double fe[3]) {
    Coll<double> k = make_coll<double>(lp, lm, rho0, fe);
    if (storage == LBM_STORE_F64_DP || (storage != LBM_STORE_F64_FX && lp > -1.0 / FIX_TAU_MAX))
        k.fix.on = 0;
    return k;
}

// Checks of a configuration shared by every entry point that takes one
// (lbm_create, lbm_sweep_noalloc): LBM_ERR_ARG for a value outside its
// range, LBM_ERR_UNSUPPORTED for MEM MR within 0.01 of Lambda_- = 1/2.
// Host-only; touches no device state.
inline lbm_status check_config(const lbm_config& c) {
    if (c.nx < 1 || c.ny < 1 || c.nz < 1) return LBM_ERR_ARG;
    if ((long long)c.nx * c.ny * c.nz > (1LL << 40)) return LBM_ERR_ARG;
    if (!(c.tau > 0.5) || !std::isfinite(c.tau) || !(c.rho0 > 0.0) || !std::isfinite(c.rho0))
        return LBM_ERR_ARG;
    if (c.coupling < 0 || c.coupling > LBM_NONE) return LBM_ERR_ARG;
    if (c.collision != LBM_BGK && c.collision != LBM_TRT) return LBM_ERR_ARG;
    if (c.storage < LBM_STORE_F64 || c.storage > LBM_STORE_F64_DP) return LBM_ERR_ARG;
    if (c.bc_z < 0 || c.bc_z > 2 || (c.bc_z == 2 && c.nz < 3)) return LBM_ERR_ARG;
    if (c.bc_z == 2 && !(std::isfinite(c.inflow[0]) && std::isfinite(c.inflow[1]) &&
                         std::isfinite(c.inflow[2]) && c.rho_out > 0.0 && std::isfinite(c.rho_out)))
        return LBM_ERR_ARG;
    for (int a = 0; a < 3; ++a)
        if (!std::isfinite(c.force_density[a]) || !std::isfinite(c.gravity[a])) return LBM_ERR_ARG;
    if (c.subsample < 0 || c.subsample > 40 || c.lbm_subcycles < 0) return LBM_ERR_ARG;
    if (c.collision == LBM_TRT) {
        // Eq. (11): lambda_- from Lambda = magic; it must lie in (-2, 0)
        const double lp = -1.0 / c.tau;
        const double denom = c.magic / (0.5 + 1.0 / lp) - 0.5;
        if (!(c.magic > 0.0) || !std::isfinite(c.magic) || denom == 0.0) return LBM_ERR_ARG;
        const double lm = 1.0 / denom;
        if (!(lm > -2.0 && lm < 0.0)) return LBM_ERR_ARG;
    }
    if (c.coupling == LBM_MEM_MR && !mr_supported(c)) return LBM_ERR_UNSUPPORTED;
    return LBM_OK;
}

// Bulk tiles of a handle's lattice: one tile is one block of k_bulk
// (BulkShape), a row or more of one z plane; FP32 takes two planes per thread.
inline void set_tiles(Geom& g, int storage) {
    const int threads = storage == LBM_STORE_F32 ? 256 : 128;
    g.tx = g.nx >= 128 ? 128 : (g.nx >= 64 ? 64 : 32);
    while (g.tx > 8 && (long long)g.ny * g.tx > 65535LL * threads) g.tx /= 2;  // grid y limit
    g.ty = threads / g.tx;
    g.ntx = (g.nx + g.tx - 1) / g.tx;
    g.nty = (g.ny + g.ty - 1) / g.ty;
    g.tz = storage == LBM_STORE_F32 ? 2 : 1;
    g.ntz = (g.nz + g.tz - 1) / g.tz;
}

// Open-boundary data of a configuration (bc_z = 2) into the geometry.
inline void set_open_boundaries(Geom& g, const lbm_config& cfg) {
    for (int a = 0; a < 3; ++a) {
        g.uin[a] = cfg.bc_z == 2 ? cfg.inflow[a] : 0.0;
        g.fhalf[a] = cfg.force_density[a] / (2.0 * cfg.rho0);
    }
    g.rho_out = cfg.bc_z == 2 ? cfg.rho_out : cfg.rho0;
    g.rho0 = cfg.rho0;
}

// Status bits raised by kernels (OR-ed into *status).
enum : int {
    ST_TOO_MANY_OBJECTS = 1,  // more than CELL_SLOTS particles touch a cell
    ST_DOMAIN = 2,            // a particle left the domain through a closed wall
    ST_REFILL_SOLID = 4,      // refill found no particle owning a cell (internal)
    ST_UNSTABLE = 8,          // a particle state became non-finite or too fast
    ST_BOUNDS = 16,           // an index check or a bounded wait failed (access skipped)
    ST_FLUID = 32,            // a fluid cell's density became non-finite or <= 0
};
static_assert((int)ST_TOO_MANY_OBJECTS == (int)LBM_STATUS_TOO_MANY_OBJECTS &&
                  (int)ST_DOMAIN == (int)LBM_STATUS_DOMAIN &&
                  (int)ST_UNSTABLE == (int)LBM_STATUS_UNSTABLE &&
                  (int)ST_BOUNDS == (int)LBM_STATUS_BOUNDS && (int)ST_FLUID == (int)LBM_STATUS_FLUID,
              "status bits of the public header");

// storage: 0 = FP64, 1 = FP32 (arithmetic in the same precision), 4 = FP16
// and 5 = BF16 shifted populations f - w_q (FP32 arithmetic); launch_bulk
// also takes 2 = FP64 storage with float-float collision
cudaError_t launch_bulk(int storage, const void* src, void* dst, const Launch& L);
cudaError_t launch_near(int storage, const void* src, void* dst, const Launch& L);
// Whether a sweep runs as one launch (launch_sweep: near and bulk cells), and the
// largest lattice that does.  us for 20 steps, near sweep on a second stream /
// one launch: FP64 PSM 32^3 756 / 643, 64^3 964 / 872, 80^3 1400 / 1469; FP64 MEM
// (two sweeps a step) 32^3 1221 / 1050, 64^3 1777 / 1571, 80^3 2511 / 2476; FP32
// PSM 64^3 684 / 637, 80^3 793 / 936; FP32 MEM 64^3 1512 / 1257, 80^3 1745 / 1491
// (and 1277 beside one another on one stream: sweep_beside).
constexpr long long SWEEP_FUSED_CELLS = 1 << 18;
bool sweep_fused(const Launch& L, int bulk_mode);
// Whether a handle's near and bulk sweeps run beside one another on one stream
// (L.gate), in place of a second stream with its fork and join: FP32 lattices whose
// bulk sweep is up to 4 (PSM) or 6 (MEM, the longer near sweep) waves of blocks, each
// of which pays for the gate's load.  us for 20 steps, second stream / gate, by
// waves: PSM 66^3 (2.5) 690 / 634, 80^3 (3.5) 713 / 697, 88^3 (4.2) 771 / 801,
// 96^3 (5.1) 841 / 921; MEM (two sweeps a step) 66^3 1367 / 1219, 88^3 1600 / 1534, 96^3
// 1768 / 1676; 64 x 64 x 192 PSM with features (3.4), 10 steps 1077 / 1049.  FP64:
// 72^3 1156 / 1173, 96^3 1646 / 1755, 128 x 128 x 512 4264 / 4497, so never.
// Near sweeps of more than 8 blocks to an SM would hold the bulk blocks up.
bool sweep_beside(const Launch& L, int bulk_mode, int sms);
cudaError_t launch_sweep(int storage, const void* src, void* dst, const Launch& L);
// charge_part != nullptr: also the re-mapping momentum charge partials,
// refill_blocks(L.refill_side) blocks x 6 doubles per particle (see k_refill)
cudaError_t launch_refill(int storage, const void* srcB, void* dst, const Launch& L,
                          const DevParticle* p_old, const DevParticle* p_new, int extrapolate,
                          double* charge_part = nullptr);
// charge[p * 6 + c] = fixed-order total of the refill's charge partials
cudaError_t launch_charge_total(const Launch& L, const double* charge_part, double* charge);
cudaError_t launch_macro(int storage, const void* state, const Launch& L, int what, void* out);
cudaError_t launch_init_eq(int storage, void* dst, const Launch& L, double rho, double ux,
                           double uy, double uz);
cudaError_t launch_from_f64(int storage, const double* in, void* dst, long long count,
                            long long ncell, cudaStream_t s);
cudaError_t launch_to_f64(int storage, const void* in, double* out, long long count,
                          long long ncell, cudaStream_t s);
// charge != nullptr: the pending re-mapping momentum charge, [p][6], over nsub
// is taken off the totals
cudaError_t launch_finalize(const Launch& L, int nsub, double* force_out,
                            const double* charge = nullptr);
// the force total and the rigid-body update (dt = nsub) in one launch
cudaError_t launch_finalize_rigid(const Launch& L, int nsub, double* force, const double* charge,
                                  double gx, double gy, double gz, int wall_contact);
// Stores n particle records with their regions in parts (and prev), the records
// that parts held before in old (prev, old: may be null).  The records travel as
// a kernel argument, copied at launch: nothing waits for the host array.
struct ParticleUpload {
    DevParticle rec[MAX_PARTICLES];
};
static_assert(sizeof(ParticleUpload) <= 16000, "kernel argument too large");
cudaError_t launch_set_particles(const Launch& L, const ParticleUpload& up, int n, DevParticle* parts,
                                 DevParticle* prev, DevParticle* old);
// batched ensemble (all cases on one stream; see lbm_batch.cu)
cudaError_t launch_batch_regions(BatchCase* cases, int n, cudaStream_t s);
cudaError_t launch_batch_map(BatchCase* cases, BatchList l, long long total, cudaStream_t s);
cudaError_t launch_batch_near(BatchCase* cases, BatchList l, long long total, int sub,
                              int* status, cudaStream_t s);
// grid <= 0: one block per tile
cudaError_t launch_batch_bulk(BatchCase* cases, BatchList l, long long total, int grid,
                              int* status, cudaStream_t s);
cudaError_t launch_batch_swap(BatchCase* cases, BatchList l, cudaStream_t s);
cudaError_t launch_batch_finalize(BatchCase* cases, int n, cudaStream_t s);
cudaError_t launch_batch_rigid(BatchCase* cases, int n, int* status, cudaStream_t s);
// p[0] = now (end = 0); p[1] += now - p[0], p[2] += 1 (end = 1); now from
// the global nanosecond timer
cudaError_t launch_stamp(unsigned long long* p, int end, cudaStream_t s);
// per case with the charge on: total of its refill-block charge partials
cudaError_t launch_batch_charge_total(BatchCase* cases, int n, cudaStream_t s);
cudaError_t launch_batch_refill(BatchCase* cases, BatchList l, long long total, int* status,
                                cudaStream_t s);
cudaError_t launch_batch_init(BatchCase* cases, int n, long long max_cells, cudaStream_t s);
int batch_bulk_blocks_per_sm();
cudaError_t launch_map(const Launch& L);
// learned force correction (lbm_learned.cu)
cudaError_t launch_features(int storage, const void* state, const Launch& L, const double* force,
                            double u_ref, float* feat);
cudaError_t launch_apply_correction(const float* y, const DevParticle* parts, int np, double u_ref,
                                    double rho0, double* force, cudaStream_t s);
// clip > 0: samples with a normalised input beyond +-clip get y = 0
cudaError_t mlp_infer(const lbm_mlp* m, const float* x, int n, float* y, float clip,
                      cudaStream_t s);
cudaError_t launch_rigid_body(const Launch& L, const double* force, double gx, double gy,
                              double gz, double dt, int wall_contact);

}  // namespace lbmgpu
