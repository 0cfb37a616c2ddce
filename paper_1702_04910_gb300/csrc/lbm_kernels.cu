// Kernels of the coupled D3Q19 step and their launchers (sm_103a).
//
// One global step (Algorithm 1 / Algorithm 2 of Rettinger & Ruede,
// arXiv:1702.04910) is built from:
//   k_bulk      fused pull stream + fluid collision for every cell that no
//               particle comes near (the whole domain but an O(D^3) box);
//   k_near      the same for the cells near a particle, with the coupling:
//               PSM solid fractions and weighted collision Eq. (20)-(26) and
//               force/torque Eq. (28)-(29), or MEM link boundary conditions
//               Eq. (12)/(14) and link forces Eq. (16); per-block force
//               partials reduced warp -> block in a fixed order;
//   k_finalize  fixed-order sum of the block partials, subcycle average;
//   k_rigid     explicit Euler rigid-body update;
//   k_refill    MEM re-mapping: PDF reconstruction Eq. (19) of uncovered
//               cells, then their collision; optionally the momentum the
//               covered and uncovered cells exchange with the fluid, as
//               fixed-order block partials (k_charge_total adds them, and
//               the next k_finalize takes them off the force);
//   k_bulk_pair the 16-bit bulk sweep, two x-neighbours per thread in packed
//               f32x2 arithmetic.
// The batched ensemble has k_batch_* counterparts of these; k_stamp reads
// the global timer around a launch for device-side timing.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "lbm_launch.h"

namespace lbmgpu {

// ---------------------------------------------------------------------------
// Programmatic dependent launch.  The kernels of a step are short and follow one
// another on a stream, so each is launched while its predecessor still runs
// (launch_after below): its blocks take their places and wait here until the
// predecessor has completed and its writes are visible, then let the successor
// be launched in turn.  Every kernel launched that way calls this before it
// touches memory, so a kernel's completion implies that of all before it.
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void step_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void step_enter() {
    step_wait();
    step_trigger();
}
// A bulk sweep beside k_near on one stream (launch_near, then launch_bulk, with
// L.gate).  k_bulk is launched once every block of k_near has begun, and has to
// see what the kernels before k_near wrote.  k_near's wait gives that view to
// k_near alone, so it is handed on by memory order: block 0 of k_near stores the
// key to the gate with release after its wait, and a block of k_bulk loads it with
// acquire before anything else.  That store precedes the trigger that lets k_bulk
// start, so the load finds it at once; a block that does not after GATE_TRIES
// loads reports ST_BOUNDS and leaves its cells.  The grid's last block waits for
// k_near, so that whatever follows the bulk sweep follows both; the force total
// closes the gate again.
constexpr int GATE_TRIES = 1 << 16;
__device__ __forceinline__ void gate_open(int* gate, int key) {
    if (gate && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0)
        asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(gate), "r"(key) : "memory");
}
__device__ __forceinline__ bool gate_pass(const int* gate, int key) {
    if (!gate) return true;
    step_trigger();
    int seen = 1;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        int v = 0;
        for (int i = 0; i < GATE_TRIES && v != key; ++i)
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(gate) : "memory");
        seen = v == key;
    }
    return __syncthreads_and(seen);
}
__device__ __forceinline__ void gate_leave(const int* gate) {
    if (gate && threadIdx.x == 0 && threadIdx.y == 0 && blockIdx.x == gridDim.x - 1 &&
        blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1)
        step_wait();
}
__device__ __forceinline__ void gate_close(int* gate) {
    if (gate && blockIdx.x == 0 && threadIdx.x == 0) *gate = 0;
}
// A pointer whose loads cannot be moved ahead of step_enter (they may be
// declared invariant).
template <typename P>
__device__ __forceinline__ P* entered(P* p) {
    asm volatile("" : "+l"(p));
    return p;
}

// ---------------------------------------------------------------------------
// per-cell force/torque slots (a cell may touch up to CELL_SLOTS particles)
struct Slots {
    int id[CELL_SLOTS];
    double v[CELL_SLOTS][6];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int s = 0; s < CELL_SLOTS; ++s) {
            id[s] = -1;
#pragma unroll
            for (int c = 0; c < 6; ++c) v[s][c] = 0.0;
        }
    }
    // returns false when every slot is taken by other particles
    __device__ __forceinline__ bool add(int p, const double (&F)[3], const double (&T)[3]) {
#pragma unroll
        for (int s = 0; s < CELL_SLOTS; ++s) {
            if (id[s] == p || id[s] < 0) {
                id[s] = p;
                v[s][0] += F[0];
                v[s][1] += F[1];
                v[s][2] += F[2];
                v[s][3] += T[0];
                v[s][4] += T[1];
                v[s][5] += T[2];
                return true;
            }
        }
        return false;
    }
    __device__ __forceinline__ double get(int p, int c) const {
        double r = 0.0;
#pragma unroll
        for (int s = 0; s < CELL_SLOTS; ++s)
            if (id[s] == p) r += v[s][c];
        return r;
    }
};

__device__ __forceinline__ void cross3(const double (&a)[3], const double (&b)[3],
                                       double (&r)[3]) {
    r[0] = a[1] * b[2] - a[2] * b[1];
    r[1] = a[2] * b[0] - a[0] * b[2];
    r[2] = a[0] * b[1] - a[1] * b[0];
}

// ---------------------------------------------------------------------------
// MEM pull for a fluid cell: stream Eq. (2); links whose upstream cell is
// solid take the boundary value Eq. (12) (BB), Eq. (14) (CLI) or Eq. (15)
// (MR, coefficients derived for the TRT link recurrence: kappa_1 = 1,
// kappa_0 = (1 - 2d - 2d^2)/(1+d)^2, kappa_-1 = d^2/(1+d)^2, kappabar_-1 =
// -kappa_0, kappabar_-2 = -kappa_-1, alpha = 4/(1+d)^2, d = delta_q; MR
// falls back to CLI where x - 2 c_q is not fluid, CLI to BB); resting
// closed walls take halfway bounce-back.  When `slots` is non-null the link
// force Eq. (16) and its torque about X_p (arm x_b - X_p) are accumulated.
//
// In pull form the link of the paper (fluid x, solid neighbour x + c_qp)
// appears while filling direction q = qbar_p: the upstream cell x - c_q is
// x + c_qp.
// Owner of a cell: from the per-step map when given, else evaluated from the
// particle records (same predicate, R6).
__device__ __forceinline__ int owner_of(const Geom& g, const DevParticle* parts, int np,
                                        const GeoMap* gm, int x, int y, int z) {
    return gm ? mapped_owner(g, parts, np, *gm, x, y, z) : cell_owner(g, parts, np, x, y, z);
}

// Post-collision momentum j~(x) of the boundary cell, loaded on the first MR
// link of the cell (Eq. (15) correction term).
struct MrCell {
    double j[3];
    bool have;
};

template <typename T>
__device__ __forceinline__ void own_momentum(const T* __restrict__ src, const Geom& g,
                                             long long idx, MrCell& mc) {
    if (mc.have) return;
    double j0 = 0.0, j1 = 0.0, j2 = 0.0;
#pragma unroll
    for (int q = 1; q < NQ; ++q) {
        const double v = ld_pdf(src + (long long)q * g.n + idx, q);
        j0 += v * cx(q);
        j1 += v * cy(q);
        j2 += v * cz(q);
    }
    mc.j[0] = j0;
    mc.j[1] = j1;
    mc.j[2] = j2;
    mc.have = true;
}

// Lattice velocities for a direction known only at run time (the link loop):
// two bits per direction holding c + 1.
template <int A>
__host__ __device__ constexpr unsigned long long c_bits() {
    unsigned long long b = 0;
    for (int q = 0; q < NQ; ++q)
        b |= (unsigned long long)((A == 0 ? cx(q) : (A == 1 ? cy(q) : cz(q))) + 1) << (2 * q);
    return b;
}
__device__ __forceinline__ int rcx(int q) { return (int)((c_bits<0>() >> (2 * q)) & 3ull) - 1; }
__device__ __forceinline__ int rcy(int q) { return (int)((c_bits<1>() >> (2 * q)) & 3ull) - 1; }
__device__ __forceinline__ int rcz(int q) { return (int)((c_bits<2>() >> (2 * q)) & 3ull) - 1; }

// Coordinates of x + sign * c_q (sign = +1 or -1), q known at run time.
__device__ __forceinline__ void shifted_rt(const Nbr& b, int x, int y, int z, int q, int sign,
                                           int& xs, int& ys, int& zs) {
    const int dx = sign * rcx(q), dy = sign * rcy(q), dz = sign * rcz(q);
    xs = dx > 0 ? b.xp : (dx < 0 ? b.xm : x);
    ys = dy > 0 ? b.yp : (dy < 0 ? b.ym : y);
    zs = dz > 0 ? b.zp : (dz < 0 ? b.zm : z);
}

// Phase 1 of the MEM pull, one direction Q: resting wall -> halfway
// bounce-back; fluid upstream cell -> stream Eq. (2); solid upstream cell ->
// bit Q of `cut`, filled by the link loop.
template <typename T, typename C, int Q>
__device__ __forceinline__ void mem_pull_one(const T* __restrict__ src, const Geom& g,
                                             const DevParticle* parts, int np, const Nbr& b, int x,
                                             int y, int z, long long idx, C (&f)[NQ], unsigned& cut,
                                             int* status) {
    constexpr int QP = opp(Q);
    int xs, ys, zs;
    shifted<Q>(b, x, y, z, -1, xs, ys, zs);
    if (cz(Q) != 0 && (zs < 0 || zs >= g.nz)) {
        f[Q] = PdfStore<T>::template load<C>(src + (long long)QP * g.n + idx, QP);
        return;
    }
    const int owner = cell_owner(g, parts, np, xs, ys, zs);
    // index checks: a failure is reported (ST_BOUNDS) and the access skipped
    if (!owner) {
        if (xs < 0 || xs >= g.nx || ys < 0 || ys >= g.ny || zs < 0 || zs >= g.nz) {
            atomicOr(status, ST_BOUNDS);
            f[Q] = (C)0.0;
            return;
        }
        f[Q] = PdfStore<T>::template load<C>(src + (long long)Q * g.n + lin(g, xs, ys, zs), Q);
        return;
    }
    if (owner < 0 || owner > np) {
        atomicOr(status, ST_BOUNDS);
        f[Q] = (C)0.0;
        return;
    }
    cut |= 1u << Q;
}

template <typename T, typename C, int Q>
struct MemPull {
    __device__ __forceinline__ static void run(const T* __restrict__ src, const Geom& g,
                                               const DevParticle* parts, int np, const Nbr& b, int x,
                                               int y, int z, long long idx, C (&f)[NQ],
                                               unsigned& cut, int* status) {
        mem_pull_one<T, C, Q>(src, g, parts, np, b, x, y, z, idx, f, cut, status);
        MemPull<T, C, Q + 1>::run(src, g, parts, np, b, x, y, z, idx, f, cut, status);
    }
};
template <typename T, typename C>
struct MemPull<T, C, NQ> {
    __device__ __forceinline__ static void run(const T* __restrict__, const Geom&,
                                               const DevParticle*, int, const Nbr&, int, int, int,
                                               long long, C (&)[NQ], unsigned&, int*) {}
};

// Phase 2: the boundary value f_q(x, t+1) of one cut link (q filled at x,
// qp = qbar the paper's link direction towards the solid cell x + c_qp):
// Eq. (12) BB, Eq. (14) CLI or Eq. (15) MR, and, when `ft` is non-null, the
// link force Eq. (16) and its torque about X_p (arm x_b - X_p) in ft[0..5],
// with the owning particle's 1-based index in *owner_out (0: no force).
template <typename T>
__device__ __forceinline__ double mem_link(const T* __restrict__ src, const Geom& g, const Coupl& cp,
                                        const DevParticle* parts, int np, const GeoMap* gm,
                                        const Nbr& b, int x, int y, int z, long long idx, int q,
                                        double* ft, int* owner_out, int* status, MrCell& mc) {
    if (ft) *owner_out = 0;
    const int qp = opp(q);
    const double cqx = rcx(qp), cqy = rcy(qp), cqz = rcz(qp);  // c_qp
    int xs, ys, zs;
    shifted_rt(b, x, y, z, q, -1, xs, ys, zs);  // x - c_q = x + c_qp, solid
    const int owner = owner_of(g, parts, np, gm, xs, ys, zs);
    if (owner < 1 || owner > np) {
        atomicOr(status, ST_BOUNDS);
        return 0.0;
    }
    const DevParticle& P = parts[owner - 1];
    // every offset from the centre follows from the cell's: x_b - X_p = r + delta c
    double arm[3];
    centre_offset(g, P, x, y, z, arm);
    const double delta = cp.variant == 0 ? 0.5 : link_delta(P, arm, cqx, cqy, cqz, qp <= 6);
    arm[0] += delta * cqx;
    arm[1] += delta * cqy;
    arm[2] += delta * cqz;
    double v[3];
    v[0] = P.u[0] + (P.w[1] * arm[2] - P.w[2] * arm[1]);
    v[1] = P.u[1] + (P.w[2] * arm[0] - P.w[0] * arm[2]);
    v[2] = P.u[2] + (P.w[0] * arm[1] - P.w[1] * arm[0]);
    const double vc = v[0] * cqx + v[1] * cqy + v[2] * cqz;
    const double ftqp = ld_pdf(src + (long long)qp * g.n + idx, qp);  // f~_qp(x)
    const double wr = 3.0 * wq(qp) * cp.rho0;                 // w_q / c_s^2 * rho0
    double val;
    bool cli_done = false;
    if (cp.variant >= 1) {
        // second node x - c_qp = x + c_q must be a fluid cell (CLI and MR)
        int x2, y2, z2;
        shifted_rt(b, x, y, z, q, +1, x2, y2, z2);
        bool ok = !(rcz(q) != 0 && (z2 < 0 || z2 >= g.nz));
        if (ok) ok = owner_of(g, parts, np, gm, x2, y2, z2) == 0;
        if (ok && (x2 < 0 || x2 >= g.nx || y2 < 0 || y2 >= g.ny || z2 < 0 || z2 >= g.nz)) {
            atomicOr(status, ST_BOUNDS);
            ok = false;
        }
        if (ok) {
            const double f2 = ld_pdf(src + (long long)qp * g.n + lin(g, x2, y2, z2), qp);
            const double fq = ld_pdf(src + (long long)q * g.n + idx, q);
            bool mr_done = false;
            if (cp.variant == 2) {
                // Eq. (15): third node x - 2 c_qp = x + 2 c_q must be fluid too
                int x3 = x2 + rcx(q), y3 = y2 + rcy(q), z3 = z2 + rcz(q);
                x3 = x3 < 0 ? x3 + g.nx : (x3 >= g.nx ? x3 - g.nx : x3);
                y3 = y3 < 0 ? y3 + g.ny : (y3 >= g.ny ? y3 - g.ny : y3);
                bool ok3 = true;
                if (g.bc_z) ok3 = z3 >= 0 && z3 < g.nz;
                else z3 = z3 < 0 ? z3 + g.nz : (z3 >= g.nz ? z3 - g.nz : z3);
                if (ok3) ok3 = owner_of(g, parts, np, gm, x3, y3, z3) == 0;
                if (ok3 && (x3 < 0 || x3 >= g.nx || y3 < 0 || y3 >= g.ny || z3 < 0 || z3 >= g.nz)) {
                    atomicOr(status, ST_BOUNDS);
                    ok3 = false;
                }
                if (ok3) {
                    const double f3 = ld_pdf(src + (long long)qp * g.n + lin(g, x3, y3, z3), qp);
                    const double fq2 = ld_pdf(src + (long long)q * g.n + lin(g, x2, y2, z2), q);
                    own_momentum(src, g, idx, mc);
                    const double d1 = 1.0 / ((1.0 + delta) * (1.0 + delta));
                    const double k0 = (1.0 - 2.0 * delta - 2.0 * delta * delta) * d1;
                    const double km1 = delta * delta * d1;
                    const double alpha = 4.0 * d1;
                    // (1 - |lambda_-|) n^-_qp(x, t), rebuilt from the stored values
                    const double odd = 0.5 * (ftqp - fq) -
                                       3.0 * wq(qp) * (cqx * mc.j[0] + cqy * mc.j[1] + cqz * mc.j[2]);
                    val = ftqp + k0 * (f2 - fq) + km1 * (f3 - fq2) - alpha * wr * vc +
                          cp.mr_cpc * d1 * odd;
                    mr_done = true;
                }
            }
            if (!mr_done) {
                const double d1 = 1.0 / (1.0 + 2.0 * delta);
                const double k0 = (1.0 - 2.0 * delta) * d1;
                const double alpha = 4.0 * d1;
                val = ftqp + k0 * f2 - k0 * fq - alpha * wr * vc;
            }
            cli_done = true;
        }
    }
    if (!cli_done) val = ftqp - 2.0 * wr * vc;
    if (ft) {
        double F[3], Tq[3];
        F[0] = (cqx - v[0]) * ftqp - (-cqx - v[0]) * val;
        F[1] = (cqy - v[1]) * ftqp - (-cqy - v[1]) * val;
        F[2] = (cqz - v[2]) * ftqp - (-cqz - v[2]) * val;
        cross3(arm, F, Tq);
        ft[0] = F[0];
        ft[1] = F[1];
        ft[2] = F[2];
        ft[3] = Tq[0];
        ft[4] = Tq[1];
        ft[5] = Tq[2];
        *owner_out = owner;
    }
    return val;
}

template <typename C, int Q>
struct MemMerge {
    __device__ __forceinline__ static void run(unsigned cut, const double (&lv)[NQ], C (&f)[NQ]) {
        if ((cut >> Q) & 1u) f[Q] = (C)lv[Q];
        MemMerge<C, Q + 1>::run(cut, lv, f);
    }
};
template <typename C>
struct MemMerge<C, NQ> {
    __device__ __forceinline__ static void run(unsigned, const double (&)[NQ], C (&)[NQ]) {}
};

// MEM pull for a fluid cell: stream Eq. (2) on every link whose upstream cell
// is fluid (phase 1, unrolled), then the boundary values of the cut links in a
// loop over them (phase 2, one copy of the link code, links in increasing q).
template <typename T, typename C>
__device__ __forceinline__ void mem_pull(const T* __restrict__ src, const Geom& g, const Coupl& cp,
                                         const DevParticle* parts, int np, int x, int y, int z,
                                         long long idx, C (&f)[NQ], int* status) {
    Nbr b = make_nbr(g, x, y, z);
    f[0] = PdfStore<T>::template load<C>(src + idx, 0);
    unsigned cut = 0;
    MemPull<T, C, 1>::run(src, g, parts, np, b, x, y, z, idx, f, cut, status);
    if (cut) {
        double lv[NQ];
        MrCell mc;
        mc.have = false;
        for (unsigned m = cut; m; m &= m - 1) {
            const int q = __ffs(m) - 1;
            int owner = 0;
            lv[q] = mem_link(src, g, cp, parts, np, (const GeoMap*)nullptr, b, x, y, z, idx, q,
                             (double*)nullptr, &owner, status, mc);
        }
        MemMerge<C, 1>::run(cut, lv, f);
    }
}

// Per-warp scratch of the warp-cooperative MEM link loop.
struct LinkWarp {
    double lv[NQ * 32];            // link values, in list order
    double ft[32][6];              // force and torque of the links of one round
    double jt[32][3];              // MR: post-collision momentum of each lane's cell
    long long idx[32];
    int x[32], y[32], z[32], own[32];
    unsigned short list[NQ * 32];  // (lane << 5) | q, lanes in order, q ascending
};

template <typename C, int Q>
struct WarpMerge {
    __device__ __forceinline__ static void run(unsigned cut, const double* lv, int k, C (&f)[NQ]) {
        if ((cut >> Q) & 1u) f[Q] = (C)lv[k++];
        WarpMerge<C, Q + 1>::run(cut, lv, k, f);
    }
};
template <typename C>
struct WarpMerge<C, NQ> {
    __device__ __forceinline__ static void run(unsigned, const double*, int, C (&)[NQ]) {}
};

// Warp-cooperative phase 2 for the near sweep (all 32 lanes call it): the cut
// links of the warp's cells are listed in lane order and spread over the lanes
// 32 at a time, so a boundary cell with many links no longer holds up its
// warp.  Each cell then adds the forces of its own links in ascending q (the
// order of the per-cell loop) and takes its link values.
template <typename T, typename C>
__device__ __forceinline__ void mem_links_warp(const T* __restrict__ src, const Geom& g,
                                               const Coupl& cp, const DevParticle* parts,
                                               const GeoMap* gm, int x, int y, int z, long long idx,
                                               unsigned cut, C (&f)[NQ], Slots& slots, int* status,
                                               LinkWarp& w, int lane) {
    const unsigned full = 0xffffffffu;
    const int nl = __popc(cut);
    int inc = nl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(full, inc, o);
        if (lane >= o) inc += t;
    }
    const int total = __shfl_sync(full, inc, 31);
    if (total == 0) return;  // warp-uniform
    const int first = inc - nl;
    int k = first;
    for (unsigned m = cut; m; m &= m - 1) w.list[k++] = (unsigned short)((lane << 5) | (__ffs(m) - 1));
    w.x[lane] = x;
    w.y[lane] = y;
    w.z[lane] = z;
    w.idx[lane] = idx;
    if (cut && cp.variant == 2) {
        MrCell mc;
        mc.have = false;
        own_momentum(src, g, idx, mc);
        w.jt[lane][0] = mc.j[0];
        w.jt[lane][1] = mc.j[1];
        w.jt[lane][2] = mc.j[2];
    }
    __syncwarp();
    // with no more particles than slots a lane keeps the forces of the links it
    // evaluates; the warp's sum is the same, and no cell can run out of slots
    const bool direct = cp.np <= CELL_SLOTS;
    for (int base = 0; base < total; base += 32) {
        const int e = base + lane;
        if (!direct) w.own[lane] = 0;
        if (e < total) {
            const int ol = w.list[e] >> 5, q = w.list[e] & 31;
            const int lx = w.x[ol], ly = w.y[ol], lz = w.z[ol];
            const Nbr b = make_nbr(g, lx, ly, lz);
            MrCell mc;
            mc.have = cp.variant == 2;
            if (mc.have) {
                mc.j[0] = w.jt[ol][0];
                mc.j[1] = w.jt[ol][1];
                mc.j[2] = w.jt[ol][2];
            }
            double ft[6];
            int own;
            w.lv[e] = mem_link(src, g, cp, parts, cp.np, gm, b, lx, ly, lz, w.idx[ol], q, ft, &own,
                               status, mc);
            if (direct) {
                if (own) {
                    const double F[3] = {ft[0], ft[1], ft[2]}, Tq[3] = {ft[3], ft[4], ft[5]};
                    slots.add(own - 1, F, Tq);
                }
            } else {
#pragma unroll
                for (int c = 0; c < 6; ++c) w.ft[lane][c] = ft[c];
                w.own[lane] = own;
            }
        }
        if (direct) continue;
        __syncwarp();
        // this round's links of this lane's cell: entries [lo, hi)
        const int lo = first > base ? first : base;
        const int hi = (first + nl) < (base + 32) ? (first + nl) : (base + 32);
        for (int e2 = lo; e2 < hi; ++e2) {
            const int s = e2 - base;
            if (w.own[s]) {
                const double F[3] = {w.ft[s][0], w.ft[s][1], w.ft[s][2]};
                const double Tq[3] = {w.ft[s][3], w.ft[s][4], w.ft[s][5]};
                if (!slots.add(w.own[s] - 1, F, Tq)) atomicOr(status, ST_TOO_MANY_OBJECTS);
            }
        }
        __syncwarp();
    }
    __syncwarp();
    WarpMerge<C, 1>::run(cut, w.lv, first, f);
    __syncwarp();
}

// Sums of six values over the warp: halves of the lanes take halves of the
// components first, so that 9 FP64 adds per lane do instead of 30.  Lane 4 c
// (c < 6) returns the sum of component c.
__device__ __forceinline__ double warp_sum6(const double (&v)[6], int lane) {
    const unsigned full = 0xffffffffu;
    double a[4], b[2], s;
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double hi = i < 2 ? v[4 + i] : 0.0;  // components 6 and 7 do not exist
        const double o = __shfl_xor_sync(full, h4 ? v[i] : hi, 16);
        a[i] = (h4 ? hi : v[i]) + o;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const double o = __shfl_xor_sync(full, h3 ? a[i] : a[2 + i], 8);
        b[i] = (h3 ? a[2 + i] : a[i]) + o;
    }
    const double o = __shfl_xor_sync(full, h2 ? b[0] : b[1], 4);
    s = (h2 ? b[1] : b[0]) + o;
    s += __shfl_xor_sync(full, s, 2);
    s += __shfl_xor_sync(full, s, 1);
    return s;
}

// ---------------------------------------------------------------------------
// PSM weighted collision Eq. (26) with C^PSM Eq. (20), B1/B2 Eq. (21)/(22),
// M1/M2/M3 Eq. (23)-(25), force/torque Eq. (28)-(29).  `eps[k]` are the
// solid fractions of particles `pid[k]` (k < nobj) at this cell.  Returns
// true when the cell's fluid density is not finite and positive.
template <typename C>
__device__ inline bool psm_collide(C (&f)[NQ], const Coll<C>& k, const Coupl& cp, const Geom& g,
                                   const DevParticle* parts, int nobj, const int (&pid)[CELL_SLOTS],
                                   const double (&eps)[CELL_SLOTS], int x, int y, int z,
                                   Slots& slots) {
    C Cf[NQ], Fq[NQ], ssum[NQ], feqU[NQ];
    C rho, ux, uy, uz;
    fluid_operator(f, k, Cf, Fq, rho, ux, uy, uz);
    equilibrium(rho, ux, uy, uz, k.rho0, feqU);
#pragma unroll
    for (int q = 0; q < NQ; ++q) ssum[q] = (C)0;
    double B = 0.0;
    const double xc = x + 0.5, yc = y + 0.5, zc = z + 0.5;
    for (int o = 0; o < nobj; ++o) {
        const DevParticle& P = parts[pid[o]];
        const double e = eps[o];
        const double Bs =
            cp.variant == 0 ? e : e * (cp.tau - 0.5) / ((1.0 - e) + (cp.tau - 0.5));
        B += Bs;
        double v[3];
        body_velocity(g, P, xc, yc, zc, v[0], v[1], v[2]);
        C feqV[NQ];
        equilibrium(rho, (C)v[0], (C)v[1], (C)v[2], k.rho0, feqV);
        double Fs[3] = {0.0, 0.0, 0.0};
        const C Bc = (C)Bs;
        const C om = (C)(1.0 - 1.0 / cp.tau);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int qb = opp(q);
            C cs;
            if (cp.variant == 0)
                cs = (f[qb] - feqU[qb]) - (f[q] - feqV[q]);
            else if (cp.variant == 1)
                cs = (feqV[q] - f[q]) + om * (f[q] - feqU[q]);
            else
                cs = (f[qb] - feqV[qb]) - (f[q] - feqV[q]);
            ssum[q] += Bc * cs;
            Fs[0] += (double)cs * cx(qb);
            Fs[1] += (double)cs * cy(qb);
            Fs[2] += (double)cs * cz(qb);
        }
        double F[3] = {Bs * Fs[0], Bs * Fs[1], Bs * Fs[2]}, arm[3], Tq[3];
        separation(g, xc, yc, zc, P, arm[0], arm[1], arm[2]);
        cross3(arm, F, Tq);
        slots.add(pid[o], F, Tq);
    }
    const C oneB = (C)(1.0 - B);
#pragma unroll
    for (int q = 0; q < NQ; ++q) f[q] = f[q] + (oneB * Cf[q] + ssum[q]) + oneB * Fq[q];
    return density_bad(rho);
}

// The FP64 form of psm_collide, written per opposite pair with s = (f_q +
// f_qbar)/2, d = (f_q - f_qbar)/2 and e+-, v+- the even / odd parts of
// f_eq(rho, U) and f_eq(rho, v):
//   fluid  (1 - B) (l+ (s - e+) + F+),  (1 - B) (l- (d - e-) + F-)
//   M1     v+ - e+,                     e- + v- - 2 d
//   M2     v+ - s + om (s - e+),        v- - d + om (d - e-),  om = 1 - 1/tau
//   M3     0,                           2 (v- - d)
// are the even and odd parts of the change (the solid ones times B_s), and
// sum_q C_q c_qbar of Eq. (28) is rho0 (U - v) for M1 and M2, twice that for
// M3.  It is bound by the FP64 pipe: ~300 operations and no arrays over q
// beside f, 154 registers in k_near, against ~700 and 254 of the general form (k_near
// PSM M1B1 D = 8: 35.1 us -> 25.4 us).  FP32 keeps the general form (195
// registers): its time hides under the bulk sweep, though in 16 bits its
// registers are what that sweep lacks beside it (k_bulk_pair).
__device__ inline bool psm_collide64(double (&f)[NQ], const Coll<double>& k, const Coupl& cp,
                                     const Geom& g, const DevParticle* parts, int nobj,
                                     const int (&pid)[CELL_SLOTS], const double (&eps)[CELL_SLOTS],
                                     int x, int y, int z, Slots& slots) {
    using C = double;
    C rho, jx, jy, jz;
    moments_j(f, rho, jx, jy, jz);
    const C ux = jx * k.inv_rho0, uy = jy * k.inv_rho0, uz = jz * k.inv_rho0;
    C vx[CELL_SLOTS], vy[CELL_SLOTS], vz[CELL_SLOTS], bv[CELL_SLOTS], Bs[CELL_SLOTS];
    double B = 0.0;
    const int variant = cp.variant;
    const double fscale = variant == 2 ? 2.0 : 1.0;
#pragma unroll
    for (int o = 0; o < CELL_SLOTS; ++o) {
        vx[o] = vy[o] = vz[o] = bv[o] = Bs[o] = (C)0;
        if (o >= nobj) continue;
        const DevParticle& P = parts[pid[o]];
        const double e = eps[o];
        const double b = variant == 0 ? e : e * (cp.tau - 0.5) / ((1.0 - e) + (cp.tau - 0.5));
        B += b;
        double r[3], v[3];
        centre_offset(g, P, x, y, z, r);
        v[0] = P.u[0] + (P.w[1] * r[2] - P.w[2] * r[1]);
        v[1] = P.u[1] + (P.w[2] * r[0] - P.w[0] * r[2]);
        v[2] = P.u[2] + (P.w[0] * r[1] - P.w[1] * r[0]);
        const double s = b * fscale;
        const double F[3] = {s * ((double)jx - cp.rho0 * v[0]), s * ((double)jy - cp.rho0 * v[1]),
                             s * ((double)jz - cp.rho0 * v[2])};
        double Tq[3];
        cross3(r, F, Tq);
        slots.add(pid[o], F, Tq);
        Bs[o] = (C)b;
        vx[o] = (C)v[0];
        vy[o] = (C)v[1];
        vz[o] = (C)v[2];
        bv[o] = rho - (C)1.5 * k.rho0 * (vx[o] * vx[o] + vy[o] * vy[o] + vz[o] * vz[o]);
    }
    const C oneB = (C)(1.0 - B), om = (C)(1.0 - 1.0 / cp.tau);
    const C olp = oneB * k.lam_p, olm = oneB * k.lam_m;
    const C bu = rho - (C)1.5 * k.rho0 * (ux * ux + uy * uy + uz * uz);
    const C uf = k.has_force ? ux * k.fx + uy * k.fy + uz * k.fz : (C)0;
    // rest direction
    {
        const C w = (C)(1.0 / 3.0), e = w * bu;
        C dp = olp * (f[0] - e);
        if (k.has_force) dp -= oneB * uf;
#pragma unroll
        for (int o = 0; o < CELL_SLOTS; ++o) {
            if (o >= nobj) continue;
            const C v = w * bv[o];
            if (variant == 0) dp += Bs[o] * (v - e);
            else if (variant == 1) dp += Bs[o] * ((v - f[0]) + om * (f[0] - e));
        }
        f[0] += dp;
    }
#pragma unroll
    for (int q = 1; q < NQ; q += 2) {
        const C w = (C)wq(q);
        const C k1 = (C)(4.5 * wq(q)) * k.rho0, k2 = (C)(3.0 * wq(q)) * k.rho0;
        const auto dot = [&](C ax, C ay, C az) {
            C d = (C)0;
            if (cx(q)) d = cx(q) > 0 ? ax : -ax;
            if (cy(q)) d = cx(q) ? (cy(q) > 0 ? d + ay : d - ay) : ay;
            if (cz(q)) d = cx(q) || cy(q) ? (cz(q) > 0 ? d + az : d - az) : az;
            return d;
        };
        const C s = (C)0.5 * (f[q] + f[q + 1]), d = (C)0.5 * (f[q] - f[q + 1]);
        const C cu = dot(ux, uy, uz);
        const C ep = w * bu + (k1 * cu) * cu, em = k2 * cu;
        C dp = olp * (s - ep), dm = olm * (d - em);
        if (k.has_force) {
            const C cf = dot(k.fx, k.fy, k.fz);
            dp += oneB * (w * ((C)9 * cu * cf - (C)3 * uf));
            dm += oneB * ((C)3 * w * cf);
        }
#pragma unroll
        for (int o = 0; o < CELL_SLOTS; ++o) {
            if (o >= nobj) continue;
            const C cv = dot(vx[o], vy[o], vz[o]);
            const C vm = k2 * cv;
            if (variant == 2) {
                dm += Bs[o] * ((C)2 * (vm - d));
                continue;
            }
            const C vp = w * bv[o] + (k1 * cv) * cv;
            if (variant == 0) {
                dp += Bs[o] * (vp - ep);
                dm += Bs[o] * ((em + vm) - (C)2 * d);
            } else {
                dp += Bs[o] * ((vp - s) + om * (s - ep));
                dm += Bs[o] * ((vm - d) + om * (d - em));
            }
        }
        f[q] += dp + dm;
        f[q + 1] += dp - dm;
    }
    return density_bad(rho);
}

// ---------------------------------------------------------------------------
// bulk sweep: every cell outside the near-particle regions.  Tiles that no
// region touches skip the per-cell test (block-uniform branch).
// Threads per block and resident blocks per SM of k_bulk by stored type and
// arithmetic (the host's tiles, set_tiles in lbm_launch.h, follow).  FP64:
// 5 x 128 threads leave the fixed-point collision 96 registers (8 B of stack,
// 4 B of them spills) and 20 warps per SM (128 x 128 x 512 cells, FP64 settling step of 2
// sweeps: 256 x 3, 80 registers, 1.27 ms; 256 x 2, 128 registers, 1.38;
// 128 x 4 1.29; 128 x 5 1.09; 128 x 6 1.21; 128 x 7 1.18).  16 bits, one
// cell per thread: 128 threads balance the last wave better (101 x 101 x 304
// cells, frame step 296 -> 259 us).  FP32 keeps 256 (0.5 % faster).
template <typename T, typename C> struct BulkShape { static constexpr int threads = 128, blocks = 6; };
template <> struct BulkShape<double, double> { static constexpr int threads = 128, blocks = 5; };
template <> struct BulkShape<float, float> { static constexpr int threads = 256, blocks = 3; };

// One tile (tX, tY, tZ) of the bulk sweep for the calling thread (tx, ty).
template <typename T, typename C, bool NOSTREAM, int CPT>
__device__ __forceinline__ void bulk_tile(const T* __restrict__ src, T* __restrict__ dst,
                                          const Geom& g, const Coll<C>& k,
                                          const DevParticle* __restrict__ parts, int np,
                                          int all_tiles, int tX, int tY, int tZ, int tx, int ty,
                                          int* __restrict__ status) {
    bool near_tile = false;
    if (!all_tiles) {
        for (int s = 0; s < np && !near_tile; ++s)
            near_tile = tile_in_reg(g, parts[s].reg, tX, tY, tZ);
    }
    const int x = tX * g.tx + tx, y = tY * g.ty + ty;
    if (x >= g.nx || y >= g.ny) return;
    // CPT cells per thread along z: all their loads are issued before the
    // first collision, doubling the bytes in flight of the 32-bit sweep
    C f[CPT][NQ];
    bool act[CPT];
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const int z = tZ * CPT + c;
        act[c] = z < g.nz;
        if (act[c] && near_tile)
            for (int s = 0; s < np; ++s)
                if (cell_in_reg(g, parts[s].reg, x, y, z)) act[c] = false;  // k_near's cell
        if (act[c]) {
            const long long idx = lin(g, x, y, z);
            if (NOSTREAM)
                load_own(src, g, idx, f[c]);
            else
                pull_plain(src, g, x, y, z, idx, f[c]);
        }
    }
    bool bad = false;
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        if (!act[c]) continue;
        const int z = tZ * CPT + c;
        bad |= collide_cell(f[c], k);
        store_own(dst, g, lin(g, x, y, z), f[c]);
    }
    if (bad) atomicOr(status, ST_FLUID);
}

// GATE: the form that runs beside k_near (gate_pass); the others are launched
// plainly and carry none of its code but, in FP32, gate_leave (null gate, no
// effect): ptxas makes a faster kernel with a branch at its end (128 x 128 x 512 MEM
// with charge, 8 steps 4082 us without, 3890 with; FP64 MEM MR, 4 steps 4265 without,
// 4331 with).
template <typename T, typename C, bool NOSTREAM, int CPT, bool GATE>
__global__ void __launch_bounds__(BulkShape<T, C>::threads, BulkShape<T, C>::blocks)
    k_bulk(const T* __restrict__ src, T* __restrict__ dst, Geom g, Coll<C> k,
           const DevParticle* __restrict__ parts, int np, int all_tiles, int* __restrict__ status,
           const int* gate, int key) {
    if constexpr (GATE) {
        if (!gate_pass(gate, key)) {
            if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(status, ST_BOUNDS);
            gate_leave(gate);
            return;
        }
        src = entered(src);
        parts = entered(parts);
    }
    bulk_tile<T, C, NOSTREAM, CPT>(src, dst, g, k, parts, np, all_tiles, blockIdx.x, blockIdx.y,
                                   blockIdx.z, threadIdx.x, threadIdx.y, status);
    if constexpr (GATE || sizeof(T) == 4) gate_leave(gate);
}

// ---------------------------------------------------------------------------
// 16-bit shifted storage, two x-neighbours per thread.  The pair (x0, x0 + 1),
// x0 even, is read and written as one 32-bit word per direction (nx even, so
// every row starts on a 4-byte boundary); a pull across x takes the two
// aligned words around the shifted pair and selects its halves with a byte
// permute.  Conversions use the packed two-value forms.  The collision runs on
// the stored shifted values g_q = f_q - w_q themselves: with rho = 1 + sum_q
// g_q and j = sum_q g_q c_q (sum_q w_q c_q = 0), the folded update
// f' = alpha f + beta fbar - (P +- M) becomes g' = alpha g + beta gbar -
// (P +- M) with rho replaced by sum_q g_q in P (alpha + beta - 1 = lambda_+
// cancels the l+ w_q term), so the same collide_fluid code applies with no
// shift on load or store, and FP32 rounds the small deviations, not f.
template <typename T> struct Pair16;
template <>
struct Pair16<__half> {
    __device__ __forceinline__ static float2 unpack(unsigned u) {
        __half2 h;
        memcpy(&h, &u, 4);
        return __half22float2(h);
    }
    __device__ __forceinline__ static unsigned pack(float a, float b) {
        const __half2 h = __floats2half2_rn(a, b);
        unsigned u;
        memcpy(&u, &h, 4);
        return u;
    }
    __device__ __forceinline__ static __half one(float a) { return __float2half_rn(a); }
};
template <>
struct Pair16<__nv_bfloat16> {
    __device__ __forceinline__ static float2 unpack(unsigned u) {
        __nv_bfloat162 h;
        memcpy(&h, &u, 4);
        return __bfloat1622float2(h);
    }
    __device__ __forceinline__ static unsigned pack(float a, float b) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        unsigned u;
        memcpy(&u, &h, 4);
        return u;
    }
    __device__ __forceinline__ static __nv_bfloat16 one(float a) { return __float2bfloat16_rn(a); }
};

__device__ __forceinline__ unsigned ld_word(const void* p) {
    return __ldg(reinterpret_cast<const unsigned*>(p));
}

// direction Q of the pair at row `row` (= lin(0, y, z)); xm2 / xp2 are the
// (periodic) even columns left / right of x0
template <typename T, int Q>
__device__ __forceinline__ void pull_pair_one(const T* __restrict__ src, const Geom& g,
                                              const NbrOff& o, long long row, int x0, int xm2,
                                              int xp2, f2 (&f)[NQ]) {
    float2 v;
    if ((cz(Q) > 0 && o.zlo) || (cz(Q) < 0 && o.zhi)) {
        v = Pair16<T>::unpack(ld_word(src + (long long)opp(Q) * g.n + row + x0));  // halfway BB
    } else {
        long long r = row;
        if (cy(Q) > 0) r += o.dym;
        else if (cy(Q) < 0) r += o.dyp;
        if (cz(Q) > 0) r += o.dzm;
        else if (cz(Q) < 0) r += o.dzp;
        const T* a = src + (long long)Q * g.n + r;
        if (cx(Q) == 0) {
            v = Pair16<T>::unpack(ld_word(a + x0));
        } else if (cx(Q) > 0) {  // cells x0 - 1, x0
            v = Pair16<T>::unpack(__byte_perm(ld_word(a + xm2), ld_word(a + x0), 0x5432));
        } else {  // cells x0 + 1, x0 + 2
            v = Pair16<T>::unpack(__byte_perm(ld_word(a + x0), ld_word(a + xp2), 0x5432));
        }
    }
    f[Q] = f2(v);  // shifted values g_q (see above), cell x0 in lane x
}

template <typename T, int Q>
struct PullPair {
    __device__ __forceinline__ static void run(const T* __restrict__ src, const Geom& g,
                                               const NbrOff& o, long long row, int x0, int xm2,
                                               int xp2, f2 (&f)[NQ]) {
        pull_pair_one<T, Q>(src, g, o, row, x0, xm2, xp2, f);
        PullPair<T, Q + 1>::run(src, g, o, row, x0, xm2, xp2, f);
    }
};
template <typename T>
struct PullPair<T, NQ> {
    __device__ __forceinline__ static void run(const T* __restrict__, const Geom&, const NbrOff&,
                                               long long, int, int, int, f2 (&)[NQ]) {}
};

// Grid (ceil(nx / (2 W)), ny, nz), one row segment per block of W = 64, 96 or 32
// threads, whichever leaves the fewest beyond the row's end (pair_width: 192
// cells per row are 96 threads; as two blocks of 64, a quarter of them idle,
// the BF16 sweep of 192 x 192 x 768 cells took 473 us, 0.67 of HBM, and takes
// 376 us, 0.85).  One row of 128 cells per 64-thread block: the near-particle sweep runs
// beside this kernel and each of its one-warp blocks holds 3.1k (MEM) to 6.2k (PSM)
// registers; with small bulk blocks an SM that hosts near blocks gives up
// only as many bulk warps as their registers need (measured in the 128 x 128
// x 512 step, FP16: 0.70 of HBM with 64 x 4, 0.745 with 64 x 2, 0.76 with
// 64 x 1; 32 x 1 and 128 x 1 are slower).
inline int pair_width(int nx) {
    const int pairs = nx / 2;
    int best = 64;
    const auto waste = [&](int w) { return (pairs + w - 1) / w * w; };
    if (waste(96) < waste(best)) best = 96;
    if (waste(32) < waste(best)) best = 32;
    return best;
}

template <typename T, int W>
__global__ void __launch_bounds__(W, 768 / W)
    k_bulk_pair(const T* __restrict__ src, T* __restrict__ dst, Geom g, Coll<float> k,
                const DevParticle* __restrict__ parts, int np, int* __restrict__ status) {
    const int bx0 = 2 * blockIdx.x * W, y = blockIdx.y, z = blockIdx.z;
    const int x0 = bx0 + 2 * threadIdx.x;
    if (x0 >= g.nx) return;
    // k_near's cells are left alone; a block whose cells no region reaches
    // (block-uniform test) skips the per-cell one
    bool near_a = false, near_b = false;
    for (int s = 0; s < np; ++s) {
        const int* r = parts[s].reg;
        if (!in_range(z, r[8], r[9], g.nz) ||
            !in_range(y, r[4], r[5], g.ny) ||
            !spans_meet(bx0, min(2 * W, g.nx - bx0), r[0], r[1], g.nx))
            continue;
        near_a = near_a || cell_in_reg(g, r, x0, y, z);
        near_b = near_b || cell_in_reg(g, r, x0 + 1, y, z);
    }
    if (near_a && near_b) return;
    const NbrOff o = make_off(g, x0, y, z);
    const long long row = lin(g, 0, y, z);
    const int xm2 = x0 == 0 ? g.nx - 2 : x0 - 2;
    const int xp2 = x0 + 2 == g.nx ? 0 : x0 + 2;
    // both cells collide in the two lanes of the packed f32x2 arithmetic
    f2 f[NQ];
    PullPair<T, 0>::run(src, g, o, row, x0, xm2, xp2, f);
    const unsigned bad = collide_fluid<f2, true>(f, k);
    if (((bad & 1u) && !near_a) || ((bad & 2u) && !near_b)) atomicOr(status, ST_FLUID);
    if (!near_a && !near_b) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            *reinterpret_cast<unsigned*>(dst + (long long)q * g.n + row + x0) =
                Pair16<T>::pack(f[q].v.x, f[q].v.y);
    } else {
        const long long idx = row + x0 + (near_a ? 1 : 0);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            dst[(long long)q * g.n + idx] = Pair16<T>::one(near_a ? f[q].v.y : f[q].v.x);
    }
}

// 16-bit shifted storage where rows cannot be taken as aligned words (odd nx)
// or the boundary planes have their own rules (open boundaries): each thread
// takes the cells z and z + 1 of one column, with 2-byte accesses, and collides
// them in the two lanes of the packed arithmetic.  The weights are added to the
// populations before and taken off after it, operation for operation as the
// scalar FP32 form does, so every lane's result has its bits.  One cell per thread in scalar FP32 was bound by issue
// (565 instructions per cell, 0.34 of HBM); this form halves the arithmetic
// and the addresses: 101 x 101 x 304 cells FP16 85 us -> 73 us (k_near beside
// it), 440 instructions per 64 cells, issue 57 %.
template <typename T>
__device__ __forceinline__ float raw16(const T* p);
template <>
__device__ __forceinline__ float raw16<__half>(const __half* p) {
    return __half2float(__ldg(p));
}
template <>
__device__ __forceinline__ float raw16<__nv_bfloat16>(const __nv_bfloat16* p) {
    return __bfloat162float(__ldg(p));
}
template <typename T, int Q>
struct PullRaw {
    __device__ __forceinline__ static void run(const T* __restrict__ src, const Geom& g,
                                               const NbrOff& o, long long idx, float (&f)[NQ]) {
        if ((cz(Q) > 0 && o.zlo) || (cz(Q) < 0 && o.zhi))
            f[Q] = raw16(src + (long long)opp(Q) * g.n + idx);
        else
            f[Q] = raw16(src + (long long)Q * g.n + idx + upstream_off<Q>(o));
        PullRaw<T, Q + 1>::run(src, g, o, idx, f);
    }
};
template <typename T>
struct PullRaw<T, NQ> {
    __device__ __forceinline__ static void run(const T* __restrict__, const Geom&, const NbrOff&,
                                               long long, float (&)[NQ]) {}
};

// Blocks are runs of 128 cells of a plane, x fastest (row tiles of 64 left a
// fifth of the lanes of a 101-cell row idle).
constexpr int ZPAIR_THREADS = 128, ZPAIR_BLOCKS = 5;
template <typename T>
__global__ void __launch_bounds__(ZPAIR_THREADS, ZPAIR_BLOCKS)
    k_bulk_zpair(const T* __restrict__ src, T* __restrict__ dst, Geom g, Coll<float> k,
                 const DevParticle* __restrict__ parts, int np, int* __restrict__ status) {
    const unsigned l = blockIdx.x * ZPAIR_THREADS + threadIdx.x;
    if (l >= (unsigned)g.nx * (unsigned)g.ny) return;
    const int y = l / (unsigned)g.nx, x = l - (unsigned)y * g.nx, z = 2 * blockIdx.z;
    bool act0 = true, act1 = z + 1 < g.nz;
    for (int s = 0; s < np; ++s) {  // k_near's cells
        const int* r = parts[s].reg;
        if (!in_range(x, r[0], r[1], g.nx) || !in_range(y, r[4], r[5], g.ny)) continue;
        act0 = act0 && !in_range(z, r[8], r[9], g.nz);
        act1 = act1 && !in_range(z + 1, r[8], r[9], g.nz);
    }
    if (!act0 && !act1) return;
    const long long idx = lin(g, x, y, z), plane = (long long)g.nx * g.ny;
    float a[NQ], b[NQ];
    f2 f[NQ];
    if (g.bc_z == 2 && (z == 0 || z + 2 >= g.nz)) {  // a boundary plane (block-uniform)
        if (act0) pull_plain(src, g, x, y, z, idx, a);
        if (act1) pull_plain(src, g, x, y, z + 1, idx + plane, b);
#pragma unroll
        for (int q = 0; q < NQ; ++q) f[q] = f2(make_float2(act0 ? a[q] : 0.0f, act1 ? b[q] : 0.0f));
    } else {
        if (act0) PullRaw<T, 0>::run(src, g, make_off(g, x, y, z), idx, a);
        if (act1) PullRaw<T, 0>::run(src, g, make_off(g, x, y, z + 1), idx + plane, b);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            f[q] = f2(make_float2(act0 ? a[q] : 0.0f, act1 ? b[q] : 0.0f)) + f2((float)wq(q));
    }
    const unsigned bad = collide_fluid<f2>(f, k);
    if (((bad & 1u) && act0) || ((bad & 2u) && act1)) atomicOr(status, ST_FLUID);
#pragma unroll
    for (int q = 0; q < NQ; ++q) f[q] = f[q] - f2((float)wq(q));
    if (act0)
#pragma unroll
        for (int q = 0; q < NQ; ++q) dst[(long long)q * g.n + idx] = Pair16<T>::one(f[q].v.x);
    if (act1)
#pragma unroll
        for (int q = 0; q < NQ; ++q) dst[(long long)q * g.n + idx + plane] = Pair16<T>::one(f[q].v.y);
}

// ---------------------------------------------------------------------------
// MEM: a cell whose centre lies farther than R + 3/2 from every sphere centre
// has no solid neighbour (neighbour centres are at most sqrt(2) away and a
// cell is solid iff its centre is within R, R6), so its pull is the plain one.
__device__ __forceinline__ bool clear_of_particles(const Geom& g, const DevParticle* sp, int np,
                                                   int x, int y, int z) {
    for (int s = 0; s < np; ++s) {
        const float r = (float)sp[s].r + 1.5f;
        if (!(cell_offset(g, sp[s], x, y, z).d2() > r * r + margin_f(r))) return false;
    }
    return true;
}

// Phase 1 of the MEM pull for a cell at offsets (kx, ky, kz) of particle p's
// region box, owners from the box's map: `own` collects the directions whose
// upstream cell is solid, `wall` those that cross a closed wall.  All 18 map
// entries are loaded before the first is used, then all PDFs: the pull is two
// memory latencies long instead of one per direction (with the link terms from
// one centre offset: k_near MEM CLI, D = 8 FP64 32.7 us -> 23.7 us, D = 24
// FP32 37.7 -> 31.9).  A neighbour outside the
// box is fluid for one particle (the box holds every cell within two of the
// sphere's surface); with more it is looked up in the other boxes.
template <int Q>
struct NearOwners {
    __device__ __forceinline__ static void run(const Geom& g, const DevParticle* sp, int np,
                                               const GeoMap& gm, const unsigned short* m0,
                                               const NbrOff& o, unsigned in, int x, int y, int z,
                                               unsigned short (&e)[NQ], unsigned& wall) {
        // bits of `in`: x - 1, x + 1, y - 1, y + 1, z - 1, z + 1 lie in the box
        constexpr int dx = -cx(Q), dy = -cy(Q), dz = -cz(Q);
        constexpr unsigned need = (dx < 0 ? 1u : dx > 0 ? 2u : 0u) | (dy < 0 ? 4u : dy > 0 ? 8u : 0u) |
                                  (dz < 0 ? 16u : dz > 0 ? 32u : 0u);
        e[Q] = 0;
        if ((dz < 0 && o.zlo) || (dz > 0 && o.zhi)) {
            wall |= 1u << Q;
        } else if ((in & need) == need) {
            e[Q] = __ldg(m0 + (dx + gm.ex * (dy + (long long)gm.ey * dz)));
        } else if (np > 1) {
            const Nbr b = make_nbr(g, x, y, z);
            int xs, ys, zs;
            shifted<Q>(b, x, y, z, -1, xs, ys, zs);
            e[Q] = (unsigned short)mapped_owner(g, sp, np, gm, xs, ys, zs);
        }
        NearOwners<Q + 1>::run(g, sp, np, gm, m0, o, in, x, y, z, e, wall);
    }
};
template <>
struct NearOwners<NQ> {
    __device__ __forceinline__ static void run(const Geom&, const DevParticle*, int, const GeoMap&,
                                               const unsigned short*, const NbrOff&, unsigned, int,
                                               int, int, unsigned short (&)[NQ], unsigned&) {}
};
template <typename T, typename C, int Q>
struct NearPull {
    __device__ __forceinline__ static void run(const T* __restrict__ src, const Geom& g,
                                               const NbrOff& o, long long idx, unsigned solid,
                                               unsigned wall, C (&f)[NQ]) {
        if ((wall >> Q) & 1u)
            f[Q] = PdfStore<T>::template load<C>(src + (long long)opp(Q) * g.n + idx, opp(Q));
        else if (!((solid >> Q) & 1u))
            f[Q] = PdfStore<T>::template load<C>(src + (long long)Q * g.n + idx + upstream_off<Q>(o), Q);
        NearPull<T, C, Q + 1>::run(src, g, o, idx, solid, wall, f);
    }
};
template <typename T, typename C>
struct NearPull<T, C, NQ> {
    __device__ __forceinline__ static void run(const T* __restrict__, const Geom&, const NbrOff&,
                                               long long, unsigned, unsigned, C (&)[NQ]) {}
};
template <typename T, typename C>
__device__ __forceinline__ bool near_pull(const T* __restrict__ src, const Geom& g,
                                          const DevParticle* sp, int np, const GeoMap& gm, int p,
                                          int kx, int ky, int kz, int x, int y, int z,
                                          long long idx, C (&f)[NQ], unsigned& cut, int* status) {
    if (kx >= gm.ex || ky >= gm.ey || kz >= gm.ez) {  // a box larger than its map: report, no access
        atomicOr(status, ST_BOUNDS);
        return false;  // (the caller stores no cell that was not pulled)
    }
    f[0] = PdfStore<T>::template load<C>(src + idx, 0);
    const int* R = sp[p].reg;
    const unsigned in = (kx > 0 ? 1u : 0u) | (kx + 1 < min(R[1], gm.ex) ? 2u : 0u) |
                        (ky > 0 ? 4u : 0u) | (ky + 1 < min(R[5], gm.ey) ? 8u : 0u) |
                        (kz > 0 ? 16u : 0u) | (kz + 1 < min(R[9], gm.ez) ? 32u : 0u);
    const NbrOff o = make_off(g, x, y, z);
    const unsigned short* m0 = gm.map + (((long long)p * gm.ez + kz) * gm.ey + ky) * gm.ex + kx;
    unsigned short e[NQ];
    unsigned wall = 0;
    NearOwners<1>::run(g, sp, np, gm, m0, o, in, x, y, z, e, wall);
    unsigned solid = 0;
#pragma unroll
    for (int q = 1; q < NQ; ++q) solid |= e[q] ? 1u << q : 0u;
    NearPull<T, C, 1>::run(src, g, o, idx, solid, wall, f);
    cut = solid;
    return true;
}

// Cell of a lane of near block blk, as offsets in the region R; false beyond it.
// PSM: 32 consecutive cells of the region.  MEM: four runs of 8 cells, a
// quarter of the region apart: the cut links lie in a thin shell and are taken
// 32 at a time, so a warp should not hold many more than the others.  Region cells
// number less than 2^32: the two buffers of a larger lattice fit no memory.
template <int KIND>
__device__ __forceinline__ bool near_cell(const int* R, long long blk, int lane, int& kx, int& ky,
                                          int& kz) {
    const unsigned ex = R[1], ey = R[5], total = ex * ey * (unsigned)R[9];
    const unsigned runs = (total + 7) / 8, used = KIND == 2 ? (runs + 3) / 4 : (total + 31) / 32;
    const unsigned b = (unsigned)blk;
    const unsigned l = KIND == 2 ? (b + (lane >> 3) * used) * 8 + (lane & 7) : b * 32 + lane;
    const bool in = b < used && l < total;
    const unsigned row = in ? l / ex : 0u, plane = in ? row / ey : 0u;
    kx = in ? (int)(l - row * ex) : 0;
    ky = (int)(row - plane * ey);
    kz = (int)plane;
    return in;
}

// One near-kernel block: block blk of particle p, whose force/torque sums on
// every particle q land in partials[((p * nblk + blk) * np + q) * 6 + c] (the
// warp's sum, fixed order).  `sp` holds the particle records in shared memory;
// all 32 lanes call it.
template <typename T, typename C, int KIND, bool NOSTREAM, typename LW>
__device__ __forceinline__ void near_block(const T* __restrict__ src, T* __restrict__ dst,
                                           const Geom& g, const Coll<C>& k, const Coupl& cp,
                                           const DevParticle* sp, const GeoMap& gm,
                                           double* __restrict__ partials, int* __restrict__ status,
                                           int p, long long nblk, long long blk, LW& lw) {
    const int lane = threadIdx.x;
    const int* R = sp[p].reg;
    int kx, ky, kz;
    bool active = near_cell<KIND>(R, blk, lane, kx, ky, kz);
    if (blk == 0 && lane == 0 && (long long)R[1] * R[5] * R[9] > nblk * NEAR_THREADS)
        atomicOr(status, ST_BOUNDS);  // a region larger than its grid
    int x = R[0] + kx, y = R[4] + ky, z = R[8] + kz;
    if (x >= g.nx) x -= g.nx;
    if (y >= g.ny) y -= g.ny;
    if (z >= g.nz) z -= g.nz;
    if (active)
        for (int s = 0; s < p; ++s)
            if (cell_in_reg(g, sp[s].reg, x, y, z)) active = false;
    Slots slots;
    slots.clear();
    if (active && (x < 0 || x >= g.nx || y < 0 || y >= g.ny || z < 0 || z >= g.nz)) {
        atomicOr(status, ST_BOUNDS);
        active = false;
    }
    if (KIND != 2) {
        C f[NQ];
        int nobj = 0;
        int pid[CELL_SLOTS];
        double eps[CELL_SLOTS];
        const long long idx = active ? lin(g, x, y, z) : 0;
        if (active) {
            if (NOSTREAM)
                load_own(src, g, idx, f);
            else
                pull_plain(src, g, x, y, z, idx, f);
            if (KIND == 1) {
                const double n3 = (double)cp.subsample * cp.subsample * cp.subsample;
                for (int s = 0; s < cp.np; ++s) {
                    int ox, oy, oz;
                    if (!region_offsets(g, sp[s].reg, x, y, z, ox, oy, oz)) continue;
                    const int cnt = map_at(gm, s, ox, oy, oz);
                    if (cnt == 0) continue;
                    const double e = (double)cnt / n3;
                    if (nobj < CELL_SLOTS) {
                        pid[nobj] = s;
                        eps[nobj] = e;
                        ++nobj;
                    } else {
                        atomicOr(status, ST_TOO_MANY_OBJECTS);
                    }
                }
            }
        }
        if constexpr (std::is_same<C, double>::value) {
            // a warp with any covered cell takes the PSM form for all of them
            // (B = 0 is the fluid collision), so that it runs one form, not two
            const bool coupled = KIND == 1 && __any_sync(0xffffffffu, nobj > 0);
            if (active) {
                const bool bad = coupled ? psm_collide64(f, k, cp, g, sp, nobj, pid, eps, x, y, z, slots)
                                         : collide_cell(f, k);
                if (bad) atomicOr(status, ST_FLUID);
            }
        } else if (active) {
            const bool bad = nobj == 0
                                 ? collide_fluid(f, k)
                                 : psm_collide(f, k, cp, g, sp, nobj, pid, eps, x, y, z, slots);
            if (bad) atomicOr(status, ST_FLUID);
        }
        if (active) store_own(dst, g, idx, f);
    }
    if constexpr (KIND == 2) {
        // MEM (Sec. 2.2): solid cells are not updated; every lane of the warp
        // takes part in the link loop, cells or not
        C f[NQ];
        bool fluid = false;
        long long idx = 0;
        unsigned cut = 0;
        if (active && !map_at(gm, p, kx, ky, kz)) {
            fluid = true;
            idx = lin(g, x, y, z);
            if (clear_of_particles(g, sp, cp.np, x, y, z)) {
                pull_plain(src, g, x, y, z, idx, f);  // no solid neighbour, no link
            } else {
                fluid = near_pull(src, g, sp, cp.np, gm, p, kx, ky, kz, x, y, z, idx, f, cut, status);
            }
        }
        mem_links_warp(src, g, cp, sp, &gm, x, y, z, idx, cut, f, slots, status, lw, lane);
        if (fluid) {
            if (collide_cell(f, k)) atomicOr(status, ST_FLUID);
            store_own(dst, g, idx, f);
        }
    }
    if (KIND == 0) return;
    // fixed-order reduction of this block's contribution for each particle
    const bool any = __any_sync(0xffffffffu, slots.id[0] >= 0);
    if (p >= cp.np || blk >= nblk) {
        if (lane == 0) atomicOr(status, ST_BOUNDS);
        return;
    }
    for (int q = 0; q < cp.np; ++q) {
        double s = 0.0;
        if (any) {  // (else no cell of this warp feels a force)
            double v[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) v[c] = slots.get(q, c);
            s = warp_sum6(v, lane);
        }
        if ((lane & 3) == 0 && lane < 24)
            partials[(((long long)p * nblk + blk) * cp.np + q) * 6 + (lane >> 2)] = s;
    }
}

// ---------------------------------------------------------------------------
// near-particle sweep over the cell region of each particle (cells within
// R + NEAR_HALO of the centre per axis).  Grid (near_nblk, np), a warp per
// block; a cell that also lies in the region of a lower-index particle is left
// to that particle's blocks.  The particle records are staged in shared memory
// (dynamic: np records).
template <typename T, typename C, int KIND, bool NOSTREAM>
__global__ void __launch_bounds__(NEAR_THREADS)
    k_near(const T* __restrict__ src, T* __restrict__ dst, Geom g, Coll<C> k, Coupl cp,
           const DevParticle* __restrict__ parts, GeoMap gm, double* __restrict__ partials,
           int* __restrict__ status, int* gate, int key) {
    extern __shared__ double sp_words[];
    __shared__ typename std::conditional<KIND == 2, LinkWarp, char>::type lw;
    step_wait();
    gate_open(gate, key);
    step_trigger();
    parts = entered(parts);
    src = entered(src);
    gm.map = entered(gm.map);
    for (int i = threadIdx.x; i < cp.np * (int)(sizeof(DevParticle) / sizeof(double)); i += NEAR_THREADS)
        sp_words[i] = reinterpret_cast<const double*>(parts)[i];
    __syncwarp();
    near_block<T, C, KIND, NOSTREAM>(src, dst, g, k, cp,
                                     reinterpret_cast<const DevParticle*>(sp_words), gm, partials,
                                     status, blockIdx.y, gridDim.x, blockIdx.x, lw);
}

// One sweep of a small lattice (FP64 or FP32 PDFs, MEM or PSM) in one launch:
// blocks 0 .. nblk * np - 1 are k_near's, the others take 32 consecutive cells of
// the lattice each, as k_bulk collides them, and skip k_near's cells.  Where the
// bulk cells are done before the chain of a near block is (SWEEP_FUSED_CELLS),
// a second stream beside it only adds its fork and join to the step.
template <typename T, typename C, int KIND>
__global__ void __launch_bounds__(NEAR_THREADS)
    k_sweep(const T* __restrict__ src, T* __restrict__ dst, Geom g, Coll<C> k, Coupl cp,
            const DevParticle* __restrict__ parts, GeoMap gm, double* __restrict__ partials,
            int* __restrict__ status, unsigned nblk) {
    extern __shared__ double sp_words[];
    __shared__ typename std::conditional<KIND == 2, LinkWarp, char>::type lw;
    step_enter();
    parts = entered(parts);
    src = entered(src);
    gm.map = entered(gm.map);
    for (int i = threadIdx.x; i < cp.np * (int)(sizeof(DevParticle) / sizeof(double)); i += NEAR_THREADS)
        sp_words[i] = reinterpret_cast<const double*>(parts)[i];
    __syncwarp();
    const DevParticle* sp = reinterpret_cast<const DevParticle*>(sp_words);
    const unsigned nnear = nblk * cp.np;
    if (blockIdx.x < nnear) {
        near_block<T, C, KIND, false>(src, dst, g, k, cp, sp, gm, partials, status,
                                      blockIdx.x / nblk, nblk, blockIdx.x % nblk, lw);
        return;
    }
    const unsigned idx = (blockIdx.x - nnear) * NEAR_THREADS + threadIdx.x;
    if (idx >= (unsigned)g.n) return;
    const unsigned row = idx / g.nx;
    const int x = (int)(idx - row * g.nx), z = (int)(row / g.ny), y = (int)(row - z * g.ny);
    for (int s = 0; s < cp.np; ++s)
        if (cell_in_reg(g, sp[s].reg, x, y, z)) return;
    C f[NQ];
    pull_plain(src, g, x, y, z, (long long)idx, f);
    if (collide_cell(f, k)) atomicOr(status, ST_FLUID);
    store_own(dst, g, (long long)idx, f);
}

// ---------------------------------------------------------------------------
// Per-step geometry map (computed once per global step, before the sweeps):
// for every cell of particle p's region, MEM: the owner under the current
// particle state (0 fluid, s+1 inside particle s, lowest s first, R6);
// PSM: the number of the n^3 supersamples inside particle p (R15).  The
// sweeps then read these instead of re-evaluating FP64 geometry per link.
// Grid (ceil(ex/32), ey, ez * np), 32 threads per block.
// Called by all 32 lanes of a warp that covers 32 consecutive kx of one row
// (ky, kz the same on every lane).  PSM: cells wholly outside or inside the
// sphere take the quick count; the warp then samples each remaining cell of
// the row together (two of the 64 samples per lane for n = 4), so a row costs
// a few cooperative sample sets instead of one 64-sample loop per lane.  The
// samples are decided in FP32 wherever that can tell (inside_f): D = 8, n = 4
// 18.1 us -> 5.7 us.
template <int KIND>
__device__ __forceinline__ void map_cell(const Geom& g, const Coupl& cp, const DevParticle* sp,
                                         unsigned short* __restrict__ map, int ex, int ey, int ez,
                                         int p, int kx, int ky, int kz) {
    const int* R = sp[p].reg;
    const bool valid = kx < R[1] && ky < R[5] && kz < R[9];
    int x = R[0] + kx, y = R[4] + ky, z = R[8] + kz;
    if (x >= g.nx) x -= g.nx;
    if (y >= g.ny) y -= g.ny;
    if (z >= g.nz) z -= g.nz;
    unsigned short* out = map + (((long long)p * ez + kz) * ey + ky) * ex + kx;
    if (KIND == 2) {
        if (valid) *out = (unsigned short)cell_owner(g, sp, cp.np, x, y, z);
        return;
    }
    const int lane = threadIdx.x & 31;
    const CellOffset co = cell_offset(g, sp[p], x, y, z);
    const int quick = valid ? solid_count_quick(sp[p], co, cp.subsample) : 0;
    if (valid && quick >= 0) *out = (unsigned short)quick;
    unsigned todo = __ballot_sync(0xffffffffu, valid && quick < 0);
    while (todo) {
        const int c = __ffs(todo) - 1;
        todo &= todo - 1;
        const int xc = __shfl_sync(0xffffffffu, x, c);
        const CellOffset cc{__shfl_sync(0xffffffffu, co.dx, c), co.dy, co.dz};
        const int cnt = solid_count_warp(g, sp[p], cc, xc, y, z, cp.subsample, lane);
        if (lane == c) *out = (unsigned short)cnt;
    }
}

template <int KIND>
__global__ void __launch_bounds__(32)
    k_map(Geom g, Coupl cp, const DevParticle* __restrict__ parts, unsigned short* __restrict__ map,
          int ex, int ey, int ez) {
    __shared__ DevParticle sp[MAX_PARTICLES];
    step_enter();
    parts = entered(parts);
    const int nd = cp.np * (int)(sizeof(DevParticle) / sizeof(double));
    for (int i = threadIdx.x; i < nd; i += blockDim.x)
        reinterpret_cast<double*>(sp)[i] = reinterpret_cast<const double*>(parts)[i];
    __syncthreads();
    map_cell<KIND>(g, cp, sp, map, ex, ey, ez, blockIdx.z / ez, blockIdx.x * 32 + threadIdx.x,
                   blockIdx.y, blockIdx.z % ez);
}

// ---------------------------------------------------------------------------
// fixed-order force/torque total of particle q (one block per particle):
// F = (S_1 + ... + S_nsub) / nsub with S_k the sum, over the near-kernel
// blocks of every particle's region, of subcycle k's partials for q.
// charge != nullptr: the pending re-mapping momentum charge of q, [q][6],
// divided by the step's lattice time nsub, is taken off.
//
// A few thousand doubles at most, so latency bounds it: thread t adds
// component t mod 6 of every 128th partial (consecutive threads read
// consecutive doubles), one warp per component adds the 128 sums.  D = 24,
// 900 partials: 13.7 us (256 threads over all six components, an eight-level
// tree of FP64 adds per subcycle) + 8.6 us of rigid-body update -> 10.2 us for
// both in one launch (k_finalize_rigid), cold L2.
constexpr int FIN_WAYS = 128, FIN_THREADS = 6 * FIN_WAYS;
__device__ __forceinline__ void finalize_block(int np, long long nblk,
                                               const double* __restrict__ partials, int nsub,
                                               double* out, int q, double* red,
                                               const double* __restrict__ charge = nullptr) {
    const int tid = threadIdx.x, c = tid % 6, way = tid / 6;
    const long long count = (long long)nsub * np * nblk;
    double acc = 0.0;
#pragma unroll 4
    for (long long m = way; m < count; m += FIN_WAYS) acc += partials[(m * np + q) * 6 + c];
    red[c * FIN_WAYS + way] = acc;
    __syncthreads();
    const int w = tid >> 5, lane = tid & 31;
    if (w < 6) {
        const double* r = red + w * FIN_WAYS + lane;
        const double v = warp_sum((r[0] + r[32]) + (r[64] + r[96]));
        if (lane == 0)
            out[q * 6 + w] = charge ? v / nsub - charge[q * 6 + w] / nsub : v / nsub;
    }
}

__global__ void __launch_bounds__(FIN_THREADS)
    k_finalize(int np, long long nblk, const double* __restrict__ partials, int nsub,
               double* __restrict__ out, const double* __restrict__ charge, int* gate) {
    __shared__ double red[FIN_THREADS];
    step_enter();
    gate_close(gate);
    finalize_block(np, nblk, entered(partials), nsub, out, blockIdx.x, red,
                   charge ? entered(charge) : nullptr);
}

// ---------------------------------------------------------------------------
// explicit Euler rigid-body update over dt, gravity + buoyancy
// (rho_p - rho0) V g; keeps the previous state in `prev`.  Called by one warp
// per particle: lane a (< 3) updates axis a, so the chain of FP64 divisions
// that bounds it is one axis long.
// (`force` may have been written by the same kernel: not __restrict__.)
__device__ __forceinline__ void rigid_one(const Geom& g, DevParticle* part, DevParticle* prev,
                                          const double* force, double rho0, double gx, double gy,
                                          double gz, double dt, int wall_contact, int* status) {
    const int a = threadIdx.x & 31;
    constexpr int WORDS = (int)(sizeof(DevParticle) / sizeof(double));
    for (int i = a; i < WORDS; i += 32)
        reinterpret_cast<double*>(prev)[i] = reinterpret_cast<const double*>(part)[i];
    __syncwarp();
    if (a >= 3) return;
    const unsigned lanes = 7u;
    const double D = part->d, R = 0.5 * D, rho = part->rho;
    double x = part->x[a], u = part->u[a], w = part->w[a];
    const double x_old = x, u_old = u, w_old = w;
    if (part->fixed == 0.0) {
        const double PI = 3.14159265358979323846;
        const double V = PI * D * D * D / 6.0;
        const double m = rho * V, I = m * D * D / 10.0;
        const double grav = a == 0 ? gx : (a == 1 ? gy : gz);
        const double Ft = force[a] + (rho - rho0) * V * grav;
        x += dt * u;
        u += dt * Ft / m;
        w += dt * force[3 + a] / I;
        // a non-finite state, or a surface moving a cell or more per step,
        // is outside what the lattice can represent: report it and keep the
        // previous state so that the cell geometry stays well defined
        const bool sane = isfinite(x) && fabs(u) < 1.0 && fabs(w) * R < 1.0;
        if (!__all_sync(lanes, sane)) {
            if (a == 0) atomicOr(status, ST_UNSTABLE);
            x = x_old;
            u = u_old;
            w = w_old;
        }
        const double L = a == 0 ? g.nx : (a == 1 ? g.ny : g.nz);
        if (!(a == 2 && g.bc_z)) {
            if (x < 0.0) x += L;
            else if (x >= L) x -= L;
        } else if (g.bc_z == 2) {
            // open boundaries: the near region must stay clear of them
            if (x - R - OPEN_MARGIN < 0.0 || x + R + OPEN_MARGIN > L) atomicOr(status, ST_DOMAIN);
        } else if (wall_contact) {
            if (x - R < 1.0) {
                x = R + 1.0;
                if (u < 0.0) u = 0.0;
            }
            if (x + R > L - 1.0) {
                x = L - 1.0 - R;
                if (u > 0.0) u = 0.0;
            }
        } else if (x - R < 0.0 || x + R > L) {
            atomicOr(status, ST_DOMAIN);
        }
    }
    part->x[a] = x;
    part->u[a] = u;
    part->w[a] = w;
    store_region_axis(g, *part, x, a);
}

// one warp per particle
__global__ void __launch_bounds__(32)
    k_rigid(Geom g, DevParticle* __restrict__ parts, DevParticle* __restrict__ prev,
            const double* __restrict__ force, double rho0, double gx, double gy, double gz,
            double dt, int wall_contact, int* __restrict__ status) {
    step_enter();
    parts = entered(parts);
    force = entered(force);
    const int p = blockIdx.x;
    rigid_one(g, parts + p, prev + p, force + 6 * p, rho0, gx, gy, gz, dt, wall_contact, status);
}

// Force total and rigid-body update of particle blockIdx.x in one launch
// (nothing else reads the force in between: no force model attached).
__global__ void __launch_bounds__(FIN_THREADS)
    k_finalize_rigid(Geom g, int np, long long nblk, const double* __restrict__ partials, int nsub,
                     double* force, const double* __restrict__ charge, DevParticle* parts,
                     DevParticle* prev, double rho0, double gx, double gy, double gz, double dt,
                     int wall_contact, int* status, int* gate) {
    __shared__ double red[FIN_THREADS];
    step_enter();
    gate_close(gate);
    parts = entered(parts);
    const int p = blockIdx.x;
    finalize_block(np, nblk, entered(partials), nsub, force, p, red,
                   charge ? entered(charge) : nullptr);
    __syncthreads();
    if (threadIdx.x < 32)
        rigid_one(g, parts + p, prev + p, force + 6 * p, rho0, gx, gy, gz, dt, wall_contact, status);
}

// One thread per particle.  (Four copies, two region kernels and a wait for the
// stream before: ten coarse FP32 steps, each with its sphere placed, 1210 us; this
// 1083.)
__global__ void __launch_bounds__(MAX_PARTICLES)
    k_set_particles(Geom g, const ParticleUpload up, int n, DevParticle* parts, DevParticle* prev,
                    DevParticle* old) {
    step_enter();
    const int i = threadIdx.x;
    if (i >= n) return;
    parts = entered(parts);
    if (old) old[i] = parts[i];
    DevParticle d = up.rec[i];
    store_region(g, d);
    parts[i] = d;
    if (prev) prev[i] = d;
}

// ---------------------------------------------------------------------------
// MEM re-mapping with PDF reconstruction (Sec. 2.2, Eq. (19)).  One thread per
// cell of the box around each particle's old position finds the candidates: a
// cell solid under p_old (owner p) and fluid under p_new.  Each candidate is
// then rebuilt by its whole warp (refill_warp) and gets:
//   extrapolate = 1: f = 3 f(x+c_n) - 3 f(x+2c_n) + f(x+3c_n) (fewer terms when
//     fewer usable fluid cells follow), with the pre-collision values of those
//     cells rebuilt from srcB (the buffer the last sweep pulled from) under
//     p_old; then the velocity constraint j = rho0 v; with no usable cell,
//     f_eq(rho_bar, v);
//   extrapolate = 0: f_eq(rho0, v);
// and is then collided (plain fluid collision) into dst.

// Pre-collision value f_q(x) of one direction q (known at run time) of a
// fluid cell x, as mem_pull rebuilds it (particle owners from the records).
template <typename T, typename C>
__device__ __forceinline__ C mem_pull_dir(const T* __restrict__ src, const Geom& g, const Coupl& cp,
                                          const DevParticle* parts, int x, int y, int z, int q,
                                          int* status) {
    const long long idx = lin(g, x, y, z);
    if (q == 0) return PdfStore<T>::template load<C>(src + idx, 0);
    const Nbr b = make_nbr(g, x, y, z);
    const int qp = opp(q);
    int xs, ys, zs;
    shifted_rt(b, x, y, z, q, -1, xs, ys, zs);
    if (rcz(q) != 0 && (zs < 0 || zs >= g.nz))
        return PdfStore<T>::template load<C>(src + (long long)qp * g.n + idx, qp);
    const int owner = cell_owner(g, parts, cp.np, xs, ys, zs);
    if (!owner) {
        if (xs < 0 || xs >= g.nx || ys < 0 || ys >= g.ny || zs < 0 || zs >= g.nz) {
            atomicOr(status, ST_BOUNDS);
            return (C)0.0;
        }
        return PdfStore<T>::template load<C>(src + (long long)q * g.n + lin(g, xs, ys, zs), q);
    }
    if (owner < 0 || owner > cp.np) {
        atomicOr(status, ST_BOUNDS);
        return (C)0.0;
    }
    MrCell mc;
    mc.have = false;
    int unused = 0;
    return (C)mem_link(src, g, cp, parts, cp.np, (const GeoMap*)nullptr, b, x, y, z, idx, q,
                       (double*)nullptr, &unused, status, mc);
}

// Per-warp scratch of the refill.
struct RefillWarp {
    double f[3][NQ];  // pre-collision values of the extrapolation cells; f[0]: the rebuilt ones
    double r[NQ];     // densities of the usable neighbours (no extrapolation cell)
    int ok[NQ];
};

// Sum over the warp, the same bits on every lane.
__device__ __forceinline__ double warp_sum_all(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// q_n = argmax_q n . c_q, lowest q on ties, n the unit vector along r.  Lane q
// weighs direction q, in FP32 on r itself;
// where two directions come within the FP32 error (exact ties on a lattice
// symmetry plane do) the unit vector and the comparison are FP64, as defined.
// All lanes call it with the same r and get the same answer.
__device__ __forceinline__ int normal_direction(const double (&r)[3], int lane) {
    const unsigned full = 0xffffffffu;
    const bool dir = lane >= 1 && lane < NQ;
    const float rx = (float)r[0], ry = (float)r[1], rz = (float)r[2];
    const float d = dir ? rx * rcx(lane) + ry * rcy(lane) + rz * rcz(lane) : 0.0f;
    const float best = __uint_as_float(__reduce_max_sync(full, __float_as_uint(fmaxf(d, 0.0f))));
    const unsigned near = __ballot_sync(
        full, dir && d >= best - 1e-5f * (fabsf(rx) + fabsf(ry) + fabsf(rz)));
    if (__popc(near) == 1) return __ffs(near) - 1;
    const double len = sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    double nrm[3] = {r[0], r[1], r[2]};
    if (len > 0.0)
        for (int a = 0; a < 3; ++a) nrm[a] /= len;
    double bd = dir ? nrm[0] * rcx(lane) + nrm[1] * rcy(lane) + nrm[2] * rcz(lane) : -1e300;
    int bq = dir ? lane : NQ;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(full, bd, o);
        const int oq = __shfl_xor_sync(full, bq, o);
        if (od > bd || (od == bd && oq < bq)) {
            bd = od;
            bq = oq;
        }
    }
    return bq;
}

// Rebuilds candidate cell (x, y, z) of particle p; all 32 lanes call it with
// the same cell.  The pulls are spread over the lanes, and lane q combines and
// corrects population q; the collision is computed by every lane alike and
// lane 0 stores.  jm receives the momentum sum_q c_q f_q of the rebuilt
// pre-collision populations (every lane; only with `momentum`).
//
// One cell is one chain of FP64 and memory latency on an otherwise idle GPU,
// so the chain's length is what counts: predicates filtered in FP32, the
// normal direction and the 19 corrections across the lanes (every lane doing
// all of it in FP64: 47 us for one cell, 61 us for the 45 of a D = 24 step;
// this form 30 us and 36 us).
template <typename T, typename C>
__device__ __forceinline__ void refill_warp(const T* __restrict__ srcB, T* __restrict__ dst,
                                            const Geom& g, const Coll<C>& k, const Coupl& cp,
                                            const DevParticle* so, const DevParticle* sn,
                                            int extrapolate, int p, int x, int y, int z,
                                            int* __restrict__ status, RefillWarp& w, int lane,
                                            bool momentum, double (&jm)[3]) {
    const DevParticle& Pn = sn[p];
    double r[3], v[3];
    centre_offset(g, Pn, x, y, z, r);
    v[0] = Pn.u[0] + (Pn.w[1] * r[2] - Pn.w[2] * r[1]);
    v[1] = Pn.u[1] + (Pn.w[2] * r[0] - Pn.w[0] * r[2]);
    v[2] = Pn.u[2] + (Pn.w[0] * r[1] - Pn.w[1] * r[0]);
    C fn[NQ];
    int m = 0;
    int nbx[3], nby[3], nbz[3];
    if (extrapolate) {
        const int qn = normal_direction(r, lane);
        for (int kk = 1; kk <= 3; ++kk) {
            int xx = wrap_i(x + kk * rcx(qn), g.nx), yy = wrap_i(y + kk * rcy(qn), g.ny),
                zz = z + kk * rcz(qn);
            if (g.bc_z) {
                if (zz < 0 || zz >= g.nz) break;
            } else {
                zz = wrap_i(zz, g.nz);
            }
            if (cell_owner(g, so, cp.np, xx, yy, zz) || cell_owner(g, sn, cp.np, xx, yy, zz))
                break;
            nbx[m] = xx;
            nby[m] = yy;
            nbz[m] = zz;
            ++m;
        }
    }
    const bool dir = lane < NQ;
    const double cxl = dir ? rcx(lane) : 0, cyl = dir ? rcy(lane) : 0, czl = dir ? rcz(lane) : 0;
    if (m > 0) {
        // the m x 19 pulls, lane by lane
        for (int i = lane; i < m * NQ; i += 32) {
            const int jn = i / NQ, q = i - jn * NQ;
            w.f[jn][q] =
                (double)mem_pull_dir<T, C>(srcB, g, cp, so, nbx[jn], nby[jn], nbz[jn], q, status);
        }
        __syncwarp();
        C fl = (C)0;
        if (dir) {
            if (m == 1) fl = (C)w.f[0][lane];
            else if (m == 2) fl = (C)2 * (C)w.f[0][lane] - (C)w.f[1][lane];
            else fl = (C)3 * (C)w.f[0][lane] - (C)3 * (C)w.f[1][lane] + (C)w.f[2][lane];
        }
        // velocity constraint: only the momentum moment changes (sum_q c_qa^2 = 10)
        const double dj0 = cp.rho0 * v[0] - warp_sum_all((double)fl * cxl);
        const double dj1 = cp.rho0 * v[1] - warp_sum_all((double)fl * cyl);
        const double dj2 = cp.rho0 * v[2] - warp_sum_all((double)fl * czl);
        fl = (C)((double)fl + (cxl * dj0 + cyl * dj1 + czl * dj2) / 10.0);
        if (dir) w.f[0][lane] = (double)fl;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NQ; ++q) fn[q] = (C)w.f[0][q];
    } else {
        double rbar = cp.rho0;
        if (extrapolate) {
            // lane q - 1 pulls neighbour x + c_q (q = 1..18) when it is usable
            if (lane < NQ - 1) {
                const int q = lane + 1;
                int xx = wrap_i(x + rcx(q), g.nx), yy = wrap_i(y + rcy(q), g.ny), zz = z + rcz(q);
                bool ok = true;
                if (g.bc_z) ok = zz >= 0 && zz < g.nz;
                else zz = wrap_i(zz, g.nz);
                if (ok)
                    ok = !cell_owner(g, so, cp.np, xx, yy, zz) && !cell_owner(g, sn, cp.np, xx, yy, zz);
                double rho = 0.0;
                if (ok) {
                    C fq[NQ];
                    mem_pull(srcB, g, cp, so, cp.np, xx, yy, zz, lin(g, xx, yy, zz), fq, status);
#pragma unroll
                    for (int qq = 0; qq < NQ; ++qq) rho += (double)fq[qq];
                }
                w.r[q] = rho;
                w.ok[q] = ok ? 1 : 0;
            }
            __syncwarp();
            double sum = 0.0;
            int cnt = 0;
            for (int q = 1; q < NQ; ++q) {
                if (!w.ok[q]) continue;
                sum += w.r[q];
                ++cnt;
            }
            if (cnt > 0) rbar = sum / cnt;
        }
        equilibrium((C)rbar, (C)v[0], (C)v[1], (C)v[2], k.rho0, fn);
        if (lane == 0)
#pragma unroll
            for (int q = 0; q < NQ; ++q) w.f[0][q] = (double)fn[q];
        __syncwarp();
    }
    if (momentum) {
        const double fl = dir ? w.f[0][lane] : 0.0;
        jm[0] = warp_sum_all(fl * cxl);
        jm[1] = warp_sum_all(fl * cyl);
        jm[2] = warp_sum_all(fl * czl);
    }
    collide_cell(fn, k);
    if (lane == 0) {
        if (x < 0 || x >= g.nx || y < 0 || y >= g.ny || z < 0 || z >= g.nz)
            atomicOr(status, ST_BOUNDS);
        else
            store_own(dst, g, lin(g, x, y, z), fn);
    }
    __syncwarp();
}

// Adds sign * (j, (x_c - X_p) x j) of cell (x, y, z) to acc, X_p the centre
// of P (minimum image in periodic directions).
__device__ __forceinline__ void add_cell_moment(double (&acc)[6], const Geom& g,
                                                const DevParticle& P, int x, int y, int z,
                                                const double (&j)[3], double sign) {
    double r[3];
    centre_offset(g, P, x, y, z, r);
    acc[0] += sign * j[0];
    acc[1] += sign * j[1];
    acc[2] += sign * j[2];
    acc[3] += sign * (r[1] * j[2] - r[2] * j[1]);
    acc[4] += sign * (r[2] * j[0] - r[0] * j[2]);
    acc[5] += sign * (r[0] * j[1] - r[1] * j[0]);
}

// Candidate test of one cell of particle p's box per lane, then the warp's
// candidates one after another.  Every lane of the warp must call this.
//
// Warp `warp` of `warps` tests cells warp, warp + warps, ... of the box: the
// cells a sphere uncovers lie side by side in the rows of its cap, and a warp
// that tested a run of a row rebuilt up to a dozen of them in turn while most
// warps had none.  A candidate is a long chain of FP64 latency, so the launch
// takes about as long as the fullest warp (D = 24 settling, ~45 cells per
// step: 92 us for runs of a row, 61 us dealt out).
//
// acc != nullptr: re-mapping momentum charge of particle p (uncovered cells
// plus, covered cells minus; moments about the new centre) added to this
// thread's six sums.  The box holds every cell of the new sphere while the
// centre moves by less than 1.5 cells per axis in a step.
template <typename T, typename C>
__device__ __forceinline__ void refill_cells(const T* __restrict__ srcB, T* __restrict__ dst,
                                             const Geom& g, const Coll<C>& k, const Coupl& cp,
                                             const DevParticle* so, const DevParticle* sn,
                                             int extrapolate, int side, int p, long long warp,
                                             long long warps, int* __restrict__ status,
                                             RefillWarp& w, int lane, double (*acc)[6] = nullptr) {
    const long long lid = warp + lane * warps;
    bool cand = lid < (long long)side * side * side;
    int x = 0, y = 0, z = 0;
    if (cand) {
        const int kx = (int)(lid % side), ky = (int)((lid / side) % side),
                  kz = (int)(lid / ((long long)side * side));
        const DevParticle& Po = so[p];
        x = (int)floor(Po.x[0] - Po.r) - 1 + kx;
        y = (int)floor(Po.x[1] - Po.r) - 1 + ky;
        z = (int)floor(Po.x[2] - Po.r) - 1 + kz;
        x = wrap_i(x, g.nx);
        y = wrap_i(y, g.ny);
        if (g.bc_z) {
            if (z < 0 || z >= g.nz) cand = false;
        } else {
            z = wrap_i(z, g.nz);
        }
    }
    const int own_old = cand ? cell_owner(g, so, cp.np, x, y, z) : -1;
    const bool test_new = own_old == p + 1 || (acc && own_old == 0);
    const int own_new = test_new ? cell_owner(g, sn, cp.np, x, y, z) : -1;
    cand = own_old == p + 1 && own_new == 0;
    const unsigned full = 0xffffffffu;
    if (acc) {
        // covered: the fluid momentum of the cell's pre-collision populations
        // leaves the fluid; lane q pulls direction q
        for (unsigned m = __ballot_sync(full, own_old == 0 && own_new == p + 1); m; m &= m - 1) {
            const int src_lane = __ffs(m) - 1;
            const int xc = __shfl_sync(full, x, src_lane), yc = __shfl_sync(full, y, src_lane),
                      zc = __shfl_sync(full, z, src_lane);
            if (lane < NQ)
                w.f[0][lane] =
                    (double)mem_pull_dir<T, C>(srcB, g, cp, so, xc, yc, zc, lane, status);
            __syncwarp();
            if (lane == src_lane) {
                double j[3] = {0.0, 0.0, 0.0};
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    j[0] += w.f[0][q] * cx(q);
                    j[1] += w.f[0][q] * cy(q);
                    j[2] += w.f[0][q] * cz(q);
                }
                add_cell_moment(*acc, g, sn[p], x, y, z, j, -1.0);
            }
            __syncwarp();
        }
    }
    for (unsigned m = __ballot_sync(full, cand); m; m &= m - 1) {
        const int src_lane = __ffs(m) - 1;
        const int cxl = __shfl_sync(full, x, src_lane), cyl = __shfl_sync(full, y, src_lane),
                  czl = __shfl_sync(full, z, src_lane);
        double jm[3];
        refill_warp<T, C>(srcB, dst, g, k, cp, so, sn, extrapolate, p, cxl, cyl, czl, status, w,
                          lane, acc != nullptr, jm);
        if (acc && lane == src_lane) add_cell_moment(*acc, g, sn[p], cxl, cyl, czl, jm, 1.0);
    }
}

// The refill box holds the new sphere only for a step of less than 1.5
// cells per axis: a faster step is reported as unstable.
__device__ __forceinline__ void charge_step_check(const Geom& g, const DevParticle& Pn,
                                                  const DevParticle& Po, int* status) {
    double d[3];
    separation(g, Pn.x[0], Pn.x[1], Pn.x[2], Po, d[0], d[1], d[2]);
    if (fabs(d[0]) >= 1.5 || fabs(d[1]) >= 1.5 || fabs(d[2]) >= 1.5) atomicOr(status, ST_UNSTABLE);
}

// Fixed-order sum of the block's per-thread charge sums into out[0..6): a
// butterfly within each warp, then the warps in turn.  Every thread of the
// REFILL_THREADS-thread block calls it.
__device__ __forceinline__ void charge_block_sum(const double (&acc)[6], double* out) {
    __shared__ double red[REFILL_THREADS / 32][6];
    const int tid = threadIdx.x, lane = tid & 31;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        double v = acc[c];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) red[tid >> 5][c] = v;
    }
    __syncthreads();
    if (tid < 6) {
        double t = 0.0;
        for (int wi = 0; wi < REFILL_THREADS / 32; ++wi) t += red[wi][tid];
        out[tid] = t;
    }
}

// Grid (ceil(side^3 / REFILL_THREADS), np).  charge_part != nullptr: block
// (bx, p) also writes its fixed-order sums of particle p's re-mapping
// momentum charge to charge_part[(p * gridDim.x + bx) * 6 + c].
template <typename T, typename C>
__global__ void __launch_bounds__(REFILL_THREADS)
    k_refill(const T* __restrict__ srcB, T* __restrict__ dst, Geom g, Coll<C> k, Coupl cp,
             const DevParticle* __restrict__ p_old, const DevParticle* __restrict__ p_new,
             int extrapolate, int side, int* __restrict__ status,
             double* __restrict__ charge_part) {
    __shared__ DevParticle so[MAX_PARTICLES], sn[MAX_PARTICLES];
    const int tid = threadIdx.x;
    step_enter();
    p_old = entered(p_old);
    p_new = entered(p_new);
    srcB = entered(srcB);
    const int nd = cp.np * (int)(sizeof(DevParticle) / sizeof(double));
    for (int i = tid; i < nd; i += blockDim.x) {
        reinterpret_cast<double*>(so)[i] = reinterpret_cast<const double*>(p_old)[i];
        reinterpret_cast<double*>(sn)[i] = reinterpret_cast<const double*>(p_new)[i];
    }
    __syncthreads();
    __shared__ RefillWarp rw[REFILL_THREADS / 32];
    const int p = blockIdx.y, lane = tid & 31;
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    refill_cells<T, C>(srcB, dst, g, k, cp, so, sn, extrapolate, side, p,
                       (long long)blockIdx.x * (REFILL_THREADS / 32) + (tid >> 5),
                       (long long)gridDim.x * (REFILL_THREADS / 32), status, rw[tid >> 5], lane,
                       charge_part ? &acc : nullptr);
    if (!charge_part) return;
    if (tid == 0) charge_step_check(g, sn[p], so[p], status);
    charge_block_sum(acc, charge_part + ((long long)p * gridDim.x + blockIdx.x) * 6);
}

// out[c] = sum over nblk refill-block partials [blk][6]; warp c of the block's
// six adds component c (one thread per component over 172 partials: 16 us;
// this form 3.9 us).
__device__ __forceinline__ void charge_total(long long nblk, const double* __restrict__ part,
                                             double* __restrict__ out) {
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
#pragma unroll 4
    for (long long b = lane; b < nblk; b += 32) s += part[b * 6 + c];
    s = warp_sum(s);
    if (lane == 0) out[c] = s;
}

// one block of six warps per particle
__global__ void __launch_bounds__(192)
    k_charge_total(long long nblk, const double* __restrict__ part, double* __restrict__ out) {
    step_enter();
    charge_total(nblk, entered(part) + (long long)blockIdx.x * nblk * 6, out + blockIdx.x * 6);
}

// ---------------------------------------------------------------------------
// macroscopic fields of the pre-collision state at the start of the next step
// what: 2 rho, 3 u, 4 eps (PSM), 5 owner flag (MEM)
template <typename T, typename C, bool NOSTREAM>
__global__ void __launch_bounds__(256)
    k_macro(const T* __restrict__ state, Geom g, Coll<C> k, Coupl cp,
            const DevParticle* __restrict__ parts, double fx, double fy, double fz, int what,
            void* out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    const int x = (int)(i % g.nx), y = (int)((i / g.nx) % g.ny), z = (int)(i / ((long long)g.nx * g.ny));
    const double xc = x + 0.5, yc = y + 0.5, zc = z + 0.5;
    double* od = reinterpret_cast<double*>(out);
    if (cp.kind == 2) {
        int own = cell_owner(g, parts, cp.np, x, y, z);
        if (what == 5) {
            reinterpret_cast<int*>(out)[i] = own;
            return;
        }
        if (what == 4) {
            od[i] = own ? 1.0 : 0.0;
            return;
        }
        double rho, u[3];
        if (own) {
            rho = cp.rho0;
            body_velocity(g, parts[own - 1], xc, yc, zc, u[0], u[1], u[2]);
        } else {
            // post-collision moments: rho is conserved, j gains f_ext
            double r = 0.0, j[3] = {0.0, 0.0, 0.0};
            for (int q = 0; q < NQ; ++q) {
                double v = ld_pdf(state + (long long)q * g.n + i, q);
                r += v;
                j[0] += v * cx(q);
                j[1] += v * cy(q);
                j[2] += v * cz(q);
            }
            rho = r;
            u[0] = (j[0] - fx) / cp.rho0 + fx / (2.0 * cp.rho0);
            u[1] = (j[1] - fy) / cp.rho0 + fy / (2.0 * cp.rho0);
            u[2] = (j[2] - fz) / cp.rho0 + fz / (2.0 * cp.rho0);
        }
        if (what == 2) od[i] = rho;
        else {
            od[3 * i + 0] = u[0];
            od[3 * i + 1] = u[1];
            od[3 * i + 2] = u[2];
        }
        return;
    }
    if (what == 5) {
        reinterpret_cast<int*>(out)[i] = 0;
        return;
    }
    double B = 0.0, vs[3] = {0.0, 0.0, 0.0}, epsum = 0.0;
    if (cp.kind == 1) {
        for (int s = 0; s < cp.np; ++s) {
            if (!cell_in_reg(g, parts[s].reg, x, y, z)) continue;
            double e = solid_fraction(g, parts[s], x, y, z, cp.subsample);
            if (e <= 0.0) continue;
            epsum += e;
            double Bs = cp.variant == 0 ? e : e * (cp.tau - 0.5) / ((1.0 - e) + (cp.tau - 0.5));
            double v[3];
            body_velocity(g, parts[s], xc, yc, zc, v[0], v[1], v[2]);
            B += Bs;
            for (int a = 0; a < 3; ++a) vs[a] += Bs * v[a];
        }
    }
    if (what == 4) {
        od[i] = epsum;
        return;
    }
    C f[NQ];
    if (NOSTREAM)
        load_own(state, g, i, f);
    else
        pull_plain(state, g, x, y, z, i, f);
    double r = 0.0, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        r += (double)f[q];
        j[0] += (double)f[q] * cx(q);
        j[1] += (double)f[q] * cy(q);
        j[2] += (double)f[q] * cz(q);
    }
    if (what == 2) {
        od[i] = r;
        return;
    }
    const double fe[3] = {fx, fy, fz};
    for (int a = 0; a < 3; ++a) {
        double ua = j[a] / cp.rho0 + fe[a] / (2.0 * cp.rho0);
        od[3 * i + a] = (1.0 - B) * ua + vs[a];
    }
}

template <typename T>
__global__ void k_init_eq(T* __restrict__ dst, Geom g, double rho, double ux, double uy, double uz,
                         double rho0) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    double e[NQ];
    equilibrium(rho, ux, uy, uz, rho0, e);
#pragma unroll
    for (int q = 0; q < NQ; ++q) dst[(long long)q * g.n + i] = PdfStore<T>::template save<double>(e[q], q);
}

template <typename T>
__global__ void k_to_f64(const T* __restrict__ in, double* __restrict__ out, long long count,
                         long long ncell) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = ld_pdf(in + i, (int)(i / ncell));
}

template <typename T>
__global__ void k_from_f64(const double* __restrict__ in, T* __restrict__ out, long long count,
                           long long ncell) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = PdfStore<T>::template save<double>(in[i], (int)(i / ncell));
}


// ---------------------------------------------------------------------------
// Batched ensemble kernels.  Each launch covers every case of a work list;
// block (or work item) t belongs to case list[i] with base[i] <= t < base[i+1].
__device__ __forceinline__ int find_item(const long long* __restrict__ base, int n, long long t) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(base + mid) <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// cell and tile ranges of each case's particle (after upload or a change of
// the bulk tiling); the previous state starts equal to the current one
__global__ void k_batch_regions(BatchCase* __restrict__ cases, int n) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    store_region(cases[c].g, *cases[c].part);
    *cases[c].prev = *cases[c].part;
}

// f = f_eq(rho0, 0) in the stored buffer of every case (fluid at rest: the
// post-collision and pre-collision fields coincide).
__global__ void k_batch_init(BatchCase* __restrict__ cases) {
    const BatchCase& B = cases[blockIdx.y];
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B.g.n) return;
    double e[NQ];
    equilibrium(B.kd.rho0, 0.0, 0.0, 0.0, B.kd.rho0, e);
#pragma unroll
    for (int q = 0; q < NQ; ++q) B.buf[B.cur][(long long)q * B.g.n + i] = e[q];
}

// geometry map: 32-thread blocks over (x chunk, y, z) of each case's region
__global__ void __launch_bounds__(32) k_batch_map(BatchCase* __restrict__ cases, BatchList l) {
    __shared__ DevParticle sp[1];
    const int i = find_item(l.base, l.n, blockIdx.x);
    const BatchCase& B = cases[l.list[i]];
    const long long local = blockIdx.x - l.base[i];
    for (int k = threadIdx.x; k < (int)(sizeof(DevParticle) / sizeof(double)); k += 32)
        reinterpret_cast<double*>(sp)[k] = reinterpret_cast<const double*>(B.part)[k];
    __syncthreads();
    const int nbx = (B.map_ext[0] + 31) / 32;
    const int bx = (int)(local % nbx);
    const long long rest = local / nbx;
    const int ky = (int)(rest % B.map_ext[1]), kz = (int)(rest / B.map_ext[1]);
    if (B.kind == 2)
        map_cell<2>(B.g, B.cp, sp, B.map, B.map_ext[0], B.map_ext[1], B.map_ext[2], 0,
                    bx * 32 + threadIdx.x, ky, kz);
    else
        map_cell<1>(B.g, B.cp, sp, B.map, B.map_ext[0], B.map_ext[1], B.map_ext[2], 0,
                    bx * 32 + threadIdx.x, ky, kz);
}

// near-particle sweep: one near block of one case per thread block
__global__ void __launch_bounds__(NEAR_THREADS)
    k_batch_near(BatchCase* __restrict__ cases, BatchList l, int sub, int* __restrict__ status) {
    __shared__ DevParticle sp[1];
    __shared__ LinkWarp lw;
    const int i = find_item(l.base, l.n, blockIdx.x);
    const BatchCase& B = cases[l.list[i]];
    const long long local = blockIdx.x - l.base[i];
    for (int k = threadIdx.x; k < (int)(sizeof(DevParticle) / sizeof(double)); k += NEAR_THREADS)
        reinterpret_cast<double*>(sp)[k] = reinterpret_cast<const double*>(B.part)[k];
    __syncwarp();
    const GeoMap gm{B.map, B.map_ext[0], B.map_ext[1], B.map_ext[2]};
    const int cur = B.cur;
    double* partials = B.partials + (long long)sub * B.nblk * 6;
    if (B.kind == 2)
        near_block<double, double, 2, false>(B.buf[cur], B.buf[1 - cur], B.g, B.kd, B.cp, sp, gm,
                                             partials, status, 0, B.nblk, local, lw);
    else
        near_block<double, double, 1, false>(B.buf[cur], B.buf[1 - cur], B.g, B.kd, B.cp, sp, gm,
                                             partials, status, 0, B.nblk, local, lw);
}

// Threads of a k_batch_bulk block and its resident blocks per SM; a work item
// is 256 cells, so each thread takes BATCH_ITEM / BATCH_THREADS of them.
constexpr int BATCH_ITEM = 256, BATCH_THREADS = 128, BATCH_BLOCKS = 5;
// A block takes up to 4 items in a row: finding the item's case and staging its
// record is a chain of dependent loads ahead of its PDFs (12 cases of D = 8..16, 3
// steps: 3375 us with one item per block, 3327 with four).  One per block while
// there are fewer than six waves of 760 blocks.
constexpr long long BATCH_CHUNK_ITEMS = 4560;

// Cell (x, y, z) of an item's thread slot t: false beyond the lattice.  Plane
// segments (layout 1) are 256 consecutive cells of an xy plane, so domains
// whose nx is not a multiple of the warp width keep every lane busy; box
// tiles of g.tx cells leave g.tx - nx mod g.tx lanes of each row idle.
__device__ __forceinline__ bool batch_cell(const Geom& g, int layout, long long local, int t,
                                           int& x, int& y, int& z) {
    if (layout == 1) {
        const int nseg = (g.nx * g.ny + BATCH_ITEM - 1) / BATCH_ITEM;
        z = (int)(local / nseg);
        const int l = ((int)local - z * nseg) * BATCH_ITEM + t;
        y = l / g.nx;
        x = l - y * g.nx;
        return l < g.nx * g.ny;
    }
    const int tX = (int)(local % g.ntx), tY = (int)((local / g.ntx) % g.nty);
    z = (int)(local / ((long long)g.ntx * g.nty));
    x = tX * g.tx + t % g.tx;
    y = tY * g.ty + t / g.tx;
    return x < g.nx && y < g.ny;
}

// bulk sweep: persistent blocks striding over the 256-cell items of all
// listed cases.  Each case has its own tiling (B.layout, chosen by the
// autotuner): 0 box tiles of g.tx x g.ty cells; 1 plane segments.  The case
// record is staged in shared memory once per run of items of a case: its constants
// are read ~60 times per cell, and as global loads they cost the registers
// that the cell's 19 values need (12 cases of D = 8..16, 6.8 M cells, 3 steps:
// constants from global memory, 256 threads, 1 KB of spills 4.10 ms; staged,
// 128 threads, 3.87 ms; the FP64 form 10.08 ms).  As shared-memory operands they
// still leave 216 B of spills per thread (k_bulk, whose constants are kernel
// parameters, 4 B): 0.65 to 0.70 of the measured HBM bandwidth.
__global__ void __launch_bounds__(BATCH_THREADS, BATCH_BLOCKS)
    k_batch_bulk(BatchCase* __restrict__ cases, BatchList l, long long total, int chunk,
                 int* __restrict__ status) {
    __shared__ BatchCase B;
    __shared__ int reg[12];
    long long lo = 0, hi = 0;  // items of the staged case
    long long t = (long long)blockIdx.x * chunk;
    for (int left = chunk; t < total; ++t) {
        if (left == 0) {  // the next chunk of a persistent block
            t += ((long long)gridDim.x - 1) * chunk;
            if (t >= total) break;
            left = chunk;
        }
        --left;
        if (t < lo || t >= hi) {
            const int i = find_item(l.base, l.n, t);
            lo = l.base[i];
            hi = l.base[i + 1];
            __syncthreads();
            const BatchCase* G = cases + l.list[i];
            for (int k = threadIdx.x; k < (int)(sizeof(BatchCase) / 8); k += BATCH_THREADS)
                reinterpret_cast<long long*>(&B)[k] = reinterpret_cast<const long long*>(G)[k];
            if (threadIdx.x < 12) reg[threadIdx.x] = G->part->reg[threadIdx.x];
            __syncthreads();
        }
        const double* src = B.buf[B.cur];
        double* dst = B.buf[1 - B.cur];
        bool bad = false;
        for (int s = threadIdx.x; s < BATCH_ITEM; s += BATCH_THREADS) {
            int x, y, z;
            if (!batch_cell(B.g, B.layout, t - lo, s, x, y, z)) continue;
            if (cell_in_reg(B.g, reg, x, y, z)) continue;  // k_batch_near's cell
            const long long idx = lin(B.g, x, y, z);
            double f[NQ];
            pull_plain(src, B.g, x, y, z, idx, f);
            bad |= collide_cell(f, B.kd);
            store_own(dst, B.g, idx, f);
        }
        if (bad) atomicOr(status, ST_FLUID);
    }
}

__global__ void k_batch_swap(BatchCase* __restrict__ cases, BatchList l) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < l.n) cases[l.list[i]].cur ^= 1;
}

__global__ void __launch_bounds__(FIN_THREADS) k_batch_finalize(BatchCase* __restrict__ cases) {
    __shared__ double red[FIN_THREADS];
    const BatchCase& B = cases[blockIdx.x];
    const int nsub = B.kind != 0 ? B.subcycles : 1;
    finalize_block(1, B.nblk, B.partials, nsub, B.force, 0, red,
                   B.remap_charge ? B.charge : nullptr);
}

// one warp per case
__global__ void __launch_bounds__(32) k_batch_rigid(BatchCase* __restrict__ cases,
                                                    int* __restrict__ status) {
    const BatchCase& B = cases[blockIdx.x];
    const double dt = B.kind != 0 ? (double)B.subcycles : 1.0;
    rigid_one(B.g, B.part, B.prev, B.force, B.kd.rho0, B.gravity[0], B.gravity[1], B.gravity[2],
              dt, B.wall_contact, status);
}

// MEM re-mapping and refilling after the step (reads the buffer the last
// sweep pulled from, writes the stored state)
__global__ void __launch_bounds__(REFILL_THREADS)
    k_batch_refill(BatchCase* __restrict__ cases, BatchList l, int* __restrict__ status) {
    __shared__ DevParticle so[1], sn[1];
    const int i = find_item(l.base, l.n, blockIdx.x);
    const BatchCase& B = cases[l.list[i]];
    const long long local = blockIdx.x - l.base[i];
    for (int k = threadIdx.x; k < (int)(sizeof(DevParticle) / sizeof(double)); k += blockDim.x) {
        reinterpret_cast<double*>(so)[k] = reinterpret_cast<const double*>(B.prev)[k];
        reinterpret_cast<double*>(sn)[k] = reinterpret_cast<const double*>(B.part)[k];
    }
    __syncthreads();
    const int cur = B.cur;
    __shared__ RefillWarp rw[REFILL_THREADS / 32];
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    refill_cells<double, double>(B.buf[1 - cur], B.buf[cur], B.g, B.kd, B.cp, so, sn, 1,
                                 B.refill_side, 0, local * (REFILL_THREADS / 32) + (threadIdx.x >> 5),
                                 refill_blocks(B.refill_side) * (REFILL_THREADS / 32), status,
                                 rw[threadIdx.x >> 5], threadIdx.x & 31,
                                 B.remap_charge ? &acc : nullptr);
    // re-mapping charge: block partial `local` of this case (see k_refill)
    if (!B.remap_charge) return;
    if (threadIdx.x == 0) charge_step_check(B.g, sn[0], so[0], status);
    charge_block_sum(acc, B.charge_part + local * 6);
}

// Per case with the charge on: charge[c] = the fixed-order total of its
// refill-block partials.  One block of six warps per case.
__global__ void __launch_bounds__(192) k_batch_charge_total(BatchCase* __restrict__ cases) {
    const BatchCase& B = cases[blockIdx.x];
    if (B.remap_charge) charge_total(refill_blocks(B.refill_side), B.charge_part, B.charge);
}

// ---------------------------------------------------------------------------
// launchers
namespace {
// Launch with one common split of the SM's 256 KB between L1 and shared memory.
// The near sweep needs 9 KB of shared memory per warp (MEM) and runs beside the
// bulk sweep, which needs none.  Left to the default, a bulk block puts its
// SM in the all-L1 split, and near blocks cannot start there until the SM has
// drained.  Measured (us per pass, default / 25 / 50 / 100 % of the largest
// shared-memory size): 24 x 24 x 40 cells FP64, 20 steps 3210 / 2340 / 2330 /
// 2390; 32^3 FP64, 50 steps 3950 / 3370 / 3370 / 3470; 128 x 128 x 512 FP32, 8
// steps of 2 sweeps 5090 / 5090 / 4900 / 5690; FP16, 20 steps 3090 / 2980 /
// 2980 / 3110.
constexpr int SMEM_CARVEOUT = 50;  // percent of the largest shared-memory size
template <typename... P, typename... A>
cudaError_t launch_with(bool early, size_t smem, void (*kernel)(P...), dim3 grid, dim3 block,
                        cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t c{};
    c.dynamicSmemBytes = smem;
    c.gridDim = grid;
    c.blockDim = block;
    c.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at[0].val.sharedMemCarveout = SMEM_CARVEOUT;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = early ? 2 : 1;
    return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t s, A&&... args) {
    return launch_with(false, 0, kernel, grid, block, s, std::forward<A>(args)...);
}
// for kernels that begin with step_enter
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t s, A&&... args) {
    return launch_with(true, 0, kernel, grid, block, s, std::forward<A>(args)...);
}

template <typename T, typename C>
const Coll<C>& coll_of(const Launch& L);
template <>
const Coll<double>& coll_of<double, double>(const Launch& L) {
    return L.kd;
}
template <>
const Coll<float>& coll_of<float, float>(const Launch& L) {
    return L.kf;
}
template <>
const Coll<dfloat>& coll_of<double, dfloat>(const Launch& L) {
    return L.kff;
}

template <typename T, typename C, int CPT>
cudaError_t bulk_cpt(const void* src, void* dst, const Launch& L) {
    dim3 grid(L.g.ntx, L.g.nty, L.g.ntz);
    const auto& k = coll_of<typename std::conditional<(sizeof(T) < 4), C, T>::type, C>(L);
    const auto go = [&](auto kernel) {
        return launch_with(L.gate != nullptr, 0, kernel, grid, L.block, L.stream, (const T*)src, (T*)dst,
                           L.g, k, L.parts, L.cp.np, L.all_tiles, L.status, (const int*)L.gate,
                           L.gate_key);
    };
    if constexpr (sizeof(T) >= 4 && !std::is_same<C, dfloat>::value)
        if (L.gate)
            return L.nostream ? go(k_bulk<T, C, true, CPT, true>) : go(k_bulk<T, C, false, CPT, true>);
    return L.nostream ? go(k_bulk<T, C, true, CPT, false>) : go(k_bulk<T, C, false, CPT, false>);
}

// k_bulk takes two z cells per thread in FP32, one elsewhere.
template <typename T, typename C = T>
cudaError_t bulk_t(const void* src, void* dst, const Launch& L) {
    if constexpr (sizeof(T) == 2) {
        // 16-bit sweep, two cells per thread: x-neighbours as words for even nx
        // without open boundaries, z-neighbours otherwise; the first sweep
        // after set-up (no stream) takes the per-cell kernel
        const int np = L.all_tiles ? 0 : L.cp.np;
        if (!L.nostream && L.g.nx % 2 == 0 && L.g.bc_z != 2) {
            const int w = pair_width(L.g.nx);
            const dim3 grid((L.g.nx / 2 + w - 1) / w, L.g.ny, L.g.nz);
            const auto go = [&](auto kernel) {
                return launch(kernel, grid, w, L.stream, (const T*)src, (T*)dst, L.g, L.kf, L.parts,
                              np, L.status);
            };
            return w == 96 ? go(k_bulk_pair<T, 96>)
                           : (w == 32 ? go(k_bulk_pair<T, 32>) : go(k_bulk_pair<T, 64>));
        }
        const long long plane = (long long)L.g.nx * L.g.ny;
        if (!L.nostream && plane < (1LL << 31))
            return launch(k_bulk_zpair<T>,
                          dim3((unsigned)((plane + ZPAIR_THREADS - 1) / ZPAIR_THREADS), 1,
                               (L.g.nz + 1) / 2),
                          ZPAIR_THREADS, L.stream, (const T*)src, (T*)dst, L.g, L.kf, L.parts, np,
                          L.status);
    }
    return bulk_cpt<T, C, sizeof(T) == 4 ? 2 : 1>(src, dst, L);  // g.tz of set_tiles
}

template <typename T, int KIND>
cudaError_t near_kind(const void* src, void* dst, const Launch& L) {
    using C = typename ComputeOf<T>::type;
    const dim3 grid((unsigned)L.near_nblk, L.cp.np), block(NEAR_THREADS);
    const size_t smem = sizeof(DevParticle) * L.cp.np;
    const auto& k = coll_of<C, C>(L);
    const GeoMap gm{L.map, L.map_ext[0], L.map_ext[1], L.map_ext[2]};
    // 16 bits: not launched ahead of the map's end, where its registers would be
    // held back from the bulk sweep for longer
    constexpr bool early = sizeof(T) > 2;
    if constexpr (KIND != 2)  // (MEM set-up collides in place: its sweeps always stream)
        if (L.nostream)
            return launch_with(early, smem, k_near<T, C, KIND, true>, grid, block, L.stream,
                               (const T*)src, (T*)dst, L.g, k, L.cp, L.parts, gm, L.partials,
                               L.status, L.gate, L.gate_key);
    return launch_with(early, smem, k_near<T, C, KIND, false>, grid, block, L.stream, (const T*)src,
                       (T*)dst, L.g, k, L.cp, L.parts, gm, L.partials, L.status, L.gate, L.gate_key);
}

template <typename T, int KIND>
cudaError_t sweep_kind(const void* src, void* dst, const Launch& L) {
    const unsigned nblk = (unsigned)L.near_nblk;
    const dim3 grid(nblk * L.cp.np + (unsigned)((L.g.n + NEAR_THREADS - 1) / NEAR_THREADS));
    const GeoMap gm{L.map, L.map_ext[0], L.map_ext[1], L.map_ext[2]};
    return launch_with(true, sizeof(DevParticle) * L.cp.np, k_sweep<T, T, KIND>, grid,
                       dim3(NEAR_THREADS), L.stream, (const T*)src, (T*)dst, L.g, coll_of<T, T>(L),
                       L.cp, L.parts, gm, L.partials, L.status, nblk);
}

template <typename T>
cudaError_t near_t(const void* src, void* dst, const Launch& L) {
    if (L.cp.np <= 0) return cudaSuccess;
    if (L.cp.kind == 1) return near_kind<T, 1>(src, dst, L);
    if (L.cp.kind == 2) return near_kind<T, 2>(src, dst, L);
    return near_kind<T, 0>(src, dst, L);
}

template <typename T>
cudaError_t refill_t(const void* srcB, void* dst, const Launch& L, const DevParticle* po,
                     const DevParticle* pn, int extrapolate, double* charge_part) {
    using C = typename ComputeOf<T>::type;
    if (L.cp.np <= 0) return cudaSuccess;
    const int side = L.refill_side;
    dim3 grid((unsigned)refill_blocks(side), L.cp.np, 1);
    return launch_after(k_refill<T, C>, grid, REFILL_THREADS, L.stream, (const T*)srcB, (T*)dst, L.g,
                  coll_of<C, C>(L), L.cp, po, pn, extrapolate, side, L.status, charge_part);
}

template <typename T>
cudaError_t macro_t(const void* state, const Launch& L, int what, void* out) {
    using C = typename ComputeOf<T>::type;
    unsigned blocks = (unsigned)((L.g.n + 255) / 256);
    const auto& k = coll_of<C, C>(L);
    const double fx = L.kd.fx, fy = L.kd.fy, fz = L.kd.fz;
    if (L.nostream)
        k_macro<T, C, true><<<blocks, 256, 0, L.stream>>>((const T*)state, L.g, k, L.cp, L.parts,
                                                          fx, fy, fz, what, out);
    else
        k_macro<T, C, false><<<blocks, 256, 0, L.stream>>>((const T*)state, L.g, k, L.cp, L.parts,
                                                           fx, fy, fz, what, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t init_eq_t(void* dst, const Launch& L, double rho, double ux, double uy, double uz) {
    unsigned blocks = (unsigned)((L.g.n + 255) / 256);
    k_init_eq<T><<<blocks, 256, 0, L.stream>>>((T*)dst, L.g, rho, ux, uy, uz, L.kd.rho0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t to_f64_t(const void* in, double* out, long long count, long long ncell,
                     cudaStream_t s) {
    unsigned blocks = (unsigned)((count + 255) / 256);
    k_to_f64<T><<<blocks, 256, 0, s>>>((const T*)in, out, count, ncell);
    return cudaGetLastError();
}

template <typename T>
cudaError_t from_f64_t(const double* in, void* dst, long long count, long long ncell,
                       cudaStream_t s) {
    unsigned blocks = (unsigned)((count + 255) / 256);
    k_from_f64<T><<<blocks, 256, 0, s>>>(in, (T*)dst, count, ncell);
    return cudaGetLastError();
}
}  // namespace

// storage codes: ST_F64 0, ST_F32 1, ST_F16 4, ST_BF16 5 (FP64 is also the
// state of the float-float (2) and fixed-point (3) bulk modes)
cudaError_t launch_bulk(int storage, const void* src, void* dst, const Launch& L) {
    switch (storage) {
        case 2: return bulk_t<double, dfloat>(src, dst, L);
        case 1: return bulk_t<float>(src, dst, L);
        case 4: return bulk_t<__half, float>(src, dst, L);
        case 5: return bulk_t<__nv_bfloat16, float>(src, dst, L);
        default: return bulk_t<double>(src, dst, L);
    }
}
cudaError_t launch_near(int storage, const void* src, void* dst, const Launch& L) {
    switch (storage) {
        case 1: return near_t<float>(src, dst, L);
        case 4: return near_t<__half>(src, dst, L);
        case 5: return near_t<__nv_bfloat16>(src, dst, L);
        default: return near_t<double>(src, dst, L);
    }
}
bool sweep_fused(const Launch& L, int bulk_mode) {
    return L.cp.np > 0 && (L.cp.kind == 1 || L.cp.kind == 2) && !L.nostream &&
           (bulk_mode == 0 || bulk_mode == 1) && L.g.n <= SWEEP_FUSED_CELLS;
}
bool sweep_beside(const Launch& L, int bulk_mode, int sms) {
    const long long blocks = (long long)L.g.ntx * L.g.nty * L.g.ntz;
    const int waves = L.cp.kind == 2 ? 6 : 4;
    return L.cp.np > 0 && L.cp.kind != 0 && bulk_mode == 1 && L.near_nblk * L.cp.np <= 8LL * sms &&
           blocks <= (long long)waves * BulkShape<float, float>::blocks * sms;
}
cudaError_t launch_sweep(int storage, const void* src, void* dst, const Launch& L) {
    if (storage == 1)
        return L.cp.kind == 1 ? sweep_kind<float, 1>(src, dst, L) : sweep_kind<float, 2>(src, dst, L);
    return L.cp.kind == 1 ? sweep_kind<double, 1>(src, dst, L) : sweep_kind<double, 2>(src, dst, L);
}
cudaError_t launch_refill(int storage, const void* srcB, void* dst, const Launch& L,
                          const DevParticle* p_old, const DevParticle* p_new, int extrapolate,
                          double* charge_part) {
    switch (storage) {
        case 1: return refill_t<float>(srcB, dst, L, p_old, p_new, extrapolate, charge_part);
        case 4: return refill_t<__half>(srcB, dst, L, p_old, p_new, extrapolate, charge_part);
        case 5:
            return refill_t<__nv_bfloat16>(srcB, dst, L, p_old, p_new, extrapolate, charge_part);
        default: return refill_t<double>(srcB, dst, L, p_old, p_new, extrapolate, charge_part);
    }
}
cudaError_t launch_charge_total(const Launch& L, const double* charge_part, double* charge) {
    if (L.cp.np <= 0) return cudaSuccess;
    return launch_after(k_charge_total, L.cp.np, 192, L.stream, refill_blocks(L.refill_side), charge_part,
                  charge);
}
cudaError_t launch_macro(int storage, const void* state, const Launch& L, int what, void* out) {
    switch (storage) {
        case 1: return macro_t<float>(state, L, what, out);
        case 4: return macro_t<__half>(state, L, what, out);
        case 5: return macro_t<__nv_bfloat16>(state, L, what, out);
        default: return macro_t<double>(state, L, what, out);
    }
}
cudaError_t launch_init_eq(int storage, void* dst, const Launch& L, double rho, double ux,
                           double uy, double uz) {
    switch (storage) {
        case 1: return init_eq_t<float>(dst, L, rho, ux, uy, uz);
        case 4: return init_eq_t<__half>(dst, L, rho, ux, uy, uz);
        case 5: return init_eq_t<__nv_bfloat16>(dst, L, rho, ux, uy, uz);
        default: return init_eq_t<double>(dst, L, rho, ux, uy, uz);
    }
}
cudaError_t launch_to_f64(int storage, const void* in, double* out, long long count,
                          long long ncell, cudaStream_t s) {
    switch (storage) {
        case 1: return to_f64_t<float>(in, out, count, ncell, s);
        case 4: return to_f64_t<__half>(in, out, count, ncell, s);
        case 5: return to_f64_t<__nv_bfloat16>(in, out, count, ncell, s);
        default:
            return cudaMemcpyAsync(out, in, sizeof(double) * count, cudaMemcpyDeviceToDevice, s);
    }
}
cudaError_t launch_from_f64(int storage, const double* in, void* dst, long long count,
                            long long ncell, cudaStream_t s) {
    switch (storage) {
        case 1: return from_f64_t<float>(in, dst, count, ncell, s);
        case 4: return from_f64_t<__half>(in, dst, count, ncell, s);
        case 5: return from_f64_t<__nv_bfloat16>(in, dst, count, ncell, s);
        default:
            return cudaMemcpyAsync(dst, in, sizeof(double) * count, cudaMemcpyDeviceToDevice, s);
    }
}
cudaError_t launch_map(const Launch& L) {
    if (L.cp.np <= 0 || L.cp.kind == 0) return cudaSuccess;
    dim3 grid((L.map_ext[0] + 31) / 32, L.map_ext[1], L.map_ext[2] * L.cp.np);
    if (L.cp.kind == 2)
        return launch_after(k_map<2>, grid, 32, L.stream, L.g, L.cp, L.parts, L.map, L.map_ext[0],
                      L.map_ext[1], L.map_ext[2]);
    return launch_after(k_map<1>, grid, 32, L.stream, L.g, L.cp, L.parts, L.map, L.map_ext[0], L.map_ext[1],
                  L.map_ext[2]);
}

cudaError_t launch_finalize(const Launch& L, int nsub, double* force_out, const double* charge) {
    if (L.cp.np <= 0) return cudaSuccess;
    return launch_after(k_finalize, L.cp.np, FIN_THREADS, L.stream, L.cp.np, L.near_nblk, L.partials, nsub,
                  force_out, charge, L.gate);
}
cudaError_t launch_rigid_body(const Launch& L, const double* force, double gx, double gy,
                              double gz, double dt, int wall_contact) {
    if (L.cp.np <= 0) return cudaSuccess;
    return launch_after(k_rigid, L.cp.np, 32, L.stream, L.g, L.parts, L.parts_prev, force, L.kd.rho0, gx,
                  gy, gz, dt, wall_contact, L.status);
}
cudaError_t launch_finalize_rigid(const Launch& L, int nsub, double* force, const double* charge,
                                  double gx, double gy, double gz, int wall_contact) {
    if (L.cp.np <= 0) return cudaSuccess;
    return launch_after(k_finalize_rigid, L.cp.np, FIN_THREADS, L.stream, L.g, L.cp.np,
                  L.near_nblk, L.partials, nsub, force, charge, L.parts, L.parts_prev,
                  L.kd.rho0, gx, gy, gz, (double)nsub, wall_contact, L.status, L.gate);
}
cudaError_t launch_set_particles(const Launch& L, const ParticleUpload& up, int n, DevParticle* parts,
                                 DevParticle* prev, DevParticle* old) {
    return launch_after(k_set_particles, 1, MAX_PARTICLES, L.stream, L.g, up, n, parts, prev, old);
}


cudaError_t launch_batch_regions(BatchCase* cases, int n, cudaStream_t s) {
    k_batch_regions<<<(n + 63) / 64, 64, 0, s>>>(cases, n);
    return cudaGetLastError();
}
cudaError_t launch_batch_init(BatchCase* cases, int n, long long max_cells, cudaStream_t s) {
    dim3 grid((unsigned)((max_cells + 255) / 256), n, 1);
    k_batch_init<<<grid, 256, 0, s>>>(cases);
    return cudaGetLastError();
}
cudaError_t launch_batch_map(BatchCase* cases, BatchList l, long long total, cudaStream_t s) {
    if (l.n == 0 || total == 0) return cudaSuccess;
    k_batch_map<<<(unsigned)total, 32, 0, s>>>(cases, l);
    return cudaGetLastError();
}
cudaError_t launch_batch_near(BatchCase* cases, BatchList l, long long total, int sub,
                              int* status, cudaStream_t s) {
    if (l.n == 0 || total == 0) return cudaSuccess;
    k_batch_near<<<(unsigned)total, NEAR_THREADS, 0, s>>>(cases, l, sub, status);
    return cudaGetLastError();
}
cudaError_t launch_batch_bulk(BatchCase* cases, BatchList l, long long total, int grid,
                              int* status, cudaStream_t s) {
    if (l.n == 0 || total == 0) return cudaSuccess;
    const int chunk = (int)std::min<long long>(4, std::max<long long>(1, total / BATCH_CHUNK_ITEMS));
    const long long chunks = (total + chunk - 1) / chunk;
    const unsigned gsz = (unsigned)(grid <= 0 || chunks < grid ? chunks : grid);
    k_batch_bulk<<<gsz, BATCH_THREADS, 0, s>>>(cases, l, total, chunk, status);
    return cudaGetLastError();
}
cudaError_t launch_batch_swap(BatchCase* cases, BatchList l, cudaStream_t s) {
    if (l.n == 0) return cudaSuccess;
    k_batch_swap<<<(l.n + 63) / 64, 64, 0, s>>>(cases, l);
    return cudaGetLastError();
}
cudaError_t launch_batch_finalize(BatchCase* cases, int n, cudaStream_t s) {
    k_batch_finalize<<<n, FIN_THREADS, 0, s>>>(cases);
    return cudaGetLastError();
}
cudaError_t launch_batch_charge_total(BatchCase* cases, int n, cudaStream_t s) {
    k_batch_charge_total<<<n, 192, 0, s>>>(cases);
    return cudaGetLastError();
}
cudaError_t launch_batch_rigid(BatchCase* cases, int n, int* status, cudaStream_t s) {
    k_batch_rigid<<<n, 32, 0, s>>>(cases, status);
    return cudaGetLastError();
}
// Device time stamp (the GPU's nanosecond global timer): end = 0 keeps it in
// p[0]; end = 1 adds the span since p[0] to p[1] and counts it in p[2].  One
// thread; launched on the stream of the work it brackets.
__global__ void k_stamp(unsigned long long* p, int end) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (!end) {
        p[0] = t;
    } else {
        p[1] += t - p[0];
        p[2] += 1;
    }
}
cudaError_t launch_stamp(unsigned long long* p, int end, cudaStream_t s) {
    k_stamp<<<1, 1, 0, s>>>(p, end);
    return cudaGetLastError();
}

cudaError_t launch_batch_refill(BatchCase* cases, BatchList l, long long total, int* status,
                                cudaStream_t s) {
    if (l.n == 0 || total == 0) return cudaSuccess;
    k_batch_refill<<<(unsigned)total, REFILL_THREADS, 0, s>>>(cases, l, status);
    return cudaGetLastError();
}
int batch_bulk_blocks_per_sm() {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch_bulk, BATCH_THREADS, 0);
    return nb > 0 ? nb : 1;
}

}  // namespace lbmgpu
