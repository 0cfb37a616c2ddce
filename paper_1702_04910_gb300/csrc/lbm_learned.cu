// Learned force correction: the near-surface feature stencil of a particle,
// a small MLP (512 -> 64 -> 64 -> 6, tanh) with hand-written forward,
// backward and Adam kernels, and its use inside the coupled step
// (declarations and contracts in include/lbm_gb300.h).
//
// The paper has no learned component; this is an extension that corrects the
// hydrodynamic force and torque of a coarsely resolved sphere (Sec. 4 studies
// how that force converges with the resolution D) towards a finely resolved
// run of the same method.
//
// Features of particle p (all FP32, computed in FP64):
//   [0,125)    solid indicator at a 5 x 5 x 5 grid of points around the
//              centre X_p, spacing h = (R + 2) / 2 (the grid spans the sphere
//              and its two-cell near-surface layer), trilinear from the cell
//              centres: PSM total solid fraction (min(sum eps_s, 1)), MEM
//              1 for a solid cell, 0 for a fluid cell (both read from the
//              step's geometry map);
//   [125,500)  (u - U_p) / u_ref at the same points, x then y then z blocks;
//              u = j~ / rho0 of the stored post-collision PDFs, the body
//              velocity in a MEM solid cell, 0 beyond a closed wall;
//   [500,512)  U_p / u_ref, Omega_p R / u_ref, F / (rho0 u_ref^2 D^2),
//              T / (rho0 u_ref^2 D^3) (F, T: this step's hydrodynamic force).
// Outputs: the correction (dF, dT) in the same units as the last two blocks.
#include <cuda_pipeline.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/lbm_gb300.h"
#include "lbm_launch.h"

using namespace lbmgpu;

namespace lbmgpu {

constexpr int FIN = LBM_MLP_IN, FH = LBM_MLP_HIDDEN, FOUT = LBM_MLP_OUT;
constexpr int NSTEN = 5, NPTS = NSTEN * NSTEN * NSTEN;
// parameter offsets (weights stored [in][out]: output index fastest)
constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + FIN * FH;
constexpr int OFF_W2 = OFF_B1 + FH;
constexpr int OFF_B2 = OFF_W2 + FH * FH;
constexpr int OFF_W3 = OFF_B2 + FH;
constexpr int OFF_B3 = OFF_W3 + FH * FOUT;
constexpr int NPARAM = OFF_B3 + FOUT;
static_assert(NPARAM == LBM_MLP_PARAMS, "parameter count");
// normalisation block: input mean [FIN], input 1/std [FIN], output scale [FOUT]
constexpr int NORM_MU = 0, NORM_IS = FIN, NORM_OS = 2 * FIN, NNORM = 2 * FIN + FOUT;

// ---------------------------------------------------------------------------
// feature stencil: 8 threads per grid point, one per corner of its trilinear
// cell, FEAT_POINTS points per block, blocks (chunk, particle).
//
// Bound by latency: 8 corners x (19 loads, ~60 FP64 operations) per point.
// With a thread per point on one SM they came one after another (53 us for one
// particle); across 8 lanes and 8 SMs each thread has one corner, and the
// corners are added by a butterfly (12 us, cold L2).
constexpr int FEAT_POINTS = 16, FEAT_THREADS = 8 * FEAT_POINTS;
constexpr int FEAT_CHUNKS = (NPTS + FEAT_POINTS - 1) / FEAT_POINTS;
template <typename T>
__global__ void __launch_bounds__(FEAT_THREADS)
    k_features(const T* __restrict__ state, Geom g, Coupl cp, const DevParticle* __restrict__ parts,
               GeoMap gm, const double* __restrict__ force, double u_ref, float* __restrict__ feat) {
    __shared__ DevParticle sp[MAX_PARTICLES];
    const int nd = cp.np * (int)(sizeof(DevParticle) / sizeof(double));
    for (int i = threadIdx.x; i < nd; i += blockDim.x)
        reinterpret_cast<double*>(sp)[i] = reinterpret_cast<const double*>(parts)[i];
    __syncthreads();
    const int p = blockIdx.y;
    const DevParticle& P = sp[p];
    float* out = feat + (long long)p * FIN;
    const int s = blockIdx.x * FEAT_POINTS + threadIdx.x / 8, corner = threadIdx.x % 8;
    double eps = 0.0, u[3] = {0.0, 0.0, 0.0};
    if (s < NPTS) {
        const int ijk[3] = {s % NSTEN, (s / NSTEN) % NSTEN, s / (NSTEN * NSTEN)};
        const double h = 0.5 * (P.r + NEAR_HALO);
        int at[3];
        double w = 1.0;
        for (int a = 0; a < 3; ++a) {
            const double c = (P.x[a] + (ijk[a] - 2) * h) - 0.5;  // cell-centre coordinate
            const double fl = floor(c), fr = c - fl;
            const int d = (corner >> a) & 1;
            at[a] = (int)fl + d;
            w *= d ? fr : 1.0 - fr;
        }
        const int X = wrap_i(at[0], g.nx), Y = wrap_i(at[1], g.ny);
        int Z = at[2];
        bool in = true;  // beyond a resting wall: eps 0, u 0
        if (g.bc_z) in = Z >= 0 && Z < g.nz;
        else Z = wrap_i(Z, g.nz);
        if (in) {
            // the step's geometry map (cells outside every region box are
            // fluid / uncovered)
            double e = 0.0, v[3] = {0.0, 0.0, 0.0};
            int own = 0;
            if (cp.kind == 2) {
                own = mapped_owner(g, sp, cp.np, gm, X, Y, Z);
                e = own ? 1.0 : 0.0;
            } else if (cp.kind == 1) {
                const double n3 = (double)cp.subsample * cp.subsample * cp.subsample;
                for (int q = 0; q < cp.np; ++q) {
                    int ox, oy, oz;
                    if (region_offsets(g, sp[q].reg, X, Y, Z, ox, oy, oz)) e += map_at(gm, q, ox, oy, oz) / n3;
                }
                e = e < 1.0 ? e : 1.0;
            }
            if (own) {
                body_velocity(g, sp[own - 1], X + 0.5, Y + 0.5, Z + 0.5, v[0], v[1], v[2]);
            } else {
                const long long idx = lin(g, X, Y, Z);
#pragma unroll
                for (int q = 1; q < NQ; ++q) {
                    const double f = ld_pdf(state + (long long)q * g.n + idx, q);
                    if (cx(q)) v[0] += cx(q) > 0 ? f : -f;
                    if (cy(q)) v[1] += cy(q) > 0 ? f : -f;
                    if (cz(q)) v[2] += cz(q) > 0 ? f : -f;
                }
                for (int a = 0; a < 3; ++a) v[a] /= cp.rho0;
            }
            eps = w * e;
            for (int a = 0; a < 3; ++a) u[a] = w * v[a];
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        eps += __shfl_xor_sync(0xffffffffu, eps, o);
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] += __shfl_xor_sync(0xffffffffu, u[a], o);
    }
    if (s < NPTS && corner < 4) {
        const int a = corner - 1;
        const double ua = corner < 2 ? u[0] : (corner == 2 ? u[1] : u[2]);
        out[NPTS * corner + s] = corner == 0 ? (float)eps : (float)((ua - P.u[a < 0 ? 0 : a]) / u_ref);
    }
    if (blockIdx.x == 0 && threadIdx.x < 3) {
        const int a = threadIdx.x;
        const double D = P.d, fs = cp.rho0 * u_ref * u_ref * D * D, ts = fs * D;
        const double* F = force + 6 * p;
        out[4 * NPTS + a] = (float)(P.u[a] / u_ref);
        out[4 * NPTS + 3 + a] = (float)(P.w[a] * P.r / u_ref);
        out[4 * NPTS + 6 + a] = (float)(F[a] / fs);
        out[4 * NPTS + 9 + a] = (float)(F[3 + a] / ts);
    }
}

// ---------------------------------------------------------------------------
// MLP inference: one 64-thread block per sample.  Inputs are normalised on
// load, x^ = (x - mu) / sigma; the network output y^ times out_scale is
// returned.  With clip > 0 a sample with any |x^_i| > clip (outside the
// training data) gets y = 0: the caller's plain force stands.
__global__ void __launch_bounds__(FH)
    k_mlp_forward(const float* __restrict__ P, const float* __restrict__ norm,
                  const float* __restrict__ X, int n, float* __restrict__ Y, float clip) {
    __shared__ float xs[FIN], h1[FH], h2[FH];
    const int smp = blockIdx.x, u = threadIdx.x;
    if (smp >= n) return;
    const float* x = X + (long long)smp * FIN;
    int out_of_range = 0;
    for (int i = u; i < FIN; i += FH) {
        const float v = (x[i] - norm[NORM_MU + i]) * norm[NORM_IS + i];
        xs[i] = v;
        out_of_range |= clip > 0.0f && !(fabsf(v) <= clip);
    }
    if (__syncthreads_or(out_of_range)) {
        if (u < FOUT) Y[(long long)smp * FOUT + u] = 0.0f;
        return;
    }
    float a = P[OFF_B1 + u];
    for (int i = 0; i < FIN; ++i) a = fmaf(P[OFF_W1 + i * FH + u], xs[i], a);
    h1[u] = tanhf(a);
    __syncthreads();
    a = P[OFF_B2 + u];
    for (int v = 0; v < FH; ++v) a = fmaf(P[OFF_W2 + v * FH + u], h1[v], a);
    h2[u] = tanhf(a);
    __syncthreads();
    if (u < FOUT) {
        a = P[OFF_B3 + u];
        for (int v = 0; v < FH; ++v) a = fmaf(P[OFF_W3 + v * FOUT + u], h2[v], a);
        Y[(long long)smp * FOUT + u] = a * norm[NORM_OS + u];
    }
}

// Forward pass and backward deltas of S samples per block, for the loss
// L = 1/(2n) sum_s sum_k w_k (y^_sk - t_sk / os_k)^2, w_k = (os_k / max_j os_j)^2
// (each output's error in the units of the largest target): H1, H2 the hidden
// values, D1, D2, D3 = dL/dz of the three layers (z: pre-activations), and the
// block's loss terms added in a fixed order into loss_b[block].
//
// What bounds it: the FP32 FMAs of the first layer (32,768 per sample) and,
// with one block per sample as before, the 150 KB of parameters each block
// reads from L2 (1.1 GB for 7200 samples).  A thread keeps S / 8 samples of one
// unit, so a weight read serves S samples of the block, and the inputs come
// from shared memory four at a time.  Every sum keeps the order of the
// one-sample form (i ascending from the bias), so the values are the same
// bits.  S follows n (gradient()).  7200 samples, cold L2: forward and delta
// kernels 175 us -> 57 us (long scoreboard first: 8 warps per scheduler).
constexpr int PASS_GROUPS = 8, PASS_THREADS = PASS_GROUPS * FH;
template <int S>
__global__ void __launch_bounds__(PASS_THREADS, 2)
    k_mlp_pass(const float* __restrict__ P, const float* __restrict__ norm,
               const float* __restrict__ X, const float* __restrict__ Tt, int n,
               float* __restrict__ H1, float* __restrict__ H2, float* __restrict__ D1,
               float* __restrict__ D2, float* __restrict__ D3, double* __restrict__ loss_b) {
    constexpr int R = S / PASS_GROUPS;  // samples per thread
    extern __shared__ float4 pass_smem[];
    float* xs = reinterpret_cast<float*>(pass_smem);  // [S][FIN]; then the arrays below
    __shared__ float h1[S][FH], h2[S][FH], d2[S][FH];
    __shared__ __align__(16) float w2[FH][FH + 1];
    __shared__ float d3[S][FOUT];
    __shared__ double ls[S];
    const int tid = threadIdx.x, u = tid % FH, g = tid / FH;
    const int s0 = blockIdx.x * S;
    static_assert(PASS_THREADS == FIN, "one input column per thread");
    const float mu = norm[NORM_MU + tid], is = norm[NORM_IS + tid];
#pragma unroll 8
    for (int s = 0; s < S; ++s)
        xs[s * FIN + tid] =
            s0 + s < n ? (X[(long long)(s0 + s) * FIN + tid] - mu) * is : 0.0f;
    // W1 in chunks of WC rows through w2's space, WS chunks in flight
    constexpr int WC = 16, WS = 4;
    float (*wc)[WC * FH] = reinterpret_cast<float (*)[WC * FH]>(&w2[0][0]);
    static_assert(sizeof(float) * WS * WC * FH <= sizeof(w2) && WC * FH == 2 * PASS_THREADS, "chunk");
    const auto chunk = [&](int c) {
        if (c < FIN / WC)
            for (int e = tid; e < WC * FH; e += PASS_THREADS)
                __pipeline_memcpy_async(&wc[c % WS][e], P + OFF_W1 + c * WC * FH + e, sizeof(float));
        __pipeline_commit();
    };
    float acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = P[OFF_B1 + u];
    for (int c = 0; c < WS - 1; ++c) chunk(c);
    for (int c = 0; c < FIN / WC; ++c) {
        __pipeline_wait_prior(WS - 2);
        __syncthreads();  // chunk c is in place and chunk c - 1 is done with
        chunk(c + WS - 1);
        const float* wv = wc[c % WS];
#pragma unroll
        for (int i = 0; i < WC; i += 4) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 x =
                    *reinterpret_cast<const float4*>(xs + (g * R + r) * FIN + c * WC + i);
                acc[r] = fmaf(wv[(i + 0) * FH + u], x.x, acc[r]);
                acc[r] = fmaf(wv[(i + 1) * FH + u], x.y, acc[r]);
                acc[r] = fmaf(wv[(i + 2) * FH + u], x.z, acc[r]);
                acc[r] = fmaf(wv[(i + 3) * FH + u], x.w, acc[r]);
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < FH * FH; e += PASS_THREADS) w2[e / FH][e % FH] = P[OFF_W2 + e];
#pragma unroll
    for (int r = 0; r < R; ++r) h1[g * R + r][u] = tanhf(acc[r]);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = P[OFF_B2 + u];
#pragma unroll 4
    for (int v = 0; v < FH; ++v) {
        const float w = w2[v][u];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = fmaf(w, h1[g * R + r][v], acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) h2[g * R + r][u] = tanhf(acc[r]);
    __syncthreads();
    const float inv_n = 1.0f / (float)n;
    float smax = norm[NORM_OS];
    for (int k = 1; k < FOUT; ++k) smax = fmaxf(smax, norm[NORM_OS + k]);
    for (int e = tid; e < S * FOUT; e += PASS_THREADS) {
        const int s = e / FOUT, k = e % FOUT;
        float a = P[OFF_B3 + k];
        for (int v = 0; v < FH; ++v) a = fmaf(P[OFF_W3 + v * FOUT + k], h2[s][v], a);
        const float rr = norm[NORM_OS + k] / smax, w = rr * rr;
        float err = 0.0f;
        if (s0 + s < n) {
            err = a - Tt[(long long)(s0 + s) * FOUT + k] / norm[NORM_OS + k];
            D3[(long long)(s0 + s) * FOUT + k] = w * err * inv_n;
        }
        d3[s][k] = w * err * inv_n;
        xs[e] = w * err * err;  // loss terms (the inputs are done with)
    }
    __syncthreads();
    if (tid < S) {
        double l = 0.0;
        for (int k = 0; k < FOUT; ++k) l += 0.5 * (double)xs[tid * FOUT + k];
        ls[tid] = l;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int s = g * R + r;
        float a = 0.0f;
        for (int k = 0; k < FOUT; ++k) a = fmaf(P[OFF_W3 + u * FOUT + k], d3[s][k], a);
        d2[s][u] = a * (1.0f - h2[s][u] * h2[s][u]);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0f;
#pragma unroll 4
    for (int v = 0; v < FH; ++v) {
        const float w = w2[u][v];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = fmaf(w, d2[g * R + r][v], acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int s = g * R + r;
        if (s0 + s >= n) continue;
        const long long o = (long long)(s0 + s) * FH + u;
        H1[o] = h1[s][u];
        H2[o] = h2[s][u];
        D2[o] = d2[s][u];
        D1[o] = acc[r] * (1.0f - h1[s][u] * h1[s][u]);
    }
    if (tid == 0) {
        double l = 0.0;
        for (int s = 0; s < S; ++s) l += ls[s];
        loss_b[blockIdx.x] = l;
    }
}

// Parameter gradient: dW[i][o] = sum_s a_s[i] d_s[o], db[o] = sum_s d_s[o],
// samples in order (a long training run amplifies any other order).  One block
// per 16 x 16 tile of a weight matrix, 2 x 2 outputs per thread; the tiles of a
// layer's first rows also add its bias.
//
// What bounds it: the chain of n dependent FMAs of every output, 4 cycles
// each, 14.5 us for 7200 samples, and above it the shared-memory reads of the
// 256 outputs that 148 blocks leave to an SM.  The operands pass through
// shared memory sample-fastest, so a thread reads four samples of a row at a
// time (4 16-byte reads for 16 FMAs, no bank conflicts between rows r and
// r + 8); row lengths are compile-time, so a chunk's loads are one address and
// immediate offsets, and the next chunk's are in flight during the sums.
// Before, one thread per parameter read both operands from global memory for
// each FMA.  7200 samples, cold L2: 811 us -> 93 us (two outputs per thread,
// 3 reads for 8 FMAs: 103 us), the same bits; the whole gradient call 977 us
// -> 169 us.  Samples cut into slices and added later would take 56 us, but
// the changed order sends a 3000-step Adam run through spikes of the loss.
constexpr int GT = 16, GRAD_K = 128, GRAD_THREADS = GT * GT / 4;
constexpr int GRAD_T1 = (FIN / GT) * (FH / GT), GRAD_T2 = (FH / GT) * (FH / GT), GRAD_T3 = FH / GT;
struct GradTile {
    __align__(16) float A[GT][GRAD_K + 4];
    __align__(16) float B[GT][GRAD_K + 4];
};
// Tile (i0, o0) of a layer: A [n][LDA] (NORM: normalised on the way), B [n][LDB].
template <int LDA, int LDB, bool NORM, bool BIAS>
__device__ __forceinline__ void grad_tile(GradTile& w, const float* __restrict__ norm,
                                          const float* __restrict__ As,
                                          const float* __restrict__ Bs, int n, int i0, int o0,
                                          float* __restrict__ W, float* __restrict__ bias) {
    const int tid = threadIdx.x;
    // loads: column lc of samples ls, ls + STEP, ... of the chunk
    constexpr int STEP = GRAD_THREADS / GT, PER = GRAD_K / STEP;
    const int lc = tid % GT, ls = tid / GT;
    const float mu = NORM ? norm[NORM_MU + i0 + lc] : 0.0f;
    const float is = NORM ? norm[NORM_IS + i0 + lc] : 1.0f;
    const bool bcol = LDB >= FH || o0 + lc < LDB;
    float ra[PER], rb[PER];
    const auto fetch = [&](int s0) {
        const float* pa = As + (long long)(s0 + ls) * LDA + i0 + lc;
        const float* pb = Bs + (long long)(s0 + ls) * LDB + o0 + lc;
        if (s0 + GRAD_K <= n) {
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                ra[k] = pa[k * STEP * LDA];
                rb[k] = bcol ? pb[k * STEP * LDB] : 0.0f;
            }
        } else {  // samples beyond n add zero (mu: its normalised value)
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const bool in = s0 + ls + k * STEP < n;
                ra[k] = in ? pa[k * STEP * LDA] : mu;
                rb[k] = in && bcol ? pb[k * STEP * LDB] : 0.0f;
            }
        }
    };
    const int ti = tid / 8, to = tid % 8;  // outputs (ti, ti + 8) x (to, to + 8)
    float acc[2][2] = {}, b0 = 0.0f, b1 = 0.0f;
    fetch(0);
    for (int s0 = 0; s0 < n; s0 += GRAD_K) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            w.A[lc][ls + k * STEP] = NORM ? (ra[k] - mu) * is : ra[k];
            w.B[lc][ls + k * STEP] = rb[k];
        }
        __syncthreads();
        if (s0 + GRAD_K < n) fetch(s0 + GRAD_K);
#pragma unroll 4
        for (int s = 0; s < GRAD_K; s += 4) {
            const float4 a0 = *reinterpret_cast<const float4*>(&w.A[ti][s]);
            const float4 a1 = *reinterpret_cast<const float4*>(&w.A[ti + 8][s]);
            const float4 u = *reinterpret_cast<const float4*>(&w.B[to][s]);
            const float4 v = *reinterpret_cast<const float4*>(&w.B[to + 8][s]);
            const auto dot = [](float4 a, float4 b, float c) {
                return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
            };
            acc[0][0] = dot(a0, u, acc[0][0]);
            acc[0][1] = dot(a0, v, acc[0][1]);
            acc[1][0] = dot(a1, u, acc[1][0]);
            acc[1][1] = dot(a1, v, acc[1][1]);
            if (BIAS) {
                b0 = b0 + u.x + u.y + u.z + u.w;
                b1 = b1 + v.x + v.y + v.z + v.w;
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int o = o0 + to + 8 * h;
        if (LDB < FH && o >= LDB) continue;
        W[(i0 + ti) * LDB + o] = acc[0][h];
        W[(i0 + ti + 8) * LDB + o] = acc[1][h];
        if (BIAS && ti == 0) bias[o] = h ? b1 : b0;
    }
}

__global__ void __launch_bounds__(GRAD_THREADS)
    k_mlp_grad(const float* __restrict__ norm, const float* __restrict__ X, int n,
               const float* __restrict__ H1, const float* __restrict__ H2,
               const float* __restrict__ D1, const float* __restrict__ D2,
               const float* __restrict__ D3, float* __restrict__ G) {
    __shared__ GradTile w;
    int t = blockIdx.x;
    constexpr int OT = FH / GT;  // tiles across the 64 outputs of a layer
    if (t < GRAD_T1) {
        const int i0 = t / OT * GT, o0 = t % OT * GT;
        if (i0 == 0) grad_tile<FIN, FH, true, true>(w, norm, X, D1, n, i0, o0, G + OFF_W1, G + OFF_B1);
        else grad_tile<FIN, FH, true, false>(w, norm, X, D1, n, i0, o0, G + OFF_W1, nullptr);
    } else if ((t -= GRAD_T1) < GRAD_T2) {
        grad_tile<FH, FH, false, true>(w, norm, H1, D2, n, t / OT * GT, t % OT * GT, G + OFF_W2,
                                       G + OFF_B2);
    } else {
        grad_tile<FH, FOUT, false, true>(w, norm, H2, D3, n, (t - GRAD_T2) * GT, 0, G + OFF_W3,
                                         G + OFF_B3);
    }
}

// loss = sum of the pass blocks' terms / n: 256 interleaved sums, then a tree
// (a fixed order; before, one thread read all n terms).
__global__ void __launch_bounds__(256)
    k_mlp_loss(const double* __restrict__ loss_b, int nb, int n, double* __restrict__ loss) {
    __shared__ double ls[256];
    double l = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) l += loss_b[b];
    ls[threadIdx.x] = l;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) ls[threadIdx.x] += ls[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = ls[0] / n;
}

// Adam (Kingma & Ba 2015) with bias correction; step t >= 1.
__global__ void k_adam(float* __restrict__ P, float* __restrict__ M, float* __restrict__ V,
                       const float* __restrict__ G, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= NPARAM) return;
    const float g = G[t];
    const float m = b1 * M[t] + (1.0f - b1) * g;
    const float v = b2 * V[t] + (1.0f - b2) * g * g;
    M[t] = m;
    V[t] = v;
    P[t] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// Input mean and 1/std (FP64 sums in sample order; std < 1e-6 -> 1) and the
// output scale: the RMS of each target (samples in order; floored at 1e-12).
__global__ void k_fit_norm(const float* __restrict__ X, const float* __restrict__ Tt, int n,
                           float* __restrict__ norm) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < FIN) {
        double s1 = 0.0;
        for (int s = 0; s < n; ++s) s1 += X[(long long)s * FIN + t];
        const double mu = s1 / n;
        double s2 = 0.0;
        for (int s = 0; s < n; ++s) {
            const double d = X[(long long)s * FIN + t] - mu;
            s2 += d * d;
        }
        const double sd = sqrt(s2 / n);
        norm[NORM_MU + t] = (float)mu;
        norm[NORM_IS + t] = (float)(sd > 1e-6 ? 1.0 / sd : 1.0);
    } else if (t < FIN + FOUT) {
        const int k = t - FIN;
        double s2 = 0.0;
        for (int s = 0; s < n; ++s) {
            const double v = Tt[(long long)s * FOUT + k];
            s2 += v * v;
        }
        const double r = sqrt(s2 / n);
        norm[NORM_OS + k] = (float)(r > 1e-12 ? r : 1e-12);
    }
}

// F += dF * rho0 u_ref^2 D^2, T += dT * rho0 u_ref^2 D^3 (one thread per particle)
__global__ void k_apply_correction(const float* __restrict__ Y, const DevParticle* __restrict__ parts,
                                   int np, double u_ref, double rho0, double* __restrict__ force) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const double D = parts[p].d, fs = rho0 * u_ref * u_ref * D * D, ts = fs * D;
    for (int a = 0; a < 3; ++a) {
        force[6 * p + a] += (double)Y[FOUT * p + a] * fs;
        force[6 * p + 3 + a] += (double)Y[FOUT * p + 3 + a] * ts;
    }
}

template <typename T>
cudaError_t features_t(const void* state, const Launch& L, const double* force, double u_ref,
                       float* feat) {
    const GeoMap gm{L.map, L.map_ext[0], L.map_ext[1], L.map_ext[2]};
    k_features<T><<<dim3(FEAT_CHUNKS, L.cp.np), FEAT_THREADS, 0, L.stream>>>(
        (const T*)state, L.g, L.cp, L.parts, gm, force, u_ref, feat);
    return cudaGetLastError();
}

cudaError_t launch_features(int storage, const void* state, const Launch& L, const double* force,
                            double u_ref, float* feat) {
    if (L.cp.np < 1) return cudaSuccess;
    switch (storage) {
        case 1: return features_t<float>(state, L, force, u_ref, feat);
        case 4: return features_t<__half>(state, L, force, u_ref, feat);
        case 5: return features_t<__nv_bfloat16>(state, L, force, u_ref, feat);
        default: return features_t<double>(state, L, force, u_ref, feat);
    }
}

cudaError_t launch_apply_correction(const float* y, const DevParticle* parts, int np, double u_ref,
                                    double rho0, double* force, cudaStream_t s) {
    if (np < 1) return cudaSuccess;
    k_apply_correction<<<1, 32, 0, s>>>(y, parts, np, u_ref, rho0, force);
    return cudaGetLastError();
}

}  // namespace lbmgpu

// ---------------------------------------------------------------------------
// host side
struct lbm_mlp {
    cudaStream_t stream;
    float* params;  // NPARAM
    float* m;       // Adam first moment
    float* v;       // Adam second moment
    float* grad;    // NPARAM
    float* norm;    // NNORM
    double* loss;   // 1
    int adam_t;
    // per-sample work buffers (grown on demand)
    int cap;
    float *h1, *h2, *d1, *d2, *d3;
    double* loss_b;  // loss terms of the pass's blocks
    char err[512];
};

namespace {

lbm_status mfail(lbm_mlp* m, lbm_status st, const char* msg) {
    if (m) std::snprintf(m->err, sizeof(m->err), "%s", msg);
    return st;
}

lbm_status mcuda(lbm_mlp* m, cudaError_t e, const char* where) {
    if (m) std::snprintf(m->err, sizeof(m->err), "%s: %s (%d)", where, cudaGetErrorString(e), (int)e);
    return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
}

#define MK(m, call, where)                                  \
    do {                                                    \
        cudaError_t e_ = (call);                            \
        if (e_ != cudaSuccess) return mcuda(m, e_, where);  \
    } while (0)

void free_work(lbm_mlp* m) {
    cudaFree(m->h1);
    cudaFree(m->h2);
    cudaFree(m->d1);
    cudaFree(m->d2);
    cudaFree(m->d3);
    cudaFree(m->loss_b);
    m->h1 = m->h2 = m->d1 = m->d2 = m->d3 = nullptr;
    m->loss_b = nullptr;
    m->cap = 0;
}

lbm_status ensure_work(lbm_mlp* m, int n) {
    if (n <= m->cap) return LBM_OK;
    MK(m, cudaStreamSynchronize(m->stream), "mlp sync");
    free_work(m);
    const size_t N = (size_t)n;
    MK(m, cudaMalloc(&m->h1, sizeof(float) * N * FH), "cudaMalloc mlp work");
    MK(m, cudaMalloc(&m->h2, sizeof(float) * N * FH), "cudaMalloc mlp work");
    MK(m, cudaMalloc(&m->d1, sizeof(float) * N * FH), "cudaMalloc mlp work");
    MK(m, cudaMalloc(&m->d2, sizeof(float) * N * FH), "cudaMalloc mlp work");
    MK(m, cudaMalloc(&m->d3, sizeof(float) * N * FOUT), "cudaMalloc mlp work");
    MK(m, cudaMalloc(&m->loss_b, sizeof(double) * N), "cudaMalloc mlp work");
    m->cap = n;
    return LBM_OK;
}

template <int S>
cudaError_t launch_pass(lbm_mlp* m, const float* x, const float* t, int n, int& blocks) {
    blocks = (n + S - 1) / S;
    const int smem = S * FIN * (int)sizeof(float);
    if (smem > 16 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(
            k_mlp_pass<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    k_mlp_pass<S><<<blocks, PASS_THREADS, smem, m->stream>>>(
        m->params, m->norm, x, t, n, m->h1, m->h2, m->d1, m->d2, m->d3, m->loss_b);
    return cudaGetLastError();
}

// forward + deltas + parameter gradient into m->grad and the loss into m->loss
lbm_status gradient(lbm_mlp* m, const float* x, const float* t, int n) {
    lbm_status st = ensure_work(m, n);
    if (st != LBM_OK) return st;
    // samples per block of the pass: 32 once that gives every SM a block
    // (152 x 32 samples), fewer for small sets, whose time is one block's chain
    int blocks = 0;
    MK(m, n >= 152 * 32 ? launch_pass<32>(m, x, t, n, blocks)
                        : (n >= 152 * 16 ? launch_pass<16>(m, x, t, n, blocks)
                                         : launch_pass<8>(m, x, t, n, blocks)),
       "mlp pass launch");
    k_mlp_grad<<<GRAD_T1 + GRAD_T2 + GRAD_T3, GRAD_THREADS, 0, m->stream>>>(
        m->norm, x, n, m->h1, m->h2, m->d1, m->d2, m->d3, m->grad);
    MK(m, cudaGetLastError(), "mlp gradient launch");
    k_mlp_loss<<<1, 256, 0, m->stream>>>(m->loss_b, blocks, n, m->loss);
    MK(m, cudaGetLastError(), "mlp loss launch");
    return LBM_OK;
}

lbm_status read_loss(lbm_mlp* m, double* loss) {
    if (!loss) return LBM_OK;
    MK(m, cudaMemcpyAsync(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream), "loss copy");
    MK(m, cudaStreamSynchronize(m->stream), "loss sync");
    return LBM_OK;
}

}  // namespace

namespace lbmgpu {
// used by the coupled step (lbm_api.cu): y = MLP(x) for n samples on stream s
cudaError_t mlp_infer(const lbm_mlp* m, const float* x, int n, float* y, float clip,
                      cudaStream_t s) {
    if (n < 1) return cudaSuccess;
    k_mlp_forward<<<n, FH, 0, s>>>(m->params, m->norm, x, n, y, clip);
    return cudaGetLastError();
}
}  // namespace lbmgpu

extern "C" {

lbm_status lbm_mlp_create(void* stream, lbm_mlp** out) {
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    lbm_mlp* m = new (std::nothrow) lbm_mlp();
    if (!m) return LBM_ERR_OOM;
    m->stream = (cudaStream_t)stream;
    cudaError_t e = cudaMalloc(&m->params, sizeof(float) * NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&m->m, sizeof(float) * NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&m->v, sizeof(float) * NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&m->grad, sizeof(float) * NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(&m->norm, sizeof(float) * NNORM);
    if (e == cudaSuccess) e = cudaMalloc(&m->loss, sizeof(double));
    if (e == cudaSuccess) e = cudaMemsetAsync(m->params, 0, sizeof(float) * NPARAM, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, sizeof(float) * NPARAM, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, sizeof(float) * NPARAM, m->stream);
    if (e == cudaSuccess) {
        // identity normalisation until set or fitted
        std::vector<float> nrm(NNORM, 1.0f);
        for (int i = 0; i < FIN; ++i) nrm[NORM_MU + i] = 0.0f;
        e = cudaMemcpy(m->norm, nrm.data(), sizeof(float) * NNORM, cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        lbm_mlp_destroy(m);
        return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
    }
    *out = m;
    return LBM_OK;
}

void lbm_mlp_destroy(lbm_mlp* m) {
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    else cudaDeviceSynchronize();
    free_work(m);
    cudaFree(m->params);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->grad);
    cudaFree(m->norm);
    cudaFree(m->loss);
    delete m;
}

const char* lbm_mlp_last_error(const lbm_mlp* m) { return m ? m->err : "no model"; }

lbm_status lbm_mlp_set_params(lbm_mlp* m, const float* host, size_t count) {
    if (!m || !host) return LBM_ERR_ARG;
    if (count != (size_t)NPARAM) return mfail(m, LBM_ERR_ARG, "count must be LBM_MLP_PARAMS");
    MK(m, cudaMemcpyAsync(m->params, host, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, m->stream),
       "params upload");
    MK(m, cudaMemsetAsync(m->m, 0, sizeof(float) * NPARAM, m->stream), "adam reset");
    MK(m, cudaMemsetAsync(m->v, 0, sizeof(float) * NPARAM, m->stream), "adam reset");
    MK(m, cudaStreamSynchronize(m->stream), "params sync");
    m->adam_t = 0;
    return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp* m, float* host, size_t count) {
    if (!m || !host) return LBM_ERR_ARG;
    if (count != (size_t)NPARAM) return mfail(m, LBM_ERR_ARG, "count must be LBM_MLP_PARAMS");
    MK(m, cudaMemcpyAsync(host, m->params, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream),
       "params download");
    MK(m, cudaStreamSynchronize(m->stream), "params sync");
    return LBM_OK;
}

lbm_status lbm_mlp_set_normalization(lbm_mlp* m, const float* host, size_t count) {
    if (!m || !host) return LBM_ERR_ARG;
    if (count != (size_t)NNORM) return mfail(m, LBM_ERR_ARG, "count must be LBM_MLP_NORM");
    MK(m, cudaMemcpyAsync(m->norm, host, sizeof(float) * NNORM, cudaMemcpyHostToDevice, m->stream),
       "normalisation upload");
    MK(m, cudaStreamSynchronize(m->stream), "normalisation sync");
    return LBM_OK;
}

lbm_status lbm_mlp_get_normalization(lbm_mlp* m, float* host, size_t count) {
    if (!m || !host) return LBM_ERR_ARG;
    if (count != (size_t)NNORM) return mfail(m, LBM_ERR_ARG, "count must be LBM_MLP_NORM");
    MK(m, cudaMemcpyAsync(host, m->norm, sizeof(float) * NNORM, cudaMemcpyDeviceToHost, m->stream),
       "normalisation download");
    MK(m, cudaStreamSynchronize(m->stream), "normalisation sync");
    return LBM_OK;
}

lbm_status lbm_mlp_fit_normalization(lbm_mlp* m, const float* x_dev, const float* t_dev, int n) {
    if (!m || !x_dev || !t_dev || n < 1) return mfail(m, LBM_ERR_ARG, "need samples");
    k_fit_norm<<<(FIN + FOUT + 127) / 128, 128, 0, m->stream>>>(x_dev, t_dev, n, m->norm);
    MK(m, cudaGetLastError(), "normalisation launch");
    return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp* m, const float* x_dev, int n, float* y_dev) {
    if (!m || !x_dev || !y_dev || n < 0) return mfail(m, LBM_ERR_ARG, "null buffer");
    MK(m, mlp_infer(m, x_dev, n, y_dev, 0.0f, m->stream), "mlp forward launch");
    return LBM_OK;
}

lbm_status lbm_mlp_gradient(lbm_mlp* m, const float* x_dev, const float* t_dev, int n,
                            float* grad_host, size_t count, double* loss) {
    if (!m || !x_dev || !t_dev || n < 1) return mfail(m, LBM_ERR_ARG, "need samples");
    if (grad_host && count != (size_t)NPARAM) return mfail(m, LBM_ERR_ARG, "count must be LBM_MLP_PARAMS");
    lbm_status st = gradient(m, x_dev, t_dev, n);
    if (st != LBM_OK) return st;
    if (grad_host) {
        MK(m, cudaMemcpyAsync(grad_host, m->grad, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, m->stream),
           "gradient download");
        if (!loss) MK(m, cudaStreamSynchronize(m->stream), "gradient sync");
    }
    return read_loss(m, loss);  // synchronises for both copies
}

lbm_status lbm_mlp_train(lbm_mlp* m, const float* x_dev, const float* t_dev, int n, int steps,
                         float lr, double* loss) {
    if (!m || !x_dev || !t_dev || n < 1 || steps < 0 || !(lr > 0.0f))
        return mfail(m, LBM_ERR_ARG, "need samples, steps >= 0 and lr > 0");
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int it = 0; it < steps; ++it) {
        lbm_status st = gradient(m, x_dev, t_dev, n);
        if (st != LBM_OK) return st;
        ++m->adam_t;
        const float c1 = 1.0f - powf(b1, (float)m->adam_t), c2 = 1.0f - powf(b2, (float)m->adam_t);
        k_adam<<<(NPARAM + 255) / 256, 256, 0, m->stream>>>(m->params, m->m, m->v, m->grad, lr, b1, b2,
                                                           eps, c1, c2);
        MK(m, cudaGetLastError(), "adam launch");
    }
    return read_loss(m, loss);  // loss of the last step's parameters before its update
}

}  // extern "C"
