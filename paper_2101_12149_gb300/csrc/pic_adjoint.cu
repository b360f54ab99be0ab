// Adjoint kernels of libpic: the discrete adjoint of one PIC step (the
// differentiation workload's pic_step_adjoint).  Reverse order of the step:
//   k_adj_yee_e / k_adj_yee_b   transposed Yee update (the two discrete curls
//                               are each other's transposes on the periodic
//                               grid), producing the adjoint of J;
//   k_adj_particles             per particle: recompute gather, Boris and
//                               advance from the stored state, then the
//                               adjoints of the Esirkepov deposit, the
//                               advance, the Boris rotation, the drive and
//                               the gather (a scatter into the field
//                               adjoints).
// Particle adjoints are indexed by particle id, so the sorts between steps
// need no reverse pass.  Cell indices and Esirkepov windows are held fixed
// (the derivative of floor() is zero); the periodic wrap is the identity.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "pic_ctx.h"
#include "pic_device.cuh"
#include "pic_step_common.cuh"

namespace pic {

constexpr int kAdjBlock = 256;

template <typename R> struct AdjArgs {
    R* lamx[3];        // adjoint of the position (cell units), by particle id
    R* lamu[3];        // adjoint of the momentum, by particle id
    R* lamE[3];
    R* lamB[3];
    const R* lamJ[3];
    R* lg[6];          // adjoints of E and B at the particles, by slot (see k_adj_scatter)
    const int* id;     // ids of the stored particle state
    double* lamA;      // adjoint of the drive amplitude (accumulated)
    double t;          // time of the step's gather
};

// Reverse sweep of the Boris rotation (boris() in pic_device.cuh): given the
// forward inputs and the adjoint of the new momentum, the adjoints of the old
// momentum, of E and of B at the particle.
template <typename R>
__device__ __forceinline__ void boris_adj(R k, const R E[3], const R B[3], const R u_old[3], const R lam_new[3],
                                          R lam_old[3], R lE[3], R lB[3]) {
    R um[3], t[3], s[3], up[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) um[a] = u_old[a] + k * E[a];
    const R ig = inv_sqrt(R(1) + um[0] * um[0] + um[1] * um[1] + um[2] * um[2]);  // 1 / gamma^-
    const R kg = k * ig;
#pragma unroll
    for (int a = 0; a < 3; ++a) t[a] = kg * B[a];
    const R tt = t[0] * t[0] + t[1] * t[1] + t[2] * t[2];
    const R sc = R(2) / (R(1) + tt);
#pragma unroll
    for (int a = 0; a < 3; ++a) s[a] = sc * t[a];
    up[0] = um[0] + (um[1] * t[2] - um[2] * t[1]);
    up[1] = um[1] + (um[2] * t[0] - um[0] * t[2]);
    up[2] = um[2] + (um[0] * t[1] - um[1] * t[0]);
    const R* g = lam_new;
    R g_um[3], g_up[3], g_s[3], g_t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lE[a] = k * g[a];
        g_um[a] = g[a];
    }
    // u_new = um + up x s + k E
    g_up[0] = s[1] * g[2] - s[2] * g[1];
    g_up[1] = s[2] * g[0] - s[0] * g[2];
    g_up[2] = s[0] * g[1] - s[1] * g[0];
    g_s[0] = g[1] * up[2] - g[2] * up[1];
    g_s[1] = g[2] * up[0] - g[0] * up[2];
    g_s[2] = g[0] * up[1] - g[1] * up[0];
    // up = um + um x t
    g_um[0] += g_up[0] + (t[1] * g_up[2] - t[2] * g_up[1]);
    g_um[1] += g_up[1] + (t[2] * g_up[0] - t[0] * g_up[2]);
    g_um[2] += g_up[2] + (t[0] * g_up[1] - t[1] * g_up[0]);
    g_t[0] = g_up[1] * um[2] - g_up[2] * um[1];
    g_t[1] = g_up[2] * um[0] - g_up[0] * um[2];
    g_t[2] = g_up[0] * um[1] - g_up[1] * um[0];
    // s = sc t, sc = 2 / (1 + |t|^2)
    R g_sc = R(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        g_t[a] += sc * g_s[a];
        g_sc += g_s[a] * t[a];
    }
    const R g_tt = R(-0.5) * sc * sc * g_sc;
    R g_gm = R(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        g_t[a] += R(2) * t[a] * g_tt;
        lB[a] = kg * g_t[a];
        g_gm -= t[a] * g_t[a];
    }
    g_gm *= ig * ig;  // dL/d gamma^- over gamma^-
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        g_um[a] += um[a] * g_gm;
        lam_old[a] = g_um[a];
        lE[a] += k * g_um[a];
    }
}

// Adjoint of the Esirkepov current of component C (cumulative along C,
// transverse T1, T2): J_C(w0,w1,w2) = coef * cum_C(w0) * Q(w1,w2), with
// Q = S0a A_b + dSa B_b, A = S0 + dS/2, B = S0/2 + dS/3 (symmetric in a and
// b).  Accumulates dL/dS0 and dL/ddS per axis; nodes are the window's wrapped
// element offsets per axis.  coef enters with cum (for dL/dQ) and once at the
// end (for dL/dcum), so a window value costs two multiply-adds.
template <int P, typename R, int C>
__device__ __forceinline__ void esirkepov_adj_component(const EsirkAxis<P, R>* ax, const int (*node)[P + 2],
                                                        const R* __restrict__ lamJ, R coef, R (*gS0)[P + 2],
                                                        R (*gdS)[P + 2]) {
    constexpr int NW = P + 2;
    constexpr int T1 = (C + 1) % 3, T2 = (C + 2) % 3;
    R cum[NW - 1], gcum[NW - 1], A2[NW], B2[NW];
    R run = R(0);
#pragma unroll
    for (int w = 0; w < NW - 1; ++w) {
        run += ax[C].dS[w];
        cum[w] = coef * run;
        gcum[w] = R(0);
    }
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        A2[w] = ax[T2].S0[w] + R(0.5) * ax[T2].dS[w];
        B2[w] = R(0.5) * ax[T2].S0[w] + R(1.0 / 3.0) * ax[T2].dS[w];
    }
#pragma unroll
    for (int w1 = 0; w1 < NW; ++w1) {
        const R S0a = ax[T1].S0[w1], dSa = ax[T1].dS[w1];
        const R A1 = S0a + R(0.5) * dSa, B1 = R(0.5) * S0a + R(1.0 / 3.0) * dSa;
#pragma unroll
        for (int w2 = 0; w2 < NW; ++w2) {
            const R Q = S0a * A2[w2] + dSa * B2[w2];
            R gQ = R(0);
#pragma unroll
            for (int w0 = 0; w0 < NW - 1; ++w0) {
                const R M = lamJ[node[C][w0] + node[T1][w1] + node[T2][w2]];
                gQ += M * cum[w0];
                gcum[w0] += M * Q;
            }
            gS0[T1][w1] += gQ * A2[w2];
            gdS[T1][w1] += gQ * B2[w2];
            gS0[T2][w2] += gQ * A1;
            gdS[T2][w2] += gQ * B1;
        }
    }
    // cum(w) = sum_{v <= w} dS(v): dL/ddS(v) = sum_{w >= v} dL/dcum(w)
    R acc = R(0);
#pragma unroll
    for (int w = NW - 2; w >= 0; --w) {
        acc += gcum[w];
        gdS[C][w] += coef * acc;
    }
}

// Gather of one field component with staggering (SX, SY, SZ) together with
// its gradient along the three axes (cell units): the forward value and what
// the reverse sweep needs of the field, in one pass over its nodes.
template <int P, typename R, bool SX, bool SY, bool SZ>
__device__ __forceinline__ R gather_grad(const GatherW<P, R>& G, const R (*dn)[P + 1], const R (*ds)[P + 1],
                                         const R* __restrict__ F, R grad[3]) {
    R v = R(0), g0 = R(0), g1 = R(0), g2 = R(0);
#pragma unroll
    for (int i = 0; i <= P; ++i) {
        const int ox = SX ? G.os[0][i] : G.on[0][i];
        R s0 = R(0), s1 = R(0), s2 = R(0);
#pragma unroll
        for (int j = 0; j <= P; ++j) {
            const R* row = F + ox + (SY ? G.os[1][j] : G.on[1][j]);
            R a0 = R(0), a2 = R(0);
#pragma unroll
            for (int k = 0; k <= P; ++k) {
                const R f = row[SZ ? G.os[2][k] : G.on[2][k]];
                a0 += (SZ ? G.ws[2][k] : G.wn[2][k]) * f;
                a2 += (SZ ? ds[2][k] : dn[2][k]) * f;
            }
            const R wy = SY ? G.ws[1][j] : G.wn[1][j];
            s0 += wy * a0;
            s1 += (SY ? ds[1][j] : dn[1][j]) * a0;
            s2 += wy * a2;
        }
        const R wx = SX ? G.ws[0][i] : G.wn[0][i];
        v += wx * s0;
        g0 += (SX ? ds[0][i] : dn[0][i]) * s0;
        g1 += wx * s1;
        g2 += wx * s2;
    }
    grad[0] = g0;
    grad[1] = g1;
    grad[2] = g2;
    return v;
}

// Adjoint of the gather of one component: lamF(node) += w(node) lam.
template <int P, typename R, bool SX, bool SY, bool SZ>
__device__ __forceinline__ void scatter_adj(const GatherW<P, R>& G, R* lF, R lam) {
#pragma unroll
    for (int i = 0; i <= P; ++i) {
        const R wx = lam * (SX ? G.ws[0][i] : G.wn[0][i]);
        const int ox = SX ? G.os[0][i] : G.on[0][i];
#pragma unroll
        for (int j = 0; j <= P; ++j) {
            const R wxy = wx * (SY ? G.ws[1][j] : G.wn[1][j]);
            R* row = lF + ox + (SY ? G.os[1][j] : G.on[1][j]);
#pragma unroll
            for (int k = 0; k <= P; ++k)
                atomicAdd(row + (SZ ? G.os[2][k] : G.on[2][k]), wxy * (SZ ? G.ws[2][k] : G.wn[2][k]));
        }
    }
}

// A value the compiler may not trace back: what is computed from it is
// computed again here, not kept in registers since its first computation.
__device__ __forceinline__ float recompute(float v) {
    asm volatile("" : "+f"(v));
    return v;
}
__device__ __forceinline__ double recompute(double v) {
    asm volatile("" : "+d"(v));
    return v;
}

// The reverse step of one particle: the forward recomputation and the
// adjoints of its deposit, advance, Boris rotation and drive; lE, lB are left
// for the gather's scatter into the field adjoints.
template <int P, typename R>
__device__ __forceinline__ void adj_particle(const StepArgs<R>& A, const AdjArgs<R>& L, int p, const int cell[3],
                                             const R f0[3], const double xg0[3], const R u_old[3], R wq,
                                             R lE[3], R lB[3], double& lamA) {
    constexpr int NW = P + 2;
    const Geom& g = A.g;
    const int id = L.id[p];
    // ---- forward recomputation ----------------------------------
    R EB[6], grad[6][3];
    {
        GatherW<P, R> G;
        int fn[3], fs[3];
        gather_weights<P, R>(f0, G, fn, fs);
        offsets_global<P, R>(G, g, cell, fn, fs);
        R dn[3][P + 1], ds[3][P + 1];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ShapeD<P, R>::dweights(f0[a], dn[a]);
            staggered_dweights<P, R>(f0[a], ds[a]);
        }
        // staggering along x, y, z: Ex (s,n,n) Ey (n,s,n) Ez (n,n,s) Bx (n,s,s) By (s,n,s) Bz (s,s,n)
        EB[0] = gather_grad<P, R, true, false, false>(G, dn, ds, A.E[0], grad[0]);
        EB[1] = gather_grad<P, R, false, true, false>(G, dn, ds, A.E[1], grad[1]);
        EB[2] = gather_grad<P, R, false, false, true>(G, dn, ds, A.E[2], grad[2]);
        EB[3] = gather_grad<P, R, false, true, true>(G, dn, ds, A.B[0], grad[3]);
        EB[4] = gather_grad<P, R, true, false, true>(G, dn, ds, A.B[1], grad[4]);
        EB[5] = gather_grad<P, R, true, true, false>(G, dn, ds, A.B[2], grad[5]);
    }
    double cs = 0.0, sn = 0.0;  // cosine and sine of the drive's phase at the particle
    if (A.drive_amp != 0.0) {
        const double xp = sizeof(R) == 8 ? xg0[0] : (double(cell[0]) + double(f0[0])) * g.d[0];
        sincos(A.drive_k * xp - A.drive_k * L.t, &sn, &cs);
        EB[1] += R(A.drive_amp * cs);
    }
    R u[3] = {u_old[0], u_old[1], u_old[2]};
    Moved<R> mv;
    {
        R EBc[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) EBc[c] = EB[c];
        push_particle<P, R, false>(A, EBc, cell, f0, xg0, u, mv);  // the drive is in EB already
    }
    // ---- adjoints of the step's outputs --------------------------
    R lx1[3], lu[3], lx0[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lx1[a] = L.lamx[a][id];
        lu[a] = L.lamu[a][id];
    }
    // ---- Esirkepov deposit -------------------------------------------
    {
        EsirkAxis<P, R> ax[3];
        int node[3][NW];
        const int st[3] = {g.n[1] * g.n[2], g.n[2], 1};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ax[a].init(mv.f0[a], mv.f1[a]);
#pragma unroll
            for (int w = 0; w < NW; ++w) node[a][w] = wrap_once(cell[a] + ax[a].b + w, g.n[a]) * st[a];
        }
        R gS0[3][NW], gdS[3][NW];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int w = 0; w < NW; ++w) gS0[a][w] = gdS[a][w] = R(0);
        esirkepov_adj_component<P, R, 0>(ax, node, L.lamJ[0], A.jc[0] * wq, gS0, gdS);
        esirkepov_adj_component<P, R, 1>(ax, node, L.lamJ[1], A.jc[1] * wq, gS0, gdS);
        esirkepov_adj_component<P, R, 2>(ax, node, L.lamJ[2], A.jc[2] * wq, gS0, gdS);
        // dS = S1 - S0: dL/dS1 = gdS, dL/dS0 = gS0 - gdS; then the chain
        // through the shape derivatives on the same window
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            EsirkAxisD<P, R> dx;
            dx.init(mv.f0[a], mv.f1[a]);
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                lx0[a] += (gS0[a][w] - gdS[a][w]) * dx.D0[w];
                lx1[a] += gdS[a][w] * dx.D1[w];
            }
        }
    }
    // ---- advance: f1 = f0 + (dt/d) u / gamma ------------------------
    {
        const R ig = inv_sqrt(R(1) + mv.u[0] * mv.u[0] + mv.u[1] * mv.u[1] + mv.u[2] * mv.u[2]);
        R sdot = R(0);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lx0[a] += lx1[a];
            sdot += A.dtc[a] * lx1[a] * mv.u[a];
        }
        sdot *= ig * ig * ig;
#pragma unroll
        for (int a = 0; a < 3; ++a) lu[a] += A.dtc[a] * lx1[a] * ig - mv.u[a] * sdot;
    }
    // ---- Boris ----------------------------------------------------
    R luo[3];
    boris_adj<R>(A.kq, EB, EB + 3, u_old, lu, luo, lE, lB);
    // ---- drive ------------------------------------------------------
    if (A.drive_amp != 0.0) {
        lamA += double(lE[1]) * cs;
        lx0[0] += R(double(lE[1]) * A.drive_amp * (-A.drive_k) * sn * g.d[0]);
    }
    // ---- gather: its gradient along the particle's position ----------
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int c = 0; c < 3; ++c) lx0[a] += lE[c] * grad[c][a] + lB[c] * grad[3 + c][a];
        L.lamx[a][id] = lx0[a];
        L.lamu[a][id] = luo[a];
    }
}

// Sum over the block (kAdjBlock threads) of the drive adjoint.
__device__ __forceinline__ void add_lam_a(double lamA, double* out) {
    for (int o = 16; o; o >>= 1) lamA += __shfl_down_sync(0xffffffffu, lamA, o);
    __shared__ double red[kAdjBlock / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lamA;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kAdjBlock / 32; ++w) s += red[w];
        if (s != 0.0) atomicAdd(out, s);
    }
}

// One particle's gather adjoint into the six field adjoints at lF[0..5].
template <int P, typename R>
__device__ __forceinline__ void scatter_adj6(const GatherW<P, R>& G, R* const lF[6], const R lE[3], const R lB[3]) {
    scatter_adj<P, R, true, false, false>(G, lF[0], lE[0]);
    scatter_adj<P, R, false, true, false>(G, lF[1], lE[1]);
    scatter_adj<P, R, false, false, true>(G, lF[2], lE[2]);
    scatter_adj<P, R, false, true, true>(G, lF[3], lB[0]);
    scatter_adj<P, R, true, false, true>(G, lF[4], lB[1]);
    scatter_adj<P, R, true, true, false>(G, lF[5], lB[2]);
}

// The gather's scatter of one particle into the global field adjoints.
template <int P, typename R>
__device__ __forceinline__ void scatter_adj_global(const StepArgs<R>& A, const AdjArgs<R>& L, const int cell[3],
                                                   const R f0[3], const R lE[3], const R lB[3]) {
    GatherW<P, R> G;
    int fn[3], fs[3];
    gather_weights<P, R>(f0, G, fn, fs);
    offsets_global<P, R>(G, A.g, cell, fn, fs);
    R* const lF[6] = {L.lamE[0], L.lamE[1], L.lamE[2], L.lamB[0], L.lamB[1], L.lamB[2]};
    scatter_adj6<P, R>(G, lF, lE, lB);
}

// One particle per thread.  SCATTER: the gather's adjoint goes into the
// global field adjoints with atomics; otherwise lE, lB are left in L.lg for
// k_adj_scatter.
template <int P, typename R, bool SCATTER>
__global__ void __launch_bounds__(kAdjBlock) k_adj_particles(StepArgs<R> A, AdjArgs<R> L) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double lamA = 0.0;
    if (p < A.np) {
        int cell[3];
        R f0[3], u_old[3], wq;
        double xg0[3];
        load_particle<R>(A, int(p), cell, f0, xg0, u_old, wq);
        R lE[3], lB[3];
        adj_particle<P, R>(A, L, int(p), cell, f0, xg0, u_old, wq, lE, lB, lamA);
        if constexpr (SCATTER) {
            // the gather's weights are computed again
            const R f[3] = {recompute(f0[0]), recompute(f0[1]), recompute(f0[2])};
            scatter_adj_global<P, R>(A, L, cell, f, lE, lB);
        } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                L.lg[a][p] = lE[a];
                L.lg[3 + a][p] = lB[a];
            }
        }
    }
    add_lam_a(lamA, L.lamA);
}

// The gather's adjoint in FP32-mixed: lamF(node) += w(node) lam for the
// particles of one work item of the tile kernel (the slab they were in at the
// last sort, whose offsets these are), or of one of `parts` equal shares of
// them.  The slab's field adjoints are summed in shared memory and added to
// the global arrays once, because 6 (P+1)^3 global atomics a particle ran at
// the L2's rate for them (64^3, order 2, 4 a cell: 430 of the 790 us that a
// reverse step's particles took).
//
// The sums are exact fixed point, as the forward deposit's (FP32 atomics in
// shared memory are a load and compare-and-swap loop: with them the step took
// 1150 us).  The largest |lam| of the block's particles, found first, gives
// the scale: the power of two with scale |lam| < 2^30; weights lie in [0, 1].
// For up to 65535 particles a block the pair of int32 sums cannot overflow
// (red_fixed in the tile kernel's deposit has the argument).
//
// A state at most one step after its sort has its particles at most one cell
// outside their slab, so the box covers cells [-kLo, W + kHi) around it; any
// other particle, and a block whose lam is not finite, takes global atomics.
constexpr int kScatterThreads = 512;
constexpr int kScatterSmemMax = 220 << 10;

template <int P> struct AdjBox {
    static constexpr int kLo = P == 3 ? 3 : 2, kHi = P == 1 ? 2 : 3;
    int e[3], vol;
    __host__ __device__ explicit AdjBox(const Geom& g) {
        for (int a = 0; a < 3; ++a) e[a] = g.W[a] + kLo + kHi;
        vol = e[0] * e[1] * e[2];
    }
    size_t bytes() const { return 12 * size_t(vol) * sizeof(int); }
};

template <int P, bool SX, bool SY, bool SZ>
__device__ __forceinline__ void scatter_fixed(const GatherW<P, float>& G, int* lo, int* hi, float lam) {
#pragma unroll
    for (int i = 0; i <= P; ++i) {
        const float wx = lam * (SX ? G.ws[0][i] : G.wn[0][i]);
        const int ox = SX ? G.os[0][i] : G.on[0][i];
#pragma unroll
        for (int j = 0; j <= P; ++j) {
            const float wxy = wx * (SY ? G.ws[1][j] : G.wn[1][j]);
            const int oxy = ox + (SY ? G.os[1][j] : G.on[1][j]);
#pragma unroll
            for (int k = 0; k <= P; ++k) {
                const int o = oxy + (SZ ? G.os[2][k] : G.on[2][k]);
                const int x = __float2int_rn(wxy * (SZ ? G.ws[2][k] : G.wn[2][k]));
                atomicAdd(lo + o, x);
                atomicAdd(hi + o, x >> 15);
            }
        }
    }
}

template <int P>
__global__ void __launch_bounds__(kScatterThreads, 1)
    k_adj_scatter(StepArgs<float> A, AdjArgs<float> L, const int* __restrict__ offsets, int parts) {
    extern __shared__ __align__(16) int adj_sm[];
    __shared__ unsigned s_max;
    const Geom& g = A.g;
    const AdjBox<P> box(g);
    const int w = int(blockIdx.x) / parts, q = int(blockIdx.x) - w * parts;
    const int wbeg = offsets[int64_t(w) * g.cpw], wcnt = offsets[int64_t(w + 1) * g.cpw] - wbeg;
    const int beg = wbeg + int(int64_t(wcnt) * q / parts), end = wbeg + int(int64_t(wcnt) * (q + 1) / parts);
    if (beg >= end) return;
    if (threadIdx.x == 0) s_max = 0u;
    for (int e = threadIdx.x; e < 12 * box.vol; e += kScatterThreads) adj_sm[e] = 0;
    __syncthreads();
    unsigned m = 0u;  // |lam| as bits: ordered like the values, infinities and NaN above all
    for (int p = beg + int(threadIdx.x); p < end; p += kScatterThreads)
#pragma unroll
        for (int c = 0; c < 6; ++c) m = max(m, __float_as_uint(L.lg[c][p]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, m);
    __syncthreads();
    m = s_max;
    if (m == 0u) return;
    const bool fixed = m < 0x7f800000u && end - beg <= 65535;
    // |lam| < 2^(x + 1) with x the exponent of the largest: scale 2^(29 - x), at most 2^126
    const int x = max(int(m >> 23) - 127, -97);
    const float scale = __uint_as_float(unsigned(29 - x + 127) << 23), inv = __uint_as_float(unsigned(x - 29 + 127) << 23);
    int o[3];
    work_origin(g, w, o[0], o[1], o[2]);
    // runs of consecutive particles, so that a warp's lanes mostly add to different nodes
    const int run = (end - beg + kScatterThreads - 1) / kScatterThreads;
    const int p0 = beg + int(threadIdx.x) * run;
    for (int p = p0; p < min(p0 + run, end); ++p) {
        int cell[3], base[3];
        cell_of(g, A.key[p], cell[0], cell[1], cell[2]);
        const float f0[3] = {A.pa[0][p], A.pa[1][p], A.pa[2][p]};
        const float lE[3] = {L.lg[0][p], L.lg[1][p], L.lg[2][p]}, lB[3] = {L.lg[3][p], L.lg[4][p], L.lg[5][p]};
        bool in = fixed;
#pragma unroll
        for (int a = 0; a < 3; ++a) {  // cell relative to the slab, in the period nearest to it
            int d = cell[a] - o[a];
            if (d > g.W[a]) d -= g.n[a];
            else if (d < -1) d += g.n[a];
            in = in && d >= -1 && d <= g.W[a];
            base[a] = d + AdjBox<P>::kLo;
        }
        if (!in) {
            scatter_adj_global<P, float>(A, L, cell, f0, lE, lB);
            continue;
        }
        GatherW<P, float> G;
        int fn[3], fs[3];
        gather_weights<P, float>(f0, G, fn, fs);
        const int st[3] = {box.e[1] * box.e[2], box.e[2], 1};
        offsets_local<P, float>(G, base, st, fn, fs);
        int* const hi = adj_sm + 6 * box.vol;
        scatter_fixed<P, true, false, false>(G, adj_sm, hi, scale * lE[0]);
        scatter_fixed<P, false, true, false>(G, adj_sm + box.vol, hi + box.vol, scale * lE[1]);
        scatter_fixed<P, false, false, true>(G, adj_sm + 2 * box.vol, hi + 2 * box.vol, scale * lE[2]);
        scatter_fixed<P, false, true, true>(G, adj_sm + 3 * box.vol, hi + 3 * box.vol, scale * lB[0]);
        scatter_fixed<P, true, false, true>(G, adj_sm + 4 * box.vol, hi + 4 * box.vol, scale * lB[1]);
        scatter_fixed<P, true, true, false>(G, adj_sm + 5 * box.vol, hi + 5 * box.vol, scale * lB[2]);
    }
    __syncthreads();
    // a warp a z-row of the box: contiguous in the global arrays too
    const int rows = 6 * box.e[0] * box.e[1];
    for (int r = int(threadIdx.x) >> 5; r < rows; r += kScatterThreads / 32) {
        const int c = r / (box.e[0] * box.e[1]), ab = r - c * (box.e[0] * box.e[1]);
        const int a = ab / box.e[1], b = ab - a * box.e[1];
        const int64_t row = (int64_t(wrap_any(o[0] - AdjBox<P>::kLo + a, g.n[0])) * g.n[1] +
                             wrap_any(o[1] - AdjBox<P>::kLo + b, g.n[1])) * g.n[2];
        float* dst = (c < 3 ? L.lamE[c] : L.lamB[c - 3]) + row;
        for (int k = int(threadIdx.x) & 31; k < box.e[2]; k += 32) {
            const int lo = adj_sm[r * box.e[2] + k], hi = adj_sm[6 * box.vol + r * box.e[2] + k];
            if ((lo | hi) == 0) continue;
            const int low = int(unsigned(lo) - (unsigned(hi) << 15));
            atomicAdd(dst + wrap_any(o[2] - AdjBox<P>::kLo + k, g.n[2]),
                      __ll2float_rn((long long)hi * 32768 + low) * inv);
        }
    }
}

// lamE -= h curl' lamB (backward-difference curl, the transpose of the curl in
// the B update).
template <typename R>
__global__ void __launch_bounds__(kAdjBlock) k_adj_yee_e(R* lE0, R* lE1, R* lE2, const R* lB0, const R* lB1,
                                                         const R* lB2, int nx, int ny, int nz, R ix, R iy, R iz, R h) {
    const int64_t C = (int64_t)nx * ny * nz;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const int k = int(c % nz), j = int((c / nz) % ny), i = int(c / ((int64_t)ny * nz));
    const int64_t sx = (int64_t)ny * nz, sy = nz;
    const int64_t im = c - (i == 0 ? -(int64_t)(nx - 1) * sx : sx);
    const int64_t jm = c - (j == 0 ? -(int64_t)(ny - 1) * sy : sy);
    const int64_t km = c - (k == 0 ? -(int64_t)(nz - 1) : 1);
    const R bx = lB0[c], by = lB1[c], bz = lB2[c];
    lE0[c] -= h * ((bz - lB2[jm]) * iy - (by - lB1[km]) * iz);
    lE1[c] -= h * ((bx - lB0[km]) * iz - (bz - lB2[im]) * ix);
    lE2[c] -= h * ((by - lB1[im]) * ix - (bx - lB0[jm]) * iy);
}

// lamJ = -dt lamE; lamB += dt curl lamE (forward-difference curl, the
// transpose of the curl in the E update).
template <typename R>
__global__ void __launch_bounds__(kAdjBlock) k_adj_yee_b(const R* lE0, const R* lE1, const R* lE2, R* lB0, R* lB1,
                                                         R* lB2, R* lJ0, R* lJ1, R* lJ2, int nx, int ny, int nz, R ix,
                                                         R iy, R iz, R dt) {
    const int64_t C = (int64_t)nx * ny * nz;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const int k = int(c % nz), j = int((c / nz) % ny), i = int(c / ((int64_t)ny * nz));
    const int64_t sx = (int64_t)ny * nz, sy = nz;
    const int64_t ip = c + (i + 1 == nx ? -(int64_t)(nx - 1) * sx : sx);
    const int64_t jp = c + (j + 1 == ny ? -(int64_t)(ny - 1) * sy : sy);
    const int64_t kp = c + (k + 1 == nz ? -(int64_t)(nz - 1) : 1);
    const R ex = lE0[c], ey = lE1[c], ez = lE2[c];
    lJ0[c] = -dt * ex;
    lJ1[c] = -dt * ey;
    lJ2[c] = -dt * ez;
    lB0[c] += dt * ((lE2[jp] - ez) * iy - (lE1[kp] - ey) * iz);
    lB1[c] += dt * ((lE0[kp] - ex) * iz - (lE2[ip] - ez) * ix);
    lB2[c] += dt * ((lE1[ip] - ey) * ix - (lE0[jp] - ex) * iy);
}

// Reverse of one Yee step (B half, E full, B half):
//   lamE -= h C^T lamB;  lamJ = -dt lamE, lamB += dt C'^T lamE;  lamE -= h C^T lamB.
template <typename R> cudaError_t adj_yee_impl(pic_ctx* c, const AdjBuffers& b) {
    const int nx = c->g.n[0], ny = c->g.n[1], nz = c->g.n[2];
    const unsigned nb = unsigned((c->g.C + kAdjBlock - 1) / kAdjBlock);
    R* lE[3];
    R* lB[3];
    R* lJ[3];
    for (int a = 0; a < 3; ++a) {
        lE[a] = static_cast<R*>(b.lamE[a]);
        lB[a] = static_cast<R*>(b.lamB[a]);
        lJ[a] = static_cast<R*>(b.lamJ[a]);
    }
    const R ix = R(1.0 / c->g.d[0]), iy = R(1.0 / c->g.d[1]), iz = R(1.0 / c->g.d[2]);
    const R h = R(0.5 * c->dt), dt = R(c->dt);
    k_adj_yee_e<R><<<nb, kAdjBlock, 0, c->stream>>>(lE[0], lE[1], lE[2], lB[0], lB[1], lB[2], nx, ny, nz, ix, iy, iz, h);
    k_adj_yee_b<R><<<nb, kAdjBlock, 0, c->stream>>>(lE[0], lE[1], lE[2], lB[0], lB[1], lB[2], lJ[0], lJ[1], lJ[2], nx,
                                                    ny, nz, ix, iy, iz, dt);
    k_adj_yee_e<R><<<nb, kAdjBlock, 0, c->stream>>>(lE[0], lE[1], lE[2], lB[0], lB[1], lB[2], nx, ny, nz, ix, iy, iz, h);
    return cudaGetLastError();
}

cudaError_t launch_adj_yee(pic_ctx* c, const AdjBuffers& b) {
    return c->prec == PIC_FP64 ? adj_yee_impl<double>(c, b) : adj_yee_impl<float>(c, b);
}

template <typename R, int P> cudaError_t adj_particles_impl(pic_ctx* c, const AdjBuffers& b, const Snapshot& s,
                                                           double t) {
    StepArgs<R> A = make_args<R>(c);
    // the stored state replaces the live particles and fields
    for (int i = 0; i < 7; ++i) {
        A.pa[i] = static_cast<R*>(s.a[i]);
        A.spa[i] = A.pa[i];
    }
    A.key = s.key;
    A.skey = s.key;
    A.sid = A.did = s.id;
    for (int d = 0; d < 3; ++d) {
        A.E[d] = static_cast<const R*>(s.F[d]);
        A.B[d] = static_cast<const R*>(s.F[3 + d]);
    }
    AdjArgs<R> L;
    for (int a = 0; a < 3; ++a) {
        L.lamx[a] = static_cast<R*>(b.lamx[a]);
        L.lamu[a] = static_cast<R*>(b.lamu[a]);
        L.lamE[a] = static_cast<R*>(b.lamE[a]);
        L.lamB[a] = static_cast<R*>(b.lamB[a]);
        L.lamJ[a] = static_cast<const R*>(b.lamJ[a]);
    }
    // between the two kernels of FP32-mixed: the particle buffer that holds no
    // state during the reverse sweep (every state is restored whole from its
    // copy into the other one)
    for (int i = 0; i < 6; ++i) L.lg[i] = static_cast<R*>(c->P[1 - c->cur].a[i]);
    L.id = s.id;
    L.lamA = b.lamA;
    L.t = t;
    if (c->np == 0) return cudaSuccess;
    const unsigned nb = unsigned((c->np + kAdjBlock - 1) / kAdjBlock);
    // FP64 is bound by its FP64 units, not by the atomics, and a state further
    // from its sort leaves particles outside their slab's box: global atomics
    if constexpr (sizeof(R) == 4) {
        const AdjBox<P> box(c->g);
        // shares of two thousand particles or more (64^3, 4 a cell: the sweep
        // takes 11.3 ms with whole slabs of 2048, 11.8 with halves: every block
        // clears and flushes the whole box)
        const int64_t per = c->np / (c->g.nwork > 0 ? c->g.nwork : 1) / 2048;
        const int parts = int(per < 1 ? 1 : per > 64 ? 64 : per);
        if (s.since_sort <= 1 && box.bytes() <= size_t(kScatterSmemMax) && c->g.nwork * parts < (int64_t(1) << 31)) {
            const cudaError_t e = cudaFuncSetAttribute(k_adj_scatter<P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       int(box.bytes()));
            if (e != cudaSuccess) return e;
            k_adj_particles<P, R, false><<<nb, kAdjBlock, 0, c->stream>>>(A, L);
            k_adj_scatter<P><<<unsigned(c->g.nwork * parts), kScatterThreads, box.bytes(), c->stream>>>(
                A, L, s.offsets, parts);
            return cudaGetLastError();
        }
    }
    k_adj_particles<P, R, true><<<nb, kAdjBlock, 0, c->stream>>>(A, L);
    return cudaGetLastError();
}

cudaError_t launch_adj_particles(pic_ctx* c, const AdjBuffers& b, const Snapshot& s, double t) {
    if (c->prec == PIC_FP64) {
        switch (c->order) {
        case 1: return adj_particles_impl<double, 1>(c, b, s, t);
        case 2: return adj_particles_impl<double, 2>(c, b, s, t);
        default: return adj_particles_impl<double, 3>(c, b, s, t);
        }
    }
    switch (c->order) {
    case 1: return adj_particles_impl<float, 1>(c, b, s, t);
    case 2: return adj_particles_impl<float, 2>(c, b, s, t);
    default: return adj_particles_impl<float, 3>(c, b, s, t);
    }
}

template <typename S, typename D> __global__ void k_copy_convert(const S* src, D* dst, int64_t n, D scale) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = D(src[i]) * scale;
}

// lamE = E dV, lamB = B dV (adjoint of L = 1/2 sum |E|^2 + |B|^2 dV); zero the rest.
cudaError_t launch_adj_init(pic_ctx* c, const AdjBuffers& b) {
    const unsigned nb = unsigned((c->g.C + kAdjBlock - 1) / kAdjBlock);
    const double dV = c->g.d[0] * c->g.d[1] * c->g.d[2];
    for (int a = 0; a < 3; ++a) {
        if (c->prec == PIC_FP64) {
            k_copy_convert<double, double><<<nb, kAdjBlock, 0, c->stream>>>(
                static_cast<const double*>(c->F[a]), static_cast<double*>(b.lamE[a]), c->g.C, dV);
            k_copy_convert<double, double><<<nb, kAdjBlock, 0, c->stream>>>(
                static_cast<const double*>(c->F[3 + a]), static_cast<double*>(b.lamB[a]), c->g.C, dV);
        } else {
            k_copy_convert<float, float><<<nb, kAdjBlock, 0, c->stream>>>(
                static_cast<const float*>(c->F[a]), static_cast<float*>(b.lamE[a]), c->g.C, float(dV));
            k_copy_convert<float, float><<<nb, kAdjBlock, 0, c->stream>>>(
                static_cast<const float*>(c->F[3 + a]), static_cast<float*>(b.lamB[a]), c->g.C, float(dV));
        }
    }
    return cudaGetLastError();
}

// dL/du (by id, component-major, FP64) from the momentum adjoint.
cudaError_t launch_adj_output(pic_ctx* c, const AdjBuffers& b, double* d_out) {
    if (c->np == 0) return cudaSuccess;
    const unsigned nb = unsigned((c->np + kAdjBlock - 1) / kAdjBlock);
    for (int a = 0; a < 3; ++a) {
        if (c->prec == PIC_FP64)
            k_copy_convert<double, double><<<nb, kAdjBlock, 0, c->stream>>>(static_cast<const double*>(b.lamu[a]),
                                                                            d_out + a * c->np, c->np, 1.0);
        else
            k_copy_convert<float, double><<<nb, kAdjBlock, 0, c->stream>>>(static_cast<const float*>(b.lamu[a]),
                                                                           d_out + a * c->np, c->np, 1.0);
    }
    return cudaGetLastError();
}

}  // namespace pic
