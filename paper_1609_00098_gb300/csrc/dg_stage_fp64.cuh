// dg_stage_fp64.cuh -- FP64 element kernels of the DG stage (templated on the
// number of LGL nodes per axis NP):
//   k_stage_fp64  : volume term + lifted surface term of eq:411 and the SSP-RK3
//                   stage combination (Sec. 3.4);
//   k_summaries   : the limiter summaries;
//   k_limit       : the MinModN / MinMod decision and linear replacement (Sec. 3.3).
// This file is compiled without floating-point contraction and every sum runs in a
// fixed order, so that the FP64 path reproduces a plain sequential evaluation of the
// same formulas operation for operation.
#pragma once

#include "dg_internal.h"
#include "dg_intfp64.cuh"
#include "dg_physics.cuh"

namespace dg {

// Launch shape of k_stage_fp64: elements per CTA and threads, so that the 15 n^2 lines
// of an element (the longest phase) fill the threads in whole rounds.
template <int NP>
struct StageShape64 {
    static constexpr int NN = NP * NP * NP, N2 = NP * NP;
    static constexpr int EPB = NP == 2 ? 4 : NP == 3 ? 2 : 1;
    static constexpr int THREADS = NP == 2 || NP == 4 ? 256 : NP == 3 || NP == 6 ? 288 : NP == 8 ? 512 : 384;
    static constexpr size_t SMEM = sizeof(double) * (15 * NN + 30 * N2) * EPB;
    // CTAs that must fit on an SM, which caps the registers (32 for n = 2, 3, 40 for n = 5,
    // 56 for n = 6, 64 for n = 4, 80 for n = 7, with up to 320, 84, 4, 0 and 104 bytes of
    // spills): more warps to hide the FP64 latency.  Step without a limiter at about 0.5 M
    // nodes (KH, LLF), us, unbounded and so: n = 2 801, 646; n = 3 1000, 883; n = 4 1026,
    // 979; n = 5 1080, 1045; n = 7 (one CTA per SM before) 1562, 1217.  n = 6 had four CTAs
    // anyway, but spills less (24^3, limiter: 4225, 4106).  n = 8 keeps its own choice (64
    // registers, two CTAs: 1129; with 320 threads 1130 to 1224).
    static constexpr int MIN_CTAS = NP == 2 ? 7 : NP == 3 ? 6 : NP == 7 ? 2 : NP <= 6 ? 4 : 0;
};

// The rare cases of the two integer-ALU phases, in FP64 instructions.
static __device__ __noinline__ void node_fluxes_native(const double *u, const double *P, double *dst, int nn)
{
    ifp::Native ar;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        double f[5];
        flux_axis(ar, u, P, ax, f);
        for (int v = 0; v < 5; ++v) dst[(ax * 5 + v) * nn] = f[v];
    }
}

static __device__ __noinline__ double scaled_sum_native(const double *g, const double *s, int st)
{
    return (g[0] * s[0] + g[1] * s[st]) + g[2] * s[2 * st];
}

template <int NP>
static __device__ __noinline__ void line_native(const double *D, double *F, int st)
{
    double f[NP];
#pragma unroll
    for (int l = 0; l < NP; ++l) f[l] = F[l * st];
    for (int i = 0; i < NP; ++i) {
        double s = D[i * NP] * f[0];
#pragma unroll
        for (int l = 1; l < NP; ++l) s = s + D[i * NP + l] * f[l];
        F[i * st] = s;
    }
}

// One stage for EPB elements per CTA, in four phases:
//   nodes   the fluxes F^a_v of the element (eq:411) into shared memory;
//   faces   the stored numerical flux minus the element's own, times the lift factor,
//           per face point and variable;
//   lines   one thread per (axis, variable, line of n nodes): the n products and sums
//           of eq:405 for the line's n nodes, in place;
//   nodes   the three axes' sums combined, the lifts added (x, y, z in turn), and the
//           stage update.
// Every sum keeps the order of a sequential evaluation node by node (products and sums
// rounded separately), so the results are its bits.
//
// Bound by the FP64 pipe and the integer ALU in about equal parts: the products of the
// fluxes, the contraction and its scaling run on the integer ALU, with the entries of D prepared
// by the host and each line's flux values prepared once for n products, which leaves
// the FP64 pipe n - 1 additions per node, axis and variable; the lift and the update
// keep theirs on the FP64 pipe, which has room for them.  With products and sums
// both on it and one thread per node, the contraction ran at half the rate (0.25e12
// against 0.50e12 product-sum pairs/s).  Lines also give 15 n^2 threads' work where
// nodes give n^3, which is what a mesh with fewer elements than SMs needs.  24^3, n =
// 6: 5430 us per launch with the faces and summaries inside, 900 now (FP64 pipe 81 %,
// integer ALU 52 %); 16^3, n = 5: 1145 and 146; 4^3, n = 4: 33 and 10.7.
template <int NP, bool PRIMS>
__global__ void __launch_bounds__(StageShape64<NP>::THREADS, StageShape64<NP>::MIN_CTAS)
    k_stage_fp64(const __grid_constant__ StageArgs a)
{
    pdl_wait();
    using SH = StageShape64<NP>;
    constexpr int NN = SH::NN, N2 = SH::N2, EPB = SH::EPB;
    extern __shared__ double smem_stage[];
    double *sF = smem_stage;                 // [EPB][3][5][NN] fluxes, then the lines' sums
    double *sL = smem_stage + EPB * 15 * NN;  // [EPB][6][5][N2] lifted face terms
    __shared__ long long sFace[EPB][6];       // index of the face at side s of axis a (2 a + s)

    const int t = threadIdx.x;
    const long long e0 = (long long)blockIdx.x * EPB;
    const int ne = EPB == 1 ? 1 : a.E - e0 < EPB ? (int)(a.E - e0) : EPB;
    if (t < 6 * ne) {
        const int ax = (t % 6) >> 1;
        const long long e = e0 + t / 6;
        const long long en = (t & 1) ? elem_neighbour_bc(e, a.K, ax, 1, a.gh) : e;
        sFace[t / 6][t % 6] = en >= 0 ? ax * a.E + en : 3 * a.E + (-1 - en);
    }
    for (int r = t; r < ne * NN; r += SH::THREADS) {
        const int el = EPB == 1 ? 0 : r / NN, q = r - el * NN;
        double u[5], P[4];
#pragma unroll
        for (int v = 0; v < 5; ++v) u[v] = a.Us[((e0 + el) * 5 + v) * NN + q];
#pragma unroll
        for (int c = 0; c < 4; ++c) P[c] = a.P[((e0 + el) * 4 + c) * NN + q];
        ifp::Fast ar;
        double *const dst = sF + el * 15 * NN + q;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            double f[5];
            flux_axis(ar, u, P, ax, f);
#pragma unroll
            for (int v = 0; v < 5; ++v) dst[(ax * 5 + v) * NN] = f[v];
        }
        if (!ar.ok) {
            const double w[5] = {u[0], u[1], u[2], u[3], u[4]}, p[4] = {P[0], P[1], P[2], P[3]};
            node_fluxes_native(w, p, dst, NN);
        }
    }
    __syncthreads();

    // lifted face terms: (2/dx_a)(F* - F)/w at the face's end of the axis
    for (int r = t; r < ne * 30 * N2; r += SH::THREADS) {
        const int el = EPB == 1 ? 0 : r / (30 * N2), rr = r - el * 30 * N2;
        const int as = rr / (5 * N2), vr = rr - as * 5 * N2, v = vr / N2, p = vr - v * N2;
        const int ax = as >> 1;
        const int sa = ax == 0 ? 1 : ax == 1 ? NP : N2, sb = ax == 0 ? NP : ax == 1 ? N2 : 1;
        const int sc = ax == 0 ? N2 : ax == 1 ? 1 : NP;
        const int q = ((as & 1) ? NP - 1 : 0) * sa + (p % NP) * sb + (p / NP) * sc;
        const double lift = (as & 1) ? (ax == 0 ? a.liftN[0] : ax == 1 ? a.liftN[1] : a.liftN[2])
                                     : (ax == 0 ? a.lift0[0] : ax == 1 ? a.lift0[1] : a.lift0[2]);
        sL[r] = lift * (a.Fs[sFace[el][as] * 5 * N2 + vr] - sF[(el * 15 + ax * 5 + v) * NN + q]);
    }
    __syncthreads();

    // volume term: sum_l D_il F_l along every line, in place
    for (int r = t; r < ne * 15 * N2; r += SH::THREADS) {
        const int av = r / N2, c = r - av * N2;  // av = (el, axis, variable)
        const int ax = (av % 15) / 5;
        const int st = ax == 0 ? 1 : ax == 1 ? NP : N2;
        double *F = sF + av * NN + (ax == 0 ? NP * c : ax == 1 ? c % NP + N2 * (c / NP) : c);
        double f[NP], s[NP];
        bool ok = true;
#pragma unroll
        for (int l = 0; l < NP; ++l) {
            f[l] = F[l * st];
            ok &= ifp::factor_ok(f[l]);
        }
        if (ok) {
#pragma unroll
            for (int l = 0; l < NP; ++l) {
                const ifp::Factor fl = ifp::factor(f[l]);
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const double p = ifp::mul_unsigned_zero(fl, a.DF[i * NP + l]);
                    s[i] = l == 0 ? p : s[i] + p;
                }
            }
        } else {  // values out of the products' range, infinities, NaN
            line_native<NP>(a.T.D, F, st);
            continue;
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) F[i * st] = s[i];
    }
    __syncthreads();

    const double dt = a.dt_ptr ? *a.dt_ptr : a.dt;
    for (int r = t; r < ne * NN; r += SH::THREADS) {
        const int el = EPB == 1 ? 0 : r / NN, q = r - el * NN;
        const int i = q % NP, j = (q / NP) % NP, k = q / N2;
        const double *Fe = sF + el * 15 * NN + q, *Le = sL + el * 30 * N2;
        // offset of the node's lifted terms on each axis, if it lies on a face
        const bool fx = i == 0 || i == NP - 1, fy = j == 0 || j == NP - 1, fz = k == 0 || k == NP - 1;
        const int ox = (i == 0 ? 0 : 5 * N2) + j + NP * k, oy = (j == 0 ? 10 * N2 : 15 * N2) + k + NP * i;
        const int oz = (k == 0 ? 20 * N2 : 25 * N2) + i + NP * j;
        double R[5];
        ifp::Fast ar;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            double acc = ar.mul(a.g[0], Fe[v * NN]);
            acc = acc + ar.mul(a.g[1], Fe[(5 + v) * NN]);
            acc = acc + ar.mul(a.g[2], Fe[(10 + v) * NN]);
            R[v] = -acc;
        }
        if (!ar.ok)
            for (int v = 0; v < 5; ++v) R[v] = -scaled_sum_native(a.g, Fe + v * NN, 5 * NN);
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            if (fx) R[v] = R[v] + (i == 0 ? Le[ox + v * N2] : -Le[ox + v * N2]);
            if (fy) R[v] = R[v] + (j == 0 ? Le[oy + v * N2] : -Le[oy + v * N2]);
            if (fz) R[v] = R[v] + (k == 0 ? Le[oz + v * N2] : -Le[oz + v * N2]);
        }
        const long long ix = (e0 + el) * 5 * NN + q;
        if (a.mode != 0) {
            if (a.first) {
#pragma unroll
                for (int v = 0; v < 5; ++v) R[v] = a.Us[ix + v * NN] + dt * R[v];
            } else {
#pragma unroll
                for (int v = 0; v < 5; ++v)
                    R[v] = a.ca * a.Un[ix + v * NN] + a.cb * (a.Us[ix + v * NN] + dt * R[v]);
            }
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) a.out[ix + v * NN] = R[v];
        // Newtonian runs without a limiter: the next stage's primitives, from the state in
        // registers (one launch less in stages 2 and 3: 48.0 -> 42.6 us per step at 4^3,
        // n = 4).  An element's primitives are read in this launch by its own CTA only,
        // before the barriers above.  (A variant of its own: as a run-time choice it took
        // 2 % from the other runs at n = 6, by its registers.)
        if (PRIMS) {
            double P[4];
            ne_primitives(a.gamma, R, P);
#pragma unroll
            for (int c = 0; c < 4; ++c) a.Pout[((e0 + el) * 4 + c) * NN + q] = P[c];
        }
    }
}

// Sum of the weighted values of an n x n' set of nodes in FP64 instructions (the rare
// case of a value out of the integer products' range).
static __device__ __noinline__ double weighted_sum_native(const double *w, const double *x, int n0, int s0, int n1, int s1)
{
    double s = 0.0;
    for (int t1 = 0; t1 < n1; ++t1)
        for (int t0 = 0; t0 < n0; ++t0) s = s + w[t0 + n0 * t1] * x[t0 * s0 + t1 * s1];
    return s;
}

// Whether u is an unphysical SR state.
__device__ __forceinline__ bool node_unphysical(const double u[5])
{
    ifp::Fast ar;
    const double s2 = ar.mul(u[1], u[1]) + ar.mul(u[2], u[2]) + ar.mul(u[3], u[3]);
    const double tt = ar.mul(u[4], u[4] + 2.0 * u[0]);
    bool bad = !ar.positive(u[0]) | !ar.positive(u[4]) | !ar.positive(tt) | !(ifp::order_key(s2) < ifp::order_key(tt));
    if (!ar.ok) {
        const double w[5] = {u[0], u[1], u[2], u[3], u[4]};
        bad = sr_unphysical_native(w);
    }
    return bad;
}

// Limiter summaries S[e][v][10] of a.G consecutive elements per CTA: [0] the cell mean
// (LGL quadrature / 8), [1+2a], [2+2a] the lower / upper face means along a, [7+a] the
// Legendre P1 coefficient along a of the mean over the other axes.  Every sum runs
// sequentially over its nodes in a fixed order, so the parallelism is over sums: warp
// 0 takes the cell means (n^3 terms each, one lane per element and variable), the other
// warps the 15 n plane means per element (n^2 terms each), of which the face means are
// the first and last and the P1 coefficients the weighted sums.
//
// FP64-pipe bound.  The terms' products run on the integer ALU, and the weight products
// are formed once per CTA.  Several elements share a CTA because a warp-wide FP64
// instruction costs the same with 5 or 30 lanes active; one element per CTA, every
// summary summing its own nodes, took two thirds of the FP64 stage's time.  24^3, n = 6:
// 209 us (FP64 pipe 62 %); 16^3, n = 5: 44 us.
template <int NP>
struct SumShape {
    static constexpr int NN = NP * NP * NP;
    static constexpr int G = NP <= 5 ? 6 : NP == 6 ? 4 : 3;  // most elements per CTA (5 G lanes of warp 0)
    // (n = 7, 8: three elements fill the shared memory of a CTA, so more threads each: 1609
    // -> 1573 us per step at n = 7 against 128; n = 5: 1 % against 192; n = 6 with 160: 2 %
    // more for the kernel at 24^3)
    static constexpr int THREADS = NP <= 4 ? 192 : NP == 6 ? 128 : 256;
    // per element: U[5][NN] and plane means [15 NP]; per CTA: weight products
    static constexpr size_t ELEM = sizeof(double) * (5 * NN + 15 * NP);
    static constexpr size_t TAB = (sizeof(double) + sizeof(ifp::Factor)) * (NN + NP * NP) + 8;
    __host__ __device__ static size_t smem(int g) { return ELEM * g + TAB; }
};

template <int NP>
__global__ void __launch_bounds__(SumShape<NP>::THREADS) k_summaries(const __grid_constant__ SummaryArgs a)
{
    pdl_wait();
    constexpr int NN = NP * NP * NP, N2 = NP * NP;
    extern __shared__ double smem_sum[];
    const int G = a.G, t = threadIdx.x;
    const long long e0 = (long long)blockIdx.x * G;
    const int ne = a.E - e0 < G ? (int)(a.E - e0) : G;
    double *sU = smem_sum;                 // [G][5][NN]
    double *sQ = sU + (size_t)G * 5 * NN;  // [G][3 axes][NP][5]
    double *sW3 = sQ + (size_t)G * 15 * NP, *sW2 = sW3 + NN;
    ifp::Factor *sF3 = reinterpret_cast<ifp::Factor *>(sW2 + N2), *sF2 = sF3 + NN;
    __shared__ double sMean[SumShape<NP>::G][5];
    __shared__ int sBad[SumShape<NP>::G];

    const double *Ug = a.U + e0 * 5 * NN;
    for (int i = t; i < ne * 5 * NN; i += blockDim.x) sU[i] = Ug[i];
    if (t < SumShape<NP>::G) sBad[t] = 0;
    for (int q = t; q < NN; q += blockDim.x) {
        const double w2 = a.T.w[q % NP] * a.T.w[(q / NP) % NP];
        const double w3 = w2 * a.T.w[q / N2];
        sW3[q] = w3;
        sF3[q] = ifp::factor(w3);
        if (q < N2) {
            sW2[q] = w2;
            sF2[q] = ifp::factor(w2);
        }
    }
    __syncthreads();

    if (a.unphys)
        for (int i = t; i < ne * NN; i += blockDim.x) {
            const int el = i / NN;
            const double *p = sU + (size_t)el * 5 * NN + (i - el * NN);
            const double u[5] = {p[0], p[NN], p[2 * NN], p[3 * NN], p[4 * NN]};
            if (node_unphysical(u)) sBad[el] = 1;
        }
    if (t < 32) {
        for (int r = t; r < ne * 5; r += 32) {
            const double *Uv = sU + (size_t)r * NN;
            double s = 0.0;
            bool ok = true;
#pragma unroll 4
            for (int q = 0; q < NN; ++q) {
                const double x = Uv[q];
                ok = ok & ifp::factor_ok(x);
                s = s + ifp::mul_unsigned_zero(ifp::factor(x), sF3[q]);
            }
            if (!ok) s = weighted_sum_native(sW3, Uv, NN, 1, 1, 0);
            sMean[r / 5][r % 5] = s * 0.125;
        }
    } else {
        for (int r = t - 32; r < ne * 15 * NP; r += SumShape<NP>::THREADS - 32) {
            const int v = r % 5, ia = (r / 5) % NP, ax = (r / (5 * NP)) % 3, el = r / (15 * NP);
            // nodes with index ia along ax; t0 runs along the next axis, t1 along the one after
            const int sa = ax == 0 ? 1 : ax == 1 ? NP : N2, sb = ax == 0 ? NP : ax == 1 ? N2 : 1;
            const int sc = ax == 0 ? N2 : ax == 1 ? 1 : NP;
            const double *Uv = sU + (size_t)(el * 5 + v) * NN + ia * sa;
            double s = 0.0;
            bool ok = true;
            for (int t1 = 0; t1 < NP; ++t1)
#pragma unroll
                for (int t0 = 0; t0 < NP; ++t0) {
                    const double x = Uv[t0 * sb + t1 * sc];
                    ok = ok & ifp::factor_ok(x);
                    s = s + ifp::mul_unsigned_zero(ifp::factor(x), sF2[t0 + NP * t1]);
                }
            if (!ok) s = weighted_sum_native(sW2, Uv, NP, sb, NP, sc);
            sQ[((el * 3 + ax) * NP + ia) * 5 + v] = s * 0.25;
        }
    }
    __syncthreads();
    for (int r = t; r < ne * 50; r += blockDim.x) {
        // kind-major: neighbouring lanes on one kind
        const int el = r % ne, v = (r / ne) % 5, kind = r / (5 * ne);
        double val;
        if (kind == 0) {
            val = sMean[el][v];
        } else if (kind <= 6) {
            const int ax = (kind - 1) / 2, ia = ((kind - 1) % 2) ? NP - 1 : 0;
            val = sQ[((el * 3 + ax) * NP + ia) * 5 + v];
        } else {
            const double *Q = sQ + (el * 3 + kind - 7) * NP * 5 + v;
            val = 0.0;
#pragma unroll
            for (int ia = 0; ia < NP; ++ia) val = val + a.T.row1[ia] * Q[ia * 5];
        }
        a.S[(e0 + el) * 50 + v * 10 + kind] = val;
    }
    if (t < ne && a.unphys) a.unphys[e0 + t] = sBad[t] ? 1 : 0;
}

// Two elements per warp: lane 16 h + 3 v + ax decides variable v along axis ax of
// element 2 w + h.  MinModN tests the six face conditions of Sec. 3.3.2 (tolerance
// 1e-8, M = 0); MinMod always limits; SR elements with an unphysical node limit every
// variable.  A limited variable becomes U0 + sum_a m_B(U_a, dU+/(dx/beta),
// dU-/(dx/beta); M)(x_a - x_a0) (eq:MinModSol) at every node, the terms added one
// after another.  The terms depend on one node index each and the first two partial
// sums on two, so they are formed once per (variable, index) and (variable, plane
// point): one FP64 addition per node is left of nine operations.  24^3, n = 6: 466 us
// per launch before, 54 now; 16^3, n = 5: 105 and 14.
template <int NP>
__global__ void __launch_bounds__(128) k_limit(const __grid_constant__ LimitArgs a)
{
    pdl_wait();
    constexpr int NN = NP * NP * NP, N2 = NP * NP;
    __shared__ double sSl[4][32], sM0[4][32];  // per warp: slopes and means by lane
    __shared__ double sP[4][15 * NP];          // [v][ax][i] slope terms
    __shared__ double sAB[4][5 * N2];          // [v][j][i] mean + x term + y term
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, half = lane >> 4, h = lane & 15;
    const long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
    const bool live = e < a.E;
    int flag = 0;
    double slope = 0.0, U0 = 0.0;
    if (live && h < 15) {
        const int v = h / 3, ax = h % 3;
        const double *Se = a.S + (e * 5 + v) * 10;
        U0 = Se[0];
        const double dm = U0 - a.S[(elem_neighbour(e, a.K, ax, -1) * 5 + v) * 10];
        const double dp = a.S[(elem_neighbour(e, a.K, ax, +1) * 5 + v) * 10] - U0;
        flag = (a.limiter == 2);
        if (a.limiter == 1) {
            const double ulo = Se[1 + 2 * ax], uhi = Se[2 + 2 * ax];
            const double vl = U0 - minmod3_bits(U0 - ulo, dm, dp);
            const double vr = U0 + minmod3_bits(uhi - U0, dm, dp);
            if (abs_gt(vl - ulo, 1e-8) || abs_gt(vr - uhi, 1e-8)) flag = 1;
        }
        const double s1 = ifp::div(2.0 * Se[7 + ax], a.dx[ax]);
        slope = abs_le(s1, a.tvb[ax]) ? s1 : minmod3_bits(s1, ifp::div(dp, a.h[ax]), ifp::div(dm, a.h[ax]));
    }
    const unsigned fb = __ballot_sync(0xffffffffu, flag) >> (16 * half);
    unsigned mask = 0;
#pragma unroll
    for (int v = 0; v < 5; ++v)
        if ((fb >> (3 * v)) & 7u) mask |= 1u << v;
    if (live && a.unphys && a.unphys[e]) mask = 0x1fu;
    if (live && h == 0 && a.troubled) a.troubled[e] = (unsigned char)mask;
    sSl[wl][lane] = slope;
    sM0[wl][lane] = U0;
    for (int hh = 0; hh < 2; ++hh) {
        const unsigned mk = __shfl_sync(0xffffffffu, mask, 16 * hh);
        const long long eh = __shfl_sync(0xffffffffu, e, 16 * hh);
        if (!mk) continue;
        __syncwarp();
        for (int r = lane; r < 15 * NP; r += 32) {
            const int va = r / NP;  // 3 v + ax
            sP[wl][r] = ifp::mul(sSl[wl][16 * hh + va], a.hx[va % 3][r % NP]);
        }
        __syncwarp();
        for (int r = lane; r < 5 * N2; r += 32) {
            const int v = r / N2, i = r % NP, j = (r / NP) % NP;
            sAB[wl][r] = (sM0[wl][16 * hh + 3 * v] + sP[wl][(3 * v) * NP + i]) + sP[wl][(3 * v + 1) * NP + j];
        }
        __syncwarp();
        for (int v = 0; v < 5; ++v) {
            if (!(mk & (1u << v))) continue;
            double *Uv = a.U + (eh * 5 + v) * NN;
            for (int q = lane; q < NN; q += 32) Uv[q] = sAB[wl][v * N2 + q % N2] + sP[wl][(3 * v + 2) * NP + q / N2];
        }
    }
}

// Dispatch helpers instantiated once per NP in dg_stage_fp64_n*.cu.
template <int NP>
cudaError_t launch_stage_np(const StageArgs &args, cudaStream_t s)
{
    using SH = StageShape64<NP>;
    StageArgs a = args;
    for (int i = 0; i < NP * NP; ++i) a.DF[i] = ifp::factor(a.T.D[i]);
    void (*const kern)(const StageArgs) = a.Pout ? k_stage_fp64<NP, true> : k_stage_fp64<NP, false>;
    if (SH::SMEM > 48 * 1024) {
        const cudaError_t err =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::SMEM);
        if (err != cudaSuccess) return err;
    }
    return launch_pdl(kern, (unsigned)((a.E + SH::EPB - 1) / SH::EPB), SH::THREADS, SH::SMEM, s, a);
}

template <int NP>
cudaError_t launch_summaries_np(const SummaryArgs &args, cudaStream_t s)
{
    SummaryArgs a = args;
    // few elements: fewer per CTA, so that every SM gets some
    const long long per = (a.E + kNumSMs - 1) / kNumSMs;
    a.G = per < 1 ? 1 : per < SumShape<NP>::G ? (int)per : SumShape<NP>::G;
    const size_t smem = SumShape<NP>::smem(a.G), most = SumShape<NP>::smem(SumShape<NP>::G);
    if (most > 48 * 1024) {
        // the limit is the kernel's, for every thread of the process: always the largest, or a
        // launch of another mesh would find it lowered
        const cudaError_t err =
            cudaFuncSetAttribute(k_summaries<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (err != cudaSuccess) return err;
    }
    return launch_pdl(k_summaries<NP>, (unsigned)((a.E + a.G - 1) / a.G), SumShape<NP>::THREADS, smem, s, a);
}

template <int NP>
cudaError_t launch_limit_np(const LimitArgs &a, cudaStream_t s)
{
    return launch_pdl(k_limit<NP>, (unsigned)((a.E + 7) / 8), 128, 0, s, a);  // 8 elements per CTA
}

}  // namespace dg

#define DG_INSTANTIATE_STAGE(NP)                                                                      \
    namespace dg {                                                                                    \
    cudaError_t launch_stage_fp64_n##NP(const StageArgs &a, cudaStream_t s)                            \
    {                                                                                                 \
        return launch_stage_np<NP>(a, s);                                                             \
    }                                                                                                 \
    cudaError_t launch_summaries_n##NP(const SummaryArgs &a, cudaStream_t s)                          \
    {                                                                                                 \
        return launch_summaries_np<NP>(a, s);                                                         \
    }                                                                                                 \
    cudaError_t launch_limit_n##NP(const LimitArgs &a, cudaStream_t s) { return launch_limit_np<NP>(a, s); } \
    }
