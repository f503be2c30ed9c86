// dg_physics.cuh -- point-wise physics of the two conservation laws, FP64,
// device side (Sec. 2.1.1 Newtonian Euler, Sec. 2.1.2 SR hydro in flat space,
// Sec. 3.2 numerical fluxes, Sec. 2.1.4 conserved-variable fix).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "dg_intfp64.cuh"

namespace dg {

// Status bits of the per-mesh device status word.
enum : unsigned { ERRBIT_C2P = 1u, ERRBIT_UNPHYSICAL = 2u, ERRBIT_TIMEOUT = 4u };

// ---------------------------------------------------------------------------
// Newtonian Euler: U = [rho, rho v_i, E], E = rho eps + rho v^2/2, p = (g-1) rho eps.
template <class A>
__device__ __forceinline__ void ne_primitives(A &ar, double g, const double u[5], double P[4])
{
    const double inv = ar.div(1.0, u[0]);
    P[0] = ar.mul(u[1], inv);
    P[1] = ar.mul(u[2], inv);
    P[2] = ar.mul(u[3], inv);
    P[3] = ar.mul(g - 1.0, u[4] - 0.5 * (ar.mul(u[1], P[0]) + ar.mul(u[2], P[1]) + ar.mul(u[3], P[2])));
}

static __device__ __noinline__ void ne_primitives_native(double g, const double *u, double *P)
{
    ifp::Native ar;
    ne_primitives(ar, g, u, P);
}

__device__ __forceinline__ void ne_primitives(double g, const double u[5], double P[4])
{
    ifp::Fast ar;
    ne_primitives(ar, g, u, P);
    if (!ar.ok) {
        const double w[5] = {u[0], u[1], u[2], u[3], u[4]};
        double Q[4];
        ne_primitives_native(g, w, Q);
#pragma unroll
        for (int c = 0; c < 4; ++c) P[c] = Q[c];
    }
}

// ---------------------------------------------------------------------------
// SR con2prim.  With E = tau + D and s = |S|, the pressure is the root of
//   f(p) = p - (g-1) rho eps(p),  v = s/(E+p), W = (1-v^2)^(-1/2), rho = D/W,
//   rho eps = tau - v^2 [(E+p) - D W/(W+1)]   (from the definitions of D, S, tau),
//   f'(p) = 1 - (g-1) v^2 (1 - D W/(E+p)),
// bracketed by [max(0, s-E), (g-1) tau]; Newton steps that leave the bracket
// become bisections, except a step landing exactly on an end that is still its
// a-priori bound (at v = 0 the root is (g-1) tau itself); the bracket follows
// the sign of f; stop once
// |dp| <= 2^-48 p and take one more Newton step.
struct C2PEval {
    double f, step;  // f and f / f'
};

// E = tau + D.  Six divisions (the step's included) and a square root bound an
// evaluation; they run on the integer ALU (dg_intfp64.cuh), the additions and the
// products on the FP64 pipe.
template <class A>
__device__ __forceinline__ C2PEval sr_c2p_eval(A &ar, double g, double D, double E, double s2, double tau, double p)
{
    const double Ep = E + p;
    const double v2 = ar.div(s2, Ep * Ep);
    const double W = ar.div(1.0, ar.root(1.0 - v2));
    const double DW = D * W;
    const double rhoeps = tau - v2 * (Ep - ar.div(DW, W + 1.0));
    C2PEval r;
    r.f = p - (g - 1.0) * rhoeps;
    r.step = ar.div(r.f, 1.0 - (g - 1.0) * v2 * (1.0 - ar.div(DW, Ep)));
    return r;
}

static __device__ __noinline__ C2PEval sr_c2p_eval_native(double g, double D, double E, double s2, double tau, double p)
{
    ifp::Native ar;
    return sr_c2p_eval(ar, g, D, E, s2, tau, p);
}

static __device__ __noinline__ bool sr_unphysical_native(const double *u)
{
    const double s2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
    return !(u[0] > 0.0) || !(u[4] > 0.0) || !(s2 < u[4] * (u[4] + 2.0 * u[0]));
}

// ---------------------------------------------------------------------------
// Divisions, square roots and most products run on the integer ALU; the additions and
// the last products of the HLL flux, as many as balance the two, on the FP64 pipe.
// The face kernel takes the axis at run time: components by selection (indexing a
// register array with a runtime value would move it to local memory).
__device__ __forceinline__ double pick_axis(int a, double x, double y, double z) { return a == 0 ? x : (a == 1 ? y : z); }

// Physical flux along axis a, common to both systems with alpha = 1, beta = 0:
// F = [U0 v_a, S_i v_a + p delta_ia, (U4 + p) v_a].
template <class A>
__device__ __forceinline__ void flux_axis(A &ar, const double u[5], const double P[4], int a, double F[5])
{
    const double va = pick_axis(a, P[0], P[1], P[2]), p = P[3];
    F[0] = ar.mul(u[0], va);
    F[1] = ar.mul(u[1], va);
    F[2] = ar.mul(u[2], va);
    F[3] = ar.mul(u[3], va);
    const double fn = pick_axis(a, F[1], F[2], F[3]) + p;
    if (a == 0) F[1] = fn;
    else if (a == 1) F[2] = fn;
    else F[3] = fn;
    F[4] = ar.mul(u[4] + p, va);
}

// Extreme characteristic speeds along axis a (eq:CharDecomp).
template <int SYS, class A>
__device__ __forceinline__ void speeds_axis(A &ar, double g, const double u[5], const double P[4], int a,
                                            double &lmin, double &lmax)
{
    const double va = pick_axis(a, P[0], P[1], P[2]), p = P[3];
    if (SYS == 0) {
        const double c = ar.root(ar.div(ar.mul(g, p), u[0]));
        lmin = va - c;
        lmax = va + c;
        return;
    }
    const double v2 = ar.mul(P[0], P[0]) + ar.mul(P[1], P[1]) + ar.mul(P[2], P[2]);
    const double w2i = 1.0 - v2;
    const double cs2 = ar.div(ar.mul(g, p), ar.mul(u[4] + u[0] + p, w2i));
    const double om = 1.0 - cs2;
    const double den = 1.0 - ar.mul(v2, cs2);
    double disc = ar.mul(w2i, den - ar.mul(ar.mul(va, va), om));
    if (disc < 0.0) disc = 0.0;
    const double rt = ar.mul(ar.root(cs2), ar.root(disc));
    const double vo = ar.mul(va, om);
    const typename A::Div dd = ar.divisor(den);
    lmin = ar.div(vo - rt, dd);
    lmax = ar.div(vo + rt, dd);
}

// Roe dissipation D = sum_i alpha_i |lambda_i| e_i of eq:Roe for the Newtonian
// ideal gas (Sec. 3.2.3): the flux Jacobian along e_a at the Roe averages
// (eq:RoeAverages) of the velocity and of h = (E + p)/rho, eigenvalues u_n - c,
// u_n (x3), u_n + c with c^2 = (g-1)(h - |v|^2/2), wave strengths from the jump on
// the left eigenvectors in the frame (normal, t1, t2) = (a, a+1, a+2).
template <class A>
__device__ __forceinline__ void roe_dissipation(A &ar, double g, int a, const double uL[5], const double PL[4],
                                                const double uR[5], const double PR[4], double D[5])
{
    const double sl = ar.root(uL[0]), sr = ar.root(uR[0]);
    const typename A::Div wsum = ar.divisor(sl + sr);
    double vh[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) vh[i] = ar.div(ar.mul(sl, PL[i]) + ar.mul(sr, PR[i]), wsum);
    const double hL = ar.div(uL[4] + PL[3], uL[0]), hR = ar.div(uR[4] + PR[3], uR[0]);
    const double hh = ar.div(ar.mul(sl, hL) + ar.mul(sr, hR), wsum);
    const double q2 = ar.mul(vh[0], vh[0]) + ar.mul(vh[1], vh[1]) + ar.mul(vh[2], vh[2]);
    const double c2 = ar.mul(g - 1.0, hh - 0.5 * q2);
    const double c = ar.root(c2);
    const double un = pick_axis(a, vh[0], vh[1], vh[2]), ut1 = pick_axis(a, vh[1], vh[2], vh[0]);
    const double ut2 = pick_axis(a, vh[2], vh[0], vh[1]);
    const double jx = uR[1] - uL[1], jy = uR[2] - uL[2], jz = uR[3] - uL[3];
    const double j1 = uR[0] - uL[0], jn = pick_axis(a, jx, jy, jz);
    const double jt1 = pick_axis(a, jy, jz, jx), jt2 = pick_axis(a, jz, jx, jy), j5 = uR[4] - uL[4];
    const double al3 = jt1 - ar.mul(ut1, j1);
    const double al4 = jt2 - ar.mul(ut2, j1);
    const double j5b = j5 - ar.mul(al3, ut1) - ar.mul(al4, ut2);
    const double al2 = ar.mul(ar.div(g - 1.0, c2), ar.mul(j1, hh - ar.mul(un, un)) + ar.mul(un, jn) - j5b);
    const double al1 = ar.div(ar.mul(j1, un + c) - jn - ar.mul(c, al2), 2.0 * c);
    const double al5 = j1 - (al1 + al2);
    const double w1 = ar.mul(fabs(un - c), al1), w2 = ar.mul(fabs(un), al2), w5 = ar.mul(fabs(un + c), al5);
    const double w3 = ar.mul(fabs(un), al3), w4 = ar.mul(fabs(un), al4);
    const double w = w1 + w2 + w5;
    const double dn = ar.mul(w1, un - c) + ar.mul(w2, un) + ar.mul(w5, un + c);
    const double d1 = ar.mul(w, ut1) + w3, d2 = ar.mul(w, ut2) + w4;
    D[0] = w;
    D[1] = pick_axis(a, dn, d2, d1);
    D[2] = pick_axis(a, d1, dn, d2);
    D[3] = pick_axis(a, d2, d1, dn);
    D[4] = ar.mul(w1, hh - ar.mul(un, c)) + ar.mul(w2, 0.5 * q2) + ar.mul(w3, ut1) + ar.mul(w4, ut2) + ar.mul(w5, hh + ar.mul(un, c));
}

// Numerical flux along +e_a between the lower state L and the upper state R:
// FLX = 0 local Lax-Friedrichs (eq:LLF), 1 HLL with Davis speeds (eq:HLL), 2 Roe
// (eq:Roe, Newtonian).
template <int SYS, int FLX, class A>
__device__ __forceinline__ void num_flux(A &ar, double g, int a, const double uL[5], const double PL[4],
                                         const double uR[5], const double PR[4], double Fs[5])
{
    double FL[5], FR[5], lminL, lmaxL, lminR, lmaxR;
    flux_axis(ar, uL, PL, a, FL);
    flux_axis(ar, uR, PR, a, FR);
    if (FLX == 2) {
        double D[5];
        roe_dissipation(ar, g, a, uL, PL, uR, PR, D);
#pragma unroll
        for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (FL[v] + FR[v]) - 0.5 * D[v];
        return;
    }
    speeds_axis<SYS>(ar, g, uL, PL, a, lminL, lmaxL);
    speeds_axis<SYS>(ar, g, uR, PR, a, lminR, lmaxR);
    if (FLX == 0) {
        const double al = ar.greatest(ar.greatest(fabs(lminL), fabs(lmaxL)), ar.greatest(fabs(lminR), fabs(lmaxR)));
        const double hal = 0.5 * al;
#pragma unroll
        for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (FL[v] + FR[v]) - ar.mul(hal, uR[v] - uL[v]);
    } else {
        const double cmin = ar.least(ar.least(lminL, lminR), 0.0);
        const double cmax = ar.greatest(ar.greatest(lmaxL, lmaxR), 0.0);
        const double den = cmax - cmin;
        if (ar.positive(den)) {
            const typename A::Div dd = ar.divisor(den);
            const double cc = ar.div(ar.mul(cmin, cmax), dd);
#pragma unroll
            for (int v = 0; v < 5; ++v)
                Fs[v] = ar.div(cmax * FL[v] - cmin * FR[v], dd) + cc * (uR[v] - uL[v]);
        } else {
#pragma unroll
            for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (FL[v] + FR[v]);
        }
    }
}

template <int SYS, int FLX>
static __device__ __noinline__ void num_flux_native(double g, int a, const double *uL, const double *PL, const double *uR,
                                                    const double *PR, double *Fs)
{
    ifp::Native ar;
    num_flux<SYS, FLX>(ar, g, a, uL, PL, uR, PR, Fs);
}

template <int SYS, int FLX>
__device__ __forceinline__ void num_flux(double g, int a, const double uL[5], const double PL[4], const double uR[5],
                                         const double PR[4], double Fs[5])
{
    ifp::Fast ar;
    num_flux<SYS, FLX>(ar, g, a, uL, PL, uR, PR, Fs);
    if (!ar.ok) {
        const double l[5] = {uL[0], uL[1], uL[2], uL[3], uL[4]}, r[5] = {uR[0], uR[1], uR[2], uR[3], uR[4]};
        const double p[4] = {PL[0], PL[1], PL[2], PL[3]}, q[4] = {PR[0], PR[1], PR[2], PR[3]};
        double F[5];
        num_flux_native<SYS, FLX>(g, a, l, p, r, q, F);
#pragma unroll
        for (int v = 0; v < 5; ++v) Fs[v] = F[v];
    }
}

// Largest |characteristic speed| over the three axes.  Per axis it is
// (|x| + c) [/ d] of the two speeds (x -+ c) [/ d] with c >= 0: rounding is monotone and
// symmetric, so these are the bits of the larger magnitude.  NaN speeds (a negative
// pressure) count as 0, as fmax over the speeds themselves would have it.
template <int SYS, class A>
__device__ __forceinline__ double max_speed(A &ar, double g, const double u[5], const double P[4])
{
    const double p = P[3];
    if (SYS == 0) {
        const double c = ar.root(ar.div(ar.mul(g, p), u[0]));
        return ar.greatest(fabs(P[0]), ar.greatest(fabs(P[1]), fabs(P[2]))) + c;
    }
    const double v2 = ar.mul(P[0], P[0]) + ar.mul(P[1], P[1]) + ar.mul(P[2], P[2]);
    const double w2i = 1.0 - v2;
    const double cs2 = ar.div(ar.mul(g, p), ar.mul(u[4] + u[0] + p, w2i));
    const double cs = ar.root(cs2);
    const double om = 1.0 - cs2;
    const double den = 1.0 - ar.mul(v2, cs2);
    const typename A::Div dd = ar.divisor(den);
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double va = P[a];
        const double disc = ar.mul(w2i, den - ar.mul(ar.mul(va, va), om));
        const double rt = ar.mul(cs, ar.root(disc));
        s = ar.greatest(s, fabs(ar.div(fabs(ar.mul(va, om)) + rt, dd)));
    }
    return s;
}

template <int SYS>
static __device__ __noinline__ double max_speed_native(double g, const double *u, const double *P)
{
    double s = 0.0;
    ifp::Native ar;
    for (int a = 0; a < 3; ++a) {
        double lo, hi;
        speeds_axis<SYS>(ar, g, u, P, a, lo, hi);
        s = fmax(s, fmax(fabs(lo), fabs(hi)));
    }
    return s;
}

template <int SYS>
__device__ __forceinline__ double max_speed(double g, const double u[5], const double P[4])
{
    ifp::Fast ar;
    double s = max_speed<SYS>(ar, g, u, P);
    if (!ar.ok) {
        const double w[5] = {u[0], u[1], u[2], u[3], u[4]}, q[4] = {P[0], P[1], P[2], P[3]};
        s = max_speed_native<SYS>(g, w, q);
    }
    return s;
}

// SR conserved-variable fix (Sec. 2.1.4): D >= d_atm, tau >= tau_atm D and
// S^2 <= (1 - 1e-12) tau (tau + 2D).  Returns the variables it set, as a bit
// mask (bit v for u[v]; the three momenta together), 0 if u is unchanged.
template <class A>
__device__ __forceinline__ unsigned sr_fix(A &ar, double d_atm, double tau_atm, double u[5])
{
    unsigned ch = 0;
    if (!(u[0] >= d_atm)) { u[0] = d_atm; ch |= 1u; }
    const double tmin = ar.mul(tau_atm, u[0]);
    if (!(u[4] >= tmin)) { u[4] = tmin; ch |= 16u; }
    const double s2 = ar.mul(u[1], u[1]) + ar.mul(u[2], u[2]) + ar.mul(u[3], u[3]);
    const double s2max = ar.mul(1.0 - 1e-12, ar.mul(u[4], u[4] + 2.0 * u[0]));
    if (s2 > s2max) {
        const double f = ar.root(ar.div(s2max, s2));
        u[1] = ar.mul(u[1], f);
        u[2] = ar.mul(u[2], f);
        u[3] = ar.mul(u[3], f);
        ch |= 14u;
    }
    return ch;
}

static __device__ __noinline__ unsigned sr_fix_native(double d_atm, double tau_atm, double *u)
{
    ifp::Native ar;
    return sr_fix(ar, d_atm, tau_atm, u);
}

__device__ __forceinline__ unsigned sr_fix(double d_atm, double tau_atm, double u[5])
{
    ifp::Fast ar;
    double w[5] = {u[0], u[1], u[2], u[3], u[4]};
    unsigned ch = sr_fix(ar, d_atm, tau_atm, w);
    if (!ar.ok) {
        double q[5] = {u[0], u[1], u[2], u[3], u[4]};
        ch = sr_fix_native(d_atm, tau_atm, q);
#pragma unroll
        for (int v = 0; v < 5; ++v) w[v] = q[v];
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) u[v] = w[v];
    return ch;
}

// The same as a call, for kernels where few nodes need it.
static __device__ __noinline__ unsigned sr_fix_call(double d_atm, double tau_atm, double *u)
{
    double w[5] = {u[0], u[1], u[2], u[3], u[4]};
    const unsigned ch = sr_fix(d_atm, tau_atm, w);
#pragma unroll
    for (int v = 0; v < 5; ++v) u[v] = w[v];
    return ch;
}

// Sign tests, minmod (eq:MinMod) and magnitude comparisons of doubles done on
// their bit patterns, on the integer ALU instead of the FP64 pipe (which bounds
// the limiter kernels).  They decide exactly as the floating-point forms, NaN included:
// - a double is > 0 iff its bits, read as a signed integer, lie in (0, +inf];
// - it is < 0 iff its sign bit is set and its magnitude bits lie in (0, inf]
//   (-0 is not negative);
// - doubles of one sign are ordered like their bits, reversed for negatives, so
//   among three positive or three negative doubles the one closest to 0 (the
//   minmod pick) has the smallest bit pattern as a signed integer;
// - |x| > c and |x| <= c for a finite c >= 0 compare the magnitude bits with c's.
constexpr long long kMagBits = 0x7fffffffffffffffLL;
constexpr long long kInfBits = 0x7ff0000000000000LL;

__device__ __forceinline__ bool bits_pos(long long b) { return b > 0 && b <= kInfBits; }
__device__ __forceinline__ bool bits_neg(long long b)
{
    const long long m = b & kMagBits;
    return b < 0 && m != 0 && m <= kInfBits;
}

__device__ __forceinline__ double minmod3_bits(double a1, double a2, double a3)
{
    const long long b1 = __double_as_longlong(a1), b2 = __double_as_longlong(a2), b3 = __double_as_longlong(a3);
    const bool pos = bits_pos(b1) & bits_pos(b2) & bits_pos(b3);
    const bool neg = bits_neg(b1) & bits_neg(b2) & bits_neg(b3);
    return (pos | neg) ? __longlong_as_double(min(b1, min(b2, b3))) : 0.0;
}

// |x| > c, for finite c >= 0
__device__ __forceinline__ bool abs_gt(double x, double c)
{
    const long long m = __double_as_longlong(x) & kMagBits;
    return m > __double_as_longlong(c) && m <= kInfBits;
}

// |x| <= c, for finite c >= 0
__device__ __forceinline__ bool abs_le(double x, double c)
{
    return (__double_as_longlong(x) & kMagBits) <= __double_as_longlong(c);
}

}  // namespace dg
