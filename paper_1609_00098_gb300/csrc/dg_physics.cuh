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
__device__ __forceinline__ void ne_primitives(double g, const double u[5], double P[4])
{
    const double inv = ifp::div(1.0, u[0]);
    P[0] = ifp::mul(u[1], inv);
    P[1] = ifp::mul(u[2], inv);
    P[2] = ifp::mul(u[3], inv);
    P[3] = ifp::mul(g - 1.0, u[4] - 0.5 * (ifp::mul(u[1], P[0]) + ifp::mul(u[2], P[1]) + ifp::mul(u[3], P[2])));
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
    double f, df;
};

// E = tau + D.  Six divisions and a square root bound an evaluation; they and the
// products run on the integer ALU (dg_intfp64.cuh).
__device__ __forceinline__ C2PEval sr_c2p_eval(double g, double D, double E, double s2, double tau, double p)
{
    C2PEval r;
    const double Ep = E + p;
    const double v2 = ifp::div(s2, ifp::mul(Ep, Ep));
    const double W = ifp::div(1.0, ifp::root(1.0 - v2));
    const double DW = ifp::mul(D, W);
    const double rhoeps = tau - ifp::mul(v2, Ep - ifp::div(DW, W + 1.0));
    r.f = p - ifp::mul(g - 1.0, rhoeps);
    r.df = 1.0 - ifp::mul(ifp::mul(g - 1.0, v2), 1.0 - ifp::div(DW, Ep));
    return r;
}

__device__ __forceinline__ bool sr_unphysical(const double u[5])
{
    const double s2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
    return !(u[0] > 0.0) || !(u[4] > 0.0) || !(s2 < u[4] * (u[4] + 2.0 * u[0]));
}

// ---------------------------------------------------------------------------
// The face kernel takes the axis at run time: components by selection (indexing a
// register array with a runtime value would move it to local memory).
__device__ __forceinline__ double pick_axis(int a, double x, double y, double z) { return a == 0 ? x : (a == 1 ? y : z); }

// Physical flux along axis a, common to both systems with alpha = 1, beta = 0:
// F = [U0 v_a, S_i v_a + p delta_ia, (U4 + p) v_a].
__device__ __forceinline__ void flux_axis(const double u[5], const double P[4], int a, double F[5])
{
    const double va = pick_axis(a, P[0], P[1], P[2]), p = P[3];
    F[0] = ifp::mul(u[0], va);
    F[1] = ifp::mul(u[1], va);
    F[2] = ifp::mul(u[2], va);
    F[3] = ifp::mul(u[3], va);
    const double fn = pick_axis(a, F[1], F[2], F[3]) + p;
    if (a == 0) F[1] = fn;
    else if (a == 1) F[2] = fn;
    else F[3] = fn;
    F[4] = ifp::mul(u[4] + p, va);
}

// Extreme characteristic speeds along axis a (eq:CharDecomp).
template <int SYS>
__device__ __forceinline__ void speeds_axis(double g, const double u[5], const double P[4], int a,
                                            double &lmin, double &lmax)
{
    const double va = pick_axis(a, P[0], P[1], P[2]), p = P[3];
    if (SYS == 0) {
        const double c = ifp::root(ifp::div(ifp::mul(g, p), u[0]));
        lmin = va - c;
        lmax = va + c;
        return;
    }
    const double v2 = ifp::mul(P[0], P[0]) + ifp::mul(P[1], P[1]) + ifp::mul(P[2], P[2]);
    const double w2i = 1.0 - v2;
    const double cs2 = ifp::div(ifp::mul(g, p), ifp::mul(u[4] + u[0] + p, w2i));
    const double om = 1.0 - cs2;
    const double den = 1.0 - ifp::mul(v2, cs2);
    double disc = ifp::mul(w2i, den - ifp::mul(ifp::mul(va, va), om));
    if (disc < 0.0) disc = 0.0;
    const double rt = ifp::mul(ifp::root(cs2), ifp::root(disc));
    const double vo = ifp::mul(va, om);
    const ifp::Divisor dd = ifp::divisor(den);
    lmin = ifp::div(vo - rt, dd);
    lmax = ifp::div(vo + rt, dd);
}

// Roe dissipation D = sum_i alpha_i |lambda_i| e_i of eq:Roe for the Newtonian
// ideal gas (Sec. 3.2.3): the flux Jacobian along e_a at the Roe averages
// (eq:RoeAverages) of the velocity and of h = (E + p)/rho, eigenvalues u_n - c,
// u_n (x3), u_n + c with c^2 = (g-1)(h - |v|^2/2), wave strengths from the jump on
// the left eigenvectors in the frame (normal, t1, t2) = (a, a+1, a+2).
__device__ __forceinline__ void roe_dissipation(double g, int a, const double uL[5], const double PL[4],
                                                const double uR[5], const double PR[4], double D[5])
{
    using ifp::mul;
    const double sl = ifp::root(uL[0]), sr = ifp::root(uR[0]);
    const ifp::Divisor wsum = ifp::divisor(sl + sr);
    double vh[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) vh[i] = ifp::div(mul(sl, PL[i]) + mul(sr, PR[i]), wsum);
    const double hL = ifp::div(uL[4] + PL[3], uL[0]), hR = ifp::div(uR[4] + PR[3], uR[0]);
    const double hh = ifp::div(mul(sl, hL) + mul(sr, hR), wsum);
    const double q2 = mul(vh[0], vh[0]) + mul(vh[1], vh[1]) + mul(vh[2], vh[2]);
    const double c2 = mul(g - 1.0, hh - 0.5 * q2);
    const double c = ifp::root(c2);
    const double un = pick_axis(a, vh[0], vh[1], vh[2]), ut1 = pick_axis(a, vh[1], vh[2], vh[0]);
    const double ut2 = pick_axis(a, vh[2], vh[0], vh[1]);
    const double jx = uR[1] - uL[1], jy = uR[2] - uL[2], jz = uR[3] - uL[3];
    const double j1 = uR[0] - uL[0], jn = pick_axis(a, jx, jy, jz);
    const double jt1 = pick_axis(a, jy, jz, jx), jt2 = pick_axis(a, jz, jx, jy), j5 = uR[4] - uL[4];
    const double al3 = jt1 - mul(ut1, j1);
    const double al4 = jt2 - mul(ut2, j1);
    const double j5b = j5 - mul(al3, ut1) - mul(al4, ut2);
    const double al2 = mul(ifp::div(g - 1.0, c2), mul(j1, hh - mul(un, un)) + mul(un, jn) - j5b);
    const double al1 = ifp::div(mul(j1, un + c) - jn - mul(c, al2), 2.0 * c);
    const double al5 = j1 - (al1 + al2);
    const double w1 = mul(fabs(un - c), al1), w2 = mul(fabs(un), al2), w5 = mul(fabs(un + c), al5);
    const double w3 = mul(fabs(un), al3), w4 = mul(fabs(un), al4);
    const double w = w1 + w2 + w5;
    const double dn = mul(w1, un - c) + mul(w2, un) + mul(w5, un + c);
    const double d1 = mul(w, ut1) + w3, d2 = mul(w, ut2) + w4;
    D[0] = w;
    D[1] = pick_axis(a, dn, d2, d1);
    D[2] = pick_axis(a, d1, dn, d2);
    D[3] = pick_axis(a, d2, d1, dn);
    D[4] = mul(w1, hh - mul(un, c)) + mul(w2, 0.5 * q2) + mul(w3, ut1) + mul(w4, ut2) + mul(w5, hh + mul(un, c));
}

// Numerical flux along +e_a between the lower state L and the upper state R:
// FLX = 0 local Lax-Friedrichs (eq:LLF), 1 HLL with Davis speeds (eq:HLL), 2 Roe
// (eq:Roe, Newtonian).
template <int SYS, int FLX>
__device__ __forceinline__ void num_flux(double g, int a, const double uL[5], const double PL[4],
                                         const double uR[5], const double PR[4], double Fs[5])
{
    double FL[5], FR[5], lminL, lmaxL, lminR, lmaxR;
    flux_axis(uL, PL, a, FL);
    flux_axis(uR, PR, a, FR);
    if (FLX == 2) {
        double D[5];
        roe_dissipation(g, a, uL, PL, uR, PR, D);
#pragma unroll
        for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (FL[v] + FR[v]) - 0.5 * D[v];
        return;
    }
    speeds_axis<SYS>(g, uL, PL, a, lminL, lmaxL);
    speeds_axis<SYS>(g, uR, PR, a, lminR, lmaxR);
    if (FLX == 0) {
        const double al = ifp::greatest(ifp::greatest(fabs(lminL), fabs(lmaxL)), ifp::greatest(fabs(lminR), fabs(lmaxR)));
        const double hal = 0.5 * al;
#pragma unroll
        for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (FL[v] + FR[v]) - ifp::mul(hal, uR[v] - uL[v]);
    } else {
        const double cmin = ifp::least(ifp::least(lminL, lminR), 0.0);
        const double cmax = ifp::greatest(ifp::greatest(lmaxL, lmaxR), 0.0);
        const double den = cmax - cmin;
        if (den > 0.0) {
            const ifp::Divisor dd = ifp::divisor(den);
            const double cc = ifp::div(ifp::mul(cmin, cmax), dd);
#pragma unroll
            for (int v = 0; v < 5; ++v)
                Fs[v] = ifp::div(ifp::mul(cmax, FL[v]) - ifp::mul(cmin, FR[v]), dd) + ifp::mul(cc, uR[v] - uL[v]);
        } else {
#pragma unroll
            for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (FL[v] + FR[v]);
        }
    }
}

// Largest |characteristic speed| over the three axes.
template <int SYS>
__device__ __forceinline__ double max_speed(double g, const double u[5], const double P[4])
{
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double lo, hi;
        speeds_axis<SYS>(g, u, P, a, lo, hi);
        s = ifp::greatest(s, ifp::greatest(fabs(lo), fabs(hi)));
    }
    return s;
}

// SR conserved-variable fix (Sec. 2.1.4): D >= d_atm, tau >= tau_atm D and
// S^2 <= (1 - 1e-12) tau (tau + 2D).  Returns the variables it set, as a bit
// mask (bit v for u[v]; the three momenta together), 0 if u is unchanged.
__device__ __forceinline__ unsigned sr_fix(double d_atm, double tau_atm, double u[5])
{
    unsigned ch = 0;
    if (!(u[0] >= d_atm)) { u[0] = d_atm; ch |= 1u; }
    const double tmin = tau_atm * u[0];
    if (!(u[4] >= tmin)) { u[4] = tmin; ch |= 16u; }
    const double s2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3];
    const double s2max = (1.0 - 1e-12) * (u[4] * (u[4] + 2.0 * u[0]));
    if (s2 > s2max) {
        const double f = sqrt(s2max / s2);
        u[1] *= f;
        u[2] *= f;
        u[3] *= f;
        ch |= 14u;
    }
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
