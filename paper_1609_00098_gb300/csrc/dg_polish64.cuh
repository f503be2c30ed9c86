// dg_polish64.cuh -- the residual of the FP64 con2prim polish of the mixed path (Sec. 2.1.2) and
// its derivative, three divisions and a root on the integer ALU (dg_intfp64.cuh).
#pragma once

#include "dg_intfp64.cuh"

namespace dg {

// f(p) = p - (g - 1) rho eps(p), and the Newton step f / f' as fq / dq, both multiplied by
// q = 1/W:  f' = 1 - c (1 - D W/Ep) with c = (g - 1) v^2 and Ep = tau + D + p, so
// q f' = q (1 - c) + c D/Ep.  Both terms are positive: nothing cancels where f' is small
// (f' falls like 1/W^2 as g -> 2, where FP32 leaves no correct digit of it at W > 1e3).
struct PolishEval {
    double f, fq, dq, scale;  // scale: the size of f's terms
};

__host__ __device__ __forceinline__ PolishEval sr_polish_eval(double g, double D, double E, double s2, double tau,
                                                              double p)
{
    PolishEval r;
    const double Ep = E + p;
    const double inv = ifp::div(1.0, Ep);
    const double v2 = s2 * inv * inv;
    const double q = ifp::root(1.0 - v2);
    // rho eps with D W/(W + 1) = D/(1 + q)
    const double rhoeps = tau - v2 * (Ep - ifp::div(D, 1.0 + q));
    const double c = (g - 1.0) * v2;
    r.f = p - (g - 1.0) * rhoeps;
    r.fq = r.f * q;
    r.dq = q * (1.0 - c) + c * (D * inv);
    r.scale = p + (g - 1.0) * (tau + v2 * Ep);
    return r;
}

}  // namespace dg
