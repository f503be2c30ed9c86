// dg_con2prim_fp64.cuh -- SR con2prim of many nodes in FP64 (Sec. 2.1.2): the
// safeguarded Newton iteration of dg_physics.cuh with its lanes kept busy.
//
// Iteration counts differ widely between nodes (1 to 46 on random states, 10 on
// average), and a warp that waits for its slowest node wastes half of its work on a
// unit that charges a warp instruction the same for one lane as for 32.  Here a warp
// works through many nodes: starting values are prepared 32 at a time and queued in
// shared memory, a lane whose node has converged takes the next one from the queue, and
// finished nodes are queued again and completed 32 at a time.  Every node runs the
// same iterations as on its own.
#pragma once

#include "dg_physics.cuh"

namespace dg {

constexpr int kC2pThreads = 128;
constexpr int kC2pRing = 64;  // queue slots per warp: fewer than 32 waiting plus one batch

struct C2pQueue {
    double D[kC2pRing], s2[kC2pRing], tau[kC2pRing], plo[kC2pRing], p[kC2pRing];
    long long i[kC2pRing];
};
struct C2pWarp {
    C2pQueue in, out;  // (out.plo unused)
};

// The iteration's two rare cases in FP64 instructions.
static __device__ __noinline__ double c2p_bisect_native(double plo, double phi) { return 0.5 * (plo + phi); }
static __device__ __noinline__ bool c2p_close_native(double pn, double p) { return fabs(pn - p) <= 0x1p-48 * pn; }

// All nodes i = 32 b + lane of the batches b = warp, warp + nwarps, ... below count.
// io.load(i, u) the conserved state (after any fix), io.guess(i) the starting pressure
// (< 0: the standard guess (g-1) tau), io.bad(i) an unphysical state, io.iterations(i,
// n, status) the iteration's end (status 0 converged, 2 not), io.finish(i, D, s2, E, p)
// the pressure.
template <class IO>
__device__ __forceinline__ void c2p_warp(IO &io, C2pWarp &Q, double g, long long count, long long warp, long long nwarps)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    long long next = warp * 32;
    int head = 0, cnt = 0, ohead = 0, ocnt = 0;  // the rings' first entry and length (uniform)
    bool act = false, last = false, lo_moved = false, hi_moved = false;
    double D = 1.0, E = 2.0, s2 = 0.0, tau = 1.0, plo = 0.0, phi = g - 1.0, p = g - 1.0;
    long long node = 0;
    int it = 0;

    auto finish_batch = [&](int n) {
        if (lane < n) {
            const int k = (ohead + lane) & (kC2pRing - 1);
            io.finish(Q.out.i[k], Q.out.D[k], Q.out.s2[k], Q.out.tau[k] + Q.out.D[k], Q.out.p[k]);
        }
        ohead += n;
        ocnt -= n;
        __syncwarp();
    };

    for (;;) {
        const unsigned idle = __ballot_sync(full, !act);
        if (idle) {
            const int want = __popc(idle);
            while (cnt < want && next < count) {
                const long long i = next + lane;
                bool ok = false;
                double u[5], t2 = 0.0, tlo = 0.0, tp = 0.0;
                if (i < count) {
                    io.load(i, u);
                    t2 = ifp::mul(u[1], u[1]) + ifp::mul(u[2], u[2]) + ifp::mul(u[3], u[3]);
                    ok = u[0] > 0.0 && u[4] > 0.0 && t2 < ifp::mul(u[4], u[4] + 2.0 * u[0]);
                    if (ok) {
                        tlo = ifp::root(t2) - (u[4] + u[0]);
                        if (tlo < 0.0) tlo = 0.0;
                        const double thi = ifp::mul(g - 1.0, u[4]), gs = io.guess(i);
                        tp = gs >= 0.0 ? gs : thi;
                        if (tp < tlo) tp = tlo;
                        if (tp > thi) tp = thi;
                    } else {
                        io.bad(i);
                    }
                }
                const unsigned b = __ballot_sync(full, ok);
                if (ok) {
                    const int k = (head + cnt + __popc(b & below)) & (kC2pRing - 1);
                    Q.in.D[k] = u[0];
                    Q.in.s2[k] = t2;
                    Q.in.tau[k] = u[4];
                    Q.in.plo[k] = tlo;
                    Q.in.p[k] = tp;
                    Q.in.i[k] = i;
                }
                cnt += __popc(b);
                next += nwarps * 32;
            }
            __syncwarp();
            const int rank = __popc(idle & below);
            if (!act && rank < cnt) {
                const int k = (head + rank) & (kC2pRing - 1);
                D = Q.in.D[k];
                s2 = Q.in.s2[k];
                tau = Q.in.tau[k];
                plo = Q.in.plo[k];
                E = tau + D;
                phi = ifp::mul(g - 1.0, tau);
                p = Q.in.p[k];
                node = Q.in.i[k];
                it = 0;
                last = lo_moved = hi_moved = false;  // an end still at its a-priori bound may be landed on
                act = true;
            }
            const int took = want < cnt ? want : cnt;
            head += took;
            cnt -= took;
            __syncwarp();
            if (!__ballot_sync(full, act)) break;
        }
        // one iteration (or, after the step below the tolerance, one more Newton step)
        ifp::Fast ar;
        C2PEval r = sr_c2p_eval(ar, g, D, E, s2, tau, p);
        if (!ar.ok) r = sr_c2p_eval_native(g, D, E, s2, tau, p);
        double pn = p - r.step;
        bool done = last;
        int iters = it + 2, status = 0;
        if (!last) {
            if (((ifp::hi32(ifp::dbits(r.f)) << 1) | ifp::lo32(ifp::dbits(r.f))) == 0u) {
                pn = p;
                done = true;
                iters = it + 1;
            } else {
                if (bits_pos((long long)ifp::dbits(r.f))) {
                    phi = p;
                    hi_moved = true;
                } else {
                    plo = p;
                    lo_moved = true;
                }
                // brackets and iterates are non-negative, so their bits order as integers
                const long long kn = (long long)ifp::dbits(pn), kl = (long long)ifp::dbits(plo);
                const long long kh = (long long)ifp::dbits(phi);
                const bool in = kn >= 0 && ((kn > kl && kn < kh) || (kn == kh && !hi_moved) || (kn == kl && !lo_moved));
                // Some lane of almost every warp bisects, and some lane is close to its end: on
                // the FP64 pipe these two would cost three of an iteration's 16 instructions.
                // (On the integer ALU they leave that pipe room for all of the evaluation's
                // products: 1760 us for 2^22 random states against 1815; one without the
                // other gains nothing.)
                if (!in) {
                    if (ifp::half_sum_ok(plo, phi)) pn = ifp::half_sum_fast(plo, phi);
                    else pn = c2p_bisect_native(plo, phi);
                }
                last = ifp::close_fast(pn, p);
                if (!ifp::close_ok(pn, p)) last = c2p_close_native(pn, p);
                if (!last && kh <= kl && kh < kInfBits) {
                    done = true;
                    iters = it + 1;
                } else if (!last && ++it == 200) {
                    done = true;
                    iters = 201;
                    status = 2;
                }
            }
        }
        p = pn;
        const unsigned fin = __ballot_sync(full, act && done);
        if (fin) {
            if (act && done) {
                io.iterations(node, iters, status);
                const int k = (ohead + ocnt + __popc(fin & below)) & (kC2pRing - 1);
                Q.out.D[k] = D;
                Q.out.s2[k] = s2;
                Q.out.tau[k] = tau;
                Q.out.p[k] = p;
                Q.out.i[k] = node;
                act = false;
            }
            ocnt += __popc(fin);
            __syncwarp();
            if (ocnt >= 32) finish_batch(32);
        }
    }
    __syncwarp();
    while (ocnt > 0) finish_batch(ocnt < 32 ? ocnt : 32);
}

// CTAs for `count` nodes: every warp resident at once (`ctas` per SM), so that each takes
// an equal share of the batches; one batch per warp when there are fewer.  k_con2prim
// runs six per SM (80 registers; 1709 us for 2^22 random states against 1740 with five and
// 1798 with seven), k_primitives_sr, which needs 96 registers, five (16^3, n = 5: 1402 us
// per step against 1455 with six).
inline unsigned c2p_grid(long long count, int ctas)
{
    const long long batches = (count + 31) / 32, warps = kC2pThreads / 32;
    const long long blocks = (batches + warps - 1) / warps;
    return (unsigned)(blocks < 1 ? 1 : blocks < kNumSMs * ctas ? blocks : kNumSMs * ctas);
}

}  // namespace dg
