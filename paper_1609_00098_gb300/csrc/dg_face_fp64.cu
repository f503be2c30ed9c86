// dg_face_fp64.cu -- numerical fluxes of the FP64 path, each interior face once.
//
// One thread per face point: the traces of the two elements (or of an element and a
// ghost holding the analytic exterior state), the numerical flux (Sec. 3.2) along +e_a,
// stored as Fs[face][v][r] with r = t0 + n t1, t0 running along the axis after a.  Face
// a E + e lies between e's lower neighbour along a and e; the upper boundary faces of
// analytic axes follow at 3 E + (ghost index).  The stage kernel lifts the stored
// flux into both elements.
//
// Bound by the FP64 pipe and the integer ALU together: divisions, square roots and
// products run on the latter (dg_intfp64.cuh), additions on the former.  Evaluated
// inside the stage kernel instead, every face was taken twice, by 2 n^2 of the CTA's
// threads, in three passes: the step of the shear layer at 24^3, n = 6 went from 12.0 to
// 9.1 ms with this kernel, that of the relativistic blast at 16^3, n = 5 from 4.7 to 4.1.
// Now 128 us per launch on the former (FP64 pipe 77 %, integer ALU 57 %), 52 on the latter.
#include "dg_internal.h"
#include "dg_physics.cuh"

namespace dg {

namespace {

constexpr int kFaceThreads = 128;

// Five CTAs per SM where their registers allow it (Newtonian LF and HLL: 96 registers,
// 106 without the bound; 24^3, n = 6: 128 us per pass against 138).
template <int SYS, int FLX>
__global__ void __launch_bounds__(kFaceThreads, SYS == 0 && FLX != 2 ? 5 : 0) k_face_fp64(const __grid_constant__ FaceArgs a)
{
    pdl_wait();
    const int n = a.n, n2 = n * n, nn = n2 * n;
    const long long total = (3 * a.E + a.nghost) * n2;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (long long)gridDim.x * blockDim.x) {
        long long f;
        int r;
        if (total <= 0x7fffffffLL) {
            const int fi = (int)g / n2;
            f = fi;
            r = (int)g - fi * n2;
        } else {
            f = g / n2;
            r = (int)(g - f * n2);
        }
        int ax;
        long long eL, eR;  // < 0: ghost -1 - index
        if (f < 3 * a.E) {
            ax = f < a.E ? 0 : f < 2 * a.E ? 1 : 2;
            eR = f - ax * a.E;
            eL = SYS == 0 ? elem_neighbour_bc(eR, a.K, ax, -1, a.gh) : elem_neighbour(eR, a.K, ax, -1);
        } else {
            const long long gi = f - 3 * a.E;
            ax = -1;
            for (int c = 0; c < 3; ++c)
                if ((a.gh.mask >> c) & 1) {
                    const long long cnt = (long long)a.K[(c + 1) % 3] * a.K[(c + 2) % 3];
                    if (gi >= a.gh.base[c][1] && gi < a.gh.base[c][1] + cnt) ax = c;
                }
            if (ax < 0) continue;  // a lower ghost: its face is an element's lower face
            const int b = (ax + 1) % 3, c = (ax + 2) % 3;
            const long long fi = gi - a.gh.base[ax][1];
            int ec[3];
            ec[b] = (int)(fi % a.K[b]);
            ec[c] = (int)(fi / a.K[b]);
            ec[ax] = a.K[ax] - 1;
            eL = ec[0] + (long long)a.K[0] * (ec[1] + (long long)a.K[1] * ec[2]);
            eR = -1 - gi;
        }
        const int sa = ax == 0 ? 1 : ax == 1 ? n : n2, sb = ax == 0 ? n : ax == 1 ? n2 : 1;
        const int sc = ax == 0 ? n2 : ax == 1 ? 1 : n;
        const int off = (r % n) * sb + (r / n) * sc;
        const double *UL = a.Us, *PL = a.P, *UR = a.Us, *PR = a.P;
        if (SYS == 0 && eL < 0) {
            UL = a.gh.U;
            PL = a.gh.P;
            eL = -1 - eL;
        }
        if (SYS == 0 && eR < 0) {
            UR = a.gh.U;
            PR = a.gh.P;
            eR = -1 - eR;
        }
        double ul[5], pl[4], ur[5], pr[4], Fs[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            ul[v] = UL[(eL * 5 + v) * nn + (n - 1) * sa + off];
            ur[v] = UR[(eR * 5 + v) * nn + off];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            pl[c] = PL[(eL * 4 + c) * nn + (n - 1) * sa + off];
            pr[c] = PR[(eR * 4 + c) * nn + off];
        }
        num_flux<SYS, FLX>(a.gamma, ax, ul, pl, ur, pr, Fs);
#pragma unroll
        for (int v = 0; v < 5; ++v) a.Fs[(f * 5 + v) * n2 + r] = Fs[v];
    }
}

}  // namespace

cudaError_t launch_face_fp64(int system, int flux, const FaceArgs &a, cudaStream_t s)
{
    const long long total = (3 * a.E + a.nghost) * a.n * a.n;
    const long long blocks = (total + kFaceThreads - 1) / kFaceThreads;
    const unsigned grid = (unsigned)(blocks < 0x7fffffffLL ? blocks : 0x7fffffffLL);
    void (*kern)(const FaceArgs);
    if (system == 0 && flux == 2) kern = k_face_fp64<0, 2>;
    else if (system == 0 && flux == 0) kern = k_face_fp64<0, 0>;
    else if (system == 0) kern = k_face_fp64<0, 1>;
    else if (flux == 0) kern = k_face_fp64<1, 0>;
    else kern = k_face_fp64<1, 1>;
    return launch_pdl(kern, grid, kFaceThreads, 0, s, a);
}

}  // namespace dg
