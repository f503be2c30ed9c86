// dg_c2p_net.cu -- learned starting guess for the SR con2prim Newton solve
// (Sec. 2.1.2): a 3 -> 64 -> 64 -> 1 SiLU MLP mapping scaled invariants of the
// conserved state to a scaled log pressure, with its own inference, gradient and
// Adam training kernels.  The 64 x 64 layer runs on the tensor cores
// (mma.sync m16n8k16, BF16 operands, FP32 accumulation) in the forward pass and
// in both backward products; the rest is FP32.  Reductions run in a fixed order,
// so training is deterministic.
//
// Parameters (flat, FP32): W1[64][3], b1[64], W2[64][64], b2[64], W3[64], b3.
// Features (E = tau + D, s = |S|): x1 = 2 (log10(tau/D) - lo1)/(hi1 - lo1) - 1,
// x2 = 2 s/E - 1, x3 = 2 (log10 D - lo3)/(hi3 - lo3) - 1; target
// y = (log10(p/E) - y_shift)/y_scale; scales = (lo1, hi1, lo3, hi3, y_shift, y_scale).
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <cstdint>
#include <cstring>

#include "dg_c2p_net.cuh"
#include "dg_mixed.cuh"

namespace dg {

// Weights in shared memory: W2 in BF16 with padded rows (144 bytes: the eight rows an
// ldmatrix touches fall in different banks), W1 and b1 together.
struct NetW {
    __nv_bfloat16 W2[64][NET_W2_LD];
    float4 W1b1[64];
    float b2[64], W3[64], b3, pad[3];  // (contiguous, 16-byte aligned)
};

__device__ __forceinline__ void net_load_weights(NetW &W, const float *P, const __nv_bfloat16 *W2b)
{
    for (int k = threadIdx.x; k < 64 * 32; k += blockDim.x)
        reinterpret_cast<uint32_t *>(&W.W2[k / 32][0])[k % 32] = reinterpret_cast<const uint32_t *>(W2b)[k];
    for (int j = threadIdx.x; j < 64; j += blockDim.x) {
        W.W1b1[j] = make_float4(P[OFF_W1 + 3 * j], P[OFF_W1 + 3 * j + 1], P[OFF_W1 + 3 * j + 2], P[OFF_B1 + j]);
        W.b2[j] = P[OFF_B2 + j];
        W.W3[j] = P[OFF_W3 + j];
    }
    if (threadIdx.x == 0) W.b3 = P[OFF_B3];
}

// Four 8 x 8 BF16 matrices, transposed.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t r[4], const void *row)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(row);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// The network's features from FP32 values (E = tau + D, smag = |S|).
__device__ __forceinline__ float net_x0(float tau, float D, const float sc[6])
{
    return 2.0f * (log10f(tau / D) - sc[0]) / (sc[1] - sc[0]) - 1.0f;
}
__device__ __forceinline__ float net_x1(float smag, float E) { return 2.0f * smag / E - 1.0f; }
__device__ __forceinline__ float net_x2(float D, const float sc[6])
{
    return 2.0f * (log10f(D) - sc[2]) / (sc[3] - sc[2]) - 1.0f;
}

// Features of a state (FP32), and whether all are finite (D and tau positive).
struct NetSample {
    float x0, x1, x2, E, smag, tau;
    bool ok;
};

__device__ __forceinline__ NetSample net_sample(const double v[5], const float sc[6])
{
    NetSample r;
    const float D = f64_to_f32(v[0]);
    const float Sx = f64_to_f32(v[1]), Sy = f64_to_f32(v[2]), Sz = f64_to_f32(v[3]);
    r.tau = f64_to_f32(v[4]);
    r.E = r.tau + D;
    r.smag = sqrtf(Sx * Sx + Sy * Sy + Sz * Sz);
    r.x0 = net_x0(r.tau, D, sc);
    r.x1 = net_x1(r.smag, r.E);
    r.x2 = net_x2(D, sc);
    r.ok = isfinite(r.x0) && isfinite(r.x1) && isfinite(r.x2);
    if (!r.ok) r.x0 = r.x1 = r.x2 = 0.0f;
    return r;
}

// sigma(z) = 1 / (1 + e^-z)
__device__ __forceinline__ float sigmoid32(float z) { return __fdividef(1.0f, 1.0f + __expf(-z)); }

// Layer 1 of two hidden units (unit, unit + 1) for two rows (x[0], x[1] their features): h[c]
// with row c >> 1 and unit c & 1.
__device__ __forceinline__ void net_layer1(const NetW &W, const float x[2][3], int unit, float h[4])
{
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float4 w = W.W1b1[unit + (c & 1)];
        const float *xr = x[c >> 1];
        h[c] = silu(fmaf(w.x, xr[0], fmaf(w.y, xr[1], fmaf(w.z, xr[2], w.w))));
    }
}

// One warp's 16 samples through layers 1 and 2.  This lane holds rows g and g + 8;
// layer 1's values are formed in the A-fragment layout of layer 2, and z2 + b2 comes out
// in its accumulator layout, rows g (c = 0, 1) and g + 8 (c = 2, 3), columns
// 8 nt + 2 tq + (c & 1).
__device__ __forceinline__ void net_forward(const NetW &W, const float x[2][3], float z2[8][4], int lane)
{
    const int tq = lane & 3;
    const int lr_n = (lane & 7) + 8 * (lane >> 4), lr_k = 8 * ((lane >> 3) & 1);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float2 b = *reinterpret_cast<const float2 *>(&W.b2[nt * 8 + 2 * tq]);
        z2[nt][0] = z2[nt][2] = b.x;
        z2[nt][1] = z2[nt][3] = b.y;
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        uint32_t hf[4];
#pragma unroll
        for (int hn = 0; hn < 2; ++hn) {
            float h[4];
            net_layer1(W, x, 16 * kk + 8 * hn + 2 * tq, h);
            hf[2 * hn] = pack_bf16x2(h[0], h[1]);
            hf[2 * hn + 1] = pack_bf16x2(h[2], h[3]);
        }
#pragma unroll
        for (int nt2 = 0; nt2 < 4; ++nt2) {
            uint32_t bq[4];
            ldmatrix_x4(bq, &W.W2[nt2 * 16 + lr_n][kk * 16 + lr_k]);
            mma_bf16(z2[2 * nt2], hf, bq);
            mma_bf16(z2[2 * nt2 + 1], hf, bq + 2);
        }
    }
}

// Guesses of `nsamp` states: a warp takes 32 samples, one per lane for the features
// and the result, as two 16-row tiles.  Layer 1 is evaluated in the registers that
// layer 2's tensor-core products take it from.
//
// Bound by the SM's special-function unit (two evaluations per SiLU, 256 per sample).
// Staged through shared memory with one thread per sample, layer 1's stores fell
// on one bank 32 at a time: 2^22 guesses took 1.5 ms, 0.35 ms here.
constexpr int NET_GUESS_THREADS = 256;

__global__ void __launch_bounds__(NET_GUESS_THREADS, 2) k_net_guess(const NetTileArgs a)
{
    __shared__ NetW W;
    net_load_weights(W, a.P, a.W2b);
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
    const long long warp = ((long long)blockIdx.x * NET_GUESS_THREADS + threadIdx.x) >> 5;
    const long long nwarps = (long long)gridDim.x * (NET_GUESS_THREADS / 32);
    for (long long s0 = warp * 32; s0 < a.nsamp; s0 += nwarps * 32) {
        const long long gs = s0 + lane;
        double v[5] = {1.0, 0.0, 0.0, 0.0, 1.0};
        if (gs < a.nsamp)
#pragma unroll
            for (int c = 0; c < 5; ++c) v[c] = a.cons[c * a.count + gs];
        const NetSample sm = net_sample(v, a.sc);
        float y = 0.0f;
#pragma unroll 1
        for (int mt = 0; mt < 2; ++mt) {
            float x[2][3];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int src = 16 * mt + 8 * r + g;
                x[r][0] = __shfl_sync(0xffffffffu, sm.x0, src);
                x[r][1] = __shfl_sync(0xffffffffu, sm.x1, src);
                x[r][2] = __shfl_sync(0xffffffffu, sm.x2, src);
            }
            float z2[8][4];
            net_forward(W, x, z2, lane);
            float ya = 0.0f, yb = 0.0f;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                const float2 w3 = *reinterpret_cast<const float2 *>(&W.W3[nt * 8 + 2 * tq]);
                ya = fmaf(w3.x, silu(z2[nt][0]), ya);
                ya = fmaf(w3.y, silu(z2[nt][1]), ya);
                yb = fmaf(w3.x, silu(z2[nt][2]), yb);
                yb = fmaf(w3.y, silu(z2[nt][3]), yb);
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                ya += __shfl_xor_sync(0xffffffffu, ya, o);
                yb += __shfl_xor_sync(0xffffffffu, yb, o);
            }
            // row r of the tile sits in the lanes g = r (mod 8): back to the sample's lane
            const float ra = __shfl_sync(0xffffffffu, ya, 4 * (lane & 7));
            const float rb = __shfl_sync(0xffffffffu, yb, 4 * (lane & 7));
            if ((lane >> 4) == mt) y = ((lane & 8) ? rb : ra) + W.b3;
        }
        if (gs < a.nsamp) {
            float pg = sm.E * exp10f(y * a.sc[5] + a.sc[4]);
            pg = fminf(fmaxf(pg, fmaxf(sm.smag - sm.E, 0.0f)), (a.gamma - 1.0f) * sm.tau);
            a.guess[gs] = (sm.ok && isfinite(pg)) ? f32_to_f64(pg) : -1.0;
        }
    }
}

// ---------------------------------------------------------------------------
// Training.  A CTA of 16 warps takes a tile of 128 samples: four groups of four warps with
// 32 samples each, a quarter (16) of every layer's columns per warp.  The warps of a group
// exchange BF16 copies of h1 and dz2 and layer 3's products through shared memory (four
// warps per 32 samples shorten the serial chain of a mini-batch, which is what training
// time is made of).  The layer-2 weight gradient dz2^T h1 over the tile is taken by all
// warps from those copies.
//
// The order of every sum is part of the result, and the same in each kind of launch: layer
// 1 as ((w0 x0 + w1 x1) + w2 x2) + b1; layer 2's bias after its products; layer 3 over the
// units of a lane (8 i + 2 tq, + 1) in turn, then over the four lanes; gradients and loss over
// a lane's four samples, the eight lanes by halves (g ^ 1, g ^ 2, g ^ 4), the four groups and
// the tiles in turn; no product is fused with a sum outside the tensor cores.
constexpr int NET_WARPS = 16, NET_THREADS = 32 * NET_WARPS, NET_GROUPS = NET_WARPS / 4, NET_ROWS = 32 * NET_GROUPS;
constexpr int NET_RED = 192 + 64 + 64 + 64 + 2;  // W1, b1, b2, W3, b3, loss
constexpr int NET_YP_LD = 80;                    // (320 bytes: eight rows' 16-byte pieces in different banks)
// CTAs of a one-launch epoch and the parameters each owns (a multiple of 8: 16-byte
// pieces of W2's BF16 rows have one owner)
constexpr int NET_CLUSTER = 16, NET_OWN = (NET_PARTIAL + 8 * NET_CLUSTER - 1) / (8 * NET_CLUSTER) * 8;
static_assert(NET_OWN <= NET_THREADS && NET_OWN * NET_CLUSTER >= NET_PARTIAL, "one parameter per thread");

struct NetTrainSmem {
    NetW W;
    __nv_bfloat16 h1[NET_ROWS][NET_W2_LD], dz2[NET_ROWS][NET_W2_LD];
    float yp[NET_ROWS][NET_YP_LD];    // layer 3's products, [16 quarter + 4 tq + unit of the lane]
    float y[NET_ROWS];
    float red[NET_GROUPS][NET_RED + 2];
    float4 feat[2][NET_ROWS];         // features and target of the tile and of the next one
    double raw[6][NET_ROWS];          // the next tile's conserved values and pressures, loaded ahead
    float recv[NET_CLUSTER][NET_OWN]; // one-launch epochs: every CTA's gradient of the parameters this CTA owns
};

// Barrier of the four warps of a group.
__device__ __forceinline__ void net_group_sync(int group)
{
    asm volatile("bar.sync %0, 128;" ::"r"(group + 1) : "memory");
}

// Sums over the eight row groups g of 8 values per lane, halving the values as the lanes pair
// up (g ^ 1, then g ^ 2, g ^ 4); the lane ends with the sum of value `idx`.
__device__ __forceinline__ float net_reduce8(float v[8], int lane, int &idx)
{
#pragma unroll
    for (int n = 4, o = 4; n >= 1; n >>= 1, o <<= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = up ? v[n + i] : v[i], send = up ? v[i] : v[n + i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    idx = (lane & 4) + ((lane & 8) >> 2) + ((lane & 16) >> 4);
    return v[0];
}

// Loss and gradient of one tile, written to S.red (the group's row, this warp's columns) and
// gw2 (this warp's part of dW2: rows 16 (warp & 3) + .., columns 16 (warp >> 2) + ..).
// feat: the tile's features and targets.  All warps of the CTA together.
__device__ __forceinline__ void net_tile(NetTrainSmem &S, const float4 *feat, float inv_batch, float gw2[2][4])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tq = lane & 3;
    const int group = warp >> 2, quarter = warp & 3;
    const int r0 = 32 * group, c0 = 16 * quarter;  // the warp's rows r0 .. r0 + 31, columns c0 .. c0 + 15
    float *red = S.red[group];
    // the lane's rows r0 + 8 i + g
    float x[4][3], t[4];
    bool ok[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        // samples past the end and such without finite features or target (D or tau not
        // positive, a pressure below the FP32 range) enter neither the loss nor the gradient
        const float4 f = feat[r0 + 8 * i + g];
        ok[i] = isfinite(f.x) && isfinite(f.y) && isfinite(f.z) && isfinite(f.w);
        x[i][0] = ok[i] ? f.x : 0.0f;
        x[i][1] = ok[i] ? f.y : 0.0f;
        x[i][2] = ok[i] ? f.z : 0.0f;
        t[i] = f.w;
    }
    // Accumulator layout below: [mt][nt][c], row r0 + 16 mt + 8 (c >> 1) + g (the lane's row 2 mt +
    // (c >> 1)), column c0 + 8 nt + 2 tq + (c & 1).
    float ds1[2][2][4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        const int col = c0 + 8 * nt + 2 * tq;
        const float4 w[2] = {S.W.W1b1[col], S.W.W1b1[col + 1]};
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            float h[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 q = w[c & 1];
                const float *xr = x[2 * mt + (c >> 1)];
                const float z = q.x * xr[0] + q.y * xr[1] + q.z * xr[2] + q.w, sg = sigmoid32(z);
                h[c] = z * sg;
                ds1[mt][nt][c] = sg * (1.0f + z * (1.0f - sg));
            }
            *reinterpret_cast<uint32_t *>(&S.h1[r0 + 16 * mt + g][col]) = pack_bf16x2(h[0], h[1]);
            *reinterpret_cast<uint32_t *>(&S.h1[r0 + 16 * mt + 8 + g][col]) = pack_bf16x2(h[2], h[3]);
        }
    }
    net_group_sync(group);
    // layer 2, this warp's columns
    const int a_r = r0 + (lane & 15), a_c = 8 * (lane >> 4);  // A fragments from row-major tiles
    const int lr_n = (lane & 7) + 8 * (lane >> 4), lr_k = 8 * ((lane >> 3) & 1);
    float z2[2][2][4], h2[2][2][4];
#pragma unroll
    for (int i = 0; i < 16; ++i) z2[i >> 3][(i >> 2) & 1][i & 3] = 0.0f;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        uint32_t af[4], bq[4];
        ldmatrix_x4(bq, &S.W.W2[c0 + lr_n][kk * 16 + lr_k]);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            ldmatrix_x4(af, &S.h1[a_r + 16 * mt][16 * kk + a_c]);
            mma_bf16(z2[mt][0], af, bq);
            mma_bf16(z2[mt][1], af, bq + 2);
        }
    }
    // layer 3: the products W3 silu(z2 + b2), then y = their sum + b3 for one of the lane's rows
    float w3[2][2];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        const float2 b = *reinterpret_cast<const float2 *>(&S.W.b2[c0 + nt * 8 + 2 * tq]);
        const float2 w = *reinterpret_cast<const float2 *>(&S.W.W3[c0 + nt * 8 + 2 * tq]);
        w3[nt][0] = w.x;
        w3[nt][1] = w.y;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float z = z2[mt][nt][c] + ((c & 1) ? b.y : b.x), sg = sigmoid32(z);
                h2[mt][nt][c] = z * sg;
                z2[mt][nt][c] = sg * (1.0f + z * (1.0f - sg));  // silu'(z2)
            }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float(*h)[4] = h2[i >> 1];
        const int c = 2 * (i & 1);
        *reinterpret_cast<float4 *>(&S.yp[r0 + 8 * i + g][16 * quarter + 4 * tq]) =
            make_float4(w3[0][0] * h[0][c], w3[0][1] * h[0][c + 1], w3[1][0] * h[1][c], w3[1][1] * h[1][c + 1]);
    }
    net_group_sync(group);
    {
        const int row = r0 + 8 * quarter + g;
        float v = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 p = *reinterpret_cast<const float4 *>(&S.yp[row][16 * q + 4 * tq]);
            v = v + p.x + p.y + p.z + p.w;
        }
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (tq == 0) S.y[row] = v + S.W.b3;
    }
    net_group_sync(group);
    float dy[4], loss = 0.0f, db3 = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float d = ok[i] ? S.y[r0 + 8 * i + g] - t[i] : 0.0f;
        dy[i] = 2.0f * d * inv_batch;
        loss += d * d;
        db3 += dy[i];
    }
    // dW3 = sum dy h2, db2 = sum dz2, dz2 = dy W3 silu'(z2): values 2 nt + e and 4 + 2 nt + e
    float p3[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) p3[i] = 0.0f;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            float dz[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float d = dy[2 * mt + (c >> 1)];
                dz[c] = d * w3[nt][c & 1] * z2[mt][nt][c];
                p3[2 * nt + (c & 1)] += d * h2[mt][nt][c];
                p3[4 + 2 * nt + (c & 1)] += dz[c];
            }
            const int col = c0 + 8 * nt + 2 * tq;
            *reinterpret_cast<uint32_t *>(&S.dz2[r0 + 16 * mt + g][col]) = pack_bf16x2(dz[0], dz[1]);
            *reinterpret_cast<uint32_t *>(&S.dz2[r0 + 16 * mt + 8 + g][col]) = pack_bf16x2(dz[2], dz[3]);
        }
    __syncthreads();
    // dh1 = dz2 W2, dz1 = dh1 silu'(z1), this warp's hidden units
    float hacc[2][2][4];
#pragma unroll
    for (int i = 0; i < 16; ++i) hacc[i >> 3][(i >> 2) & 1][i & 3] = 0.0f;
    const int t_k = (lane & 7) + 8 * ((lane >> 3) & 1), t_n = 8 * (lane >> 4);  // B fragments, transposed loads
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        uint32_t af[4], bq[4];
        ldmatrix_x4_trans(bq, &S.W.W2[kk * 16 + t_k][c0 + t_n]);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            ldmatrix_x4(af, &S.dz2[a_r + 16 * mt][16 * kk + a_c]);
            mma_bf16(hacc[mt][0], af, bq);
            mma_bf16(hacc[mt][1], af, bq + 2);
        }
    }
    // dW2 over the whole tile
    {
        const int j0 = 16 * (warp & 3), i0 = 16 * (warp >> 2);
        const int a_s = (lane & 7) + 8 * (lane >> 4), a_j = 8 * ((lane >> 3) & 1);
#pragma unroll
        for (int i = 0; i < 8; ++i) gw2[i >> 2][i & 3] = 0.0f;
#pragma unroll
        for (int kk = 0; kk < NET_ROWS / 16; ++kk) {
            uint32_t af[4], bq[4];
            ldmatrix_x4_trans(af, &S.dz2[16 * kk + a_s][j0 + a_j]);
            ldmatrix_x4_trans(bq, &S.h1[16 * kk + t_k][i0 + t_n]);
            mma_bf16(gw2[0], af, bq);
            mma_bf16(gw2[1], af, bq + 2);
        }
    }
    // db1 = sum dz1, dW1 = sum dz1 x
    float pa[8], pb[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) pa[i] = pb[i] = 0.0f;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int i = 2 * nt + (c & 1);
                const float dz = hacc[mt][nt][c] * ds1[mt][nt][c], *xr = x[2 * mt + (c >> 1)];
                pa[i] += dz;
                pa[4 + i] += dz * xr[0];
                pb[i] += dz * xr[1];
                pb[4 + i] += dz * xr[2];
            }
    int idx;
    const float s3 = net_reduce8(p3, lane, idx), sa = net_reduce8(pa, lane, idx), sb = net_reduce8(pb, lane, idx);
    const int col = c0 + 8 * ((idx >> 1) & 1) + 2 * tq + (idx & 1);
    red[(idx < 4 ? 320 : 256) + col] = s3;
    if (idx < 4) red[192 + col] = sa;
    else red[3 * col] = sa;
    red[3 * col + (idx < 4 ? 1 : 2)] = sb;
    if (quarter == 0) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            loss += __shfl_xor_sync(0xffffffffu, loss, o);
            db3 += __shfl_xor_sync(0xffffffffu, db3, o);
        }
        if (lane == 0) {
            red[384] = db3;
            red[385] = loss;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// The conserved values and pressures of tile tl on their way into S.raw.
__device__ __forceinline__ void net_load_raw(NetTrainSmem &S, const NetTileArgs &a, long long base, long long nsamp,
                                             long long tl)
{
    for (int i = threadIdx.x; i < 6 * NET_ROWS; i += NET_THREADS) {
        const int v = i / NET_ROWS, r = i % NET_ROWS;
        const long long s = tl * NET_ROWS + r;
        if (s >= nsamp) continue;
        const double *src = (v < 5 ? a.cons + v * a.count : a.p) + base + s;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&S.raw[v][r]);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
    }
}

__device__ __forceinline__ void net_wait_raw() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Features and targets of the tile in S.raw: four warps for each, one sample per thread.
__device__ __forceinline__ void net_store_feature(const NetTrainSmem &S, float4 *feat, long long nsamp, long long tl,
                                                  const float sc[6])
{
    const int q = threadIdx.x / NET_ROWS, r = threadIdx.x % NET_ROWS;
    float f = __int_as_float(0x7fc00000);  // past the end: not a sample
    if (tl * NET_ROWS + r < nsamp) {
        const float D = f64_to_f32(S.raw[0][r]), tau = f64_to_f32(S.raw[4][r]);
        if (q == 0) {
            f = net_x0(tau, D, sc);
        } else if (q == 1) {
            const float Sx = f64_to_f32(S.raw[1][r]), Sy = f64_to_f32(S.raw[2][r]), Sz = f64_to_f32(S.raw[3][r]);
            f = net_x1(sqrtf(Sx * Sx + Sy * Sy + Sz * Sz), tau + D);
        } else if (q == 2) {
            f = net_x2(D, sc);
        } else {
            f = (log10f(f64_to_f32(S.raw[5][r]) / (tau + D)) - sc[4]) / sc[5];
        }
    }
    reinterpret_cast<float *>(&feat[r])[q] = f;
}

// The features of a CTA's first tile.
__device__ __forceinline__ void net_first_tile(NetTrainSmem &S, const NetTileArgs &a, int buf, long long base,
                                               long long nsamp, long long tl)
{
    net_load_raw(S, a, base, nsamp, tl);
    net_wait_raw();
    __syncthreads();
    net_store_feature(S, S.feat[buf], nsamp, tl, a.sc);
    __syncthreads();
}

// The gradient and loss of tile tl of `nsamp` samples from sample `base` on, the four groups'
// sums added in order: put2(k, v0, v1) receives the pairs of dW2, put(k, v) the other
// parameters and the loss sum (k = NET_PARAMS).  S.feat[buf] holds the tile's features on
// entry; on return (after the CTA's next barrier) S.feat[buf] those of tile ntl of the
// nnsamp samples from nbase on.
template <class Put2, class Put>
__device__ __forceinline__ void net_cta_grad(NetTrainSmem &S, const NetTileArgs &a, int &buf, long long nbase,
                                             long long nnsamp, long long ntl, float inv_batch, Put2 put2, Put put)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, tq = lane & 3;
    float gw2[2][4];
    net_load_raw(S, a, nbase, nnsamp, ntl);
    net_tile(S, S.feat[buf], inv_batch, gw2);  // (its last barrier also ends the loads)
    buf ^= 1;
    net_store_feature(S, S.feat[buf], nnsamp, ntl, a.sc);
    const int j = 16 * (warp & 3) + g, i = 16 * (warp >> 2) + 2 * tq;
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        put2(OFF_W2 + j * 64 + i + 8 * n, gw2[n][0], gw2[n][1]);
        put2(OFF_W2 + (j + 8) * 64 + i + 8 * n, gw2[n][2], gw2[n][3]);
    }
    if (threadIdx.x < NET_RED) {
        const int k = threadIdx.x;
        const float v = S.red[0][k] + S.red[1][k] + S.red[2][k] + S.red[3][k];
        put(k < 192 ? OFF_W1 + k : k < 256 ? OFF_B1 + k - 192 : k < 320 ? OFF_B2 + k - 256 : k < 384 ? OFF_W3 + k - 320
            : k == 384 ? OFF_B3 : NET_PARAMS, v);
    }
}
static_assert(NET_GROUPS == 4, "the sum over groups");
static_assert(NET_RED <= NET_THREADS && NET_THREADS == 4 * NET_ROWS, "one thread per sum; four per sample");

// One mini-batch's gradients, tile by tile into its rows of a.partial (batches of many tiles).
__global__ void __launch_bounds__(NET_THREADS, 1) k_net_grad(const NetTileArgs a)
{
    extern __shared__ __align__(16) unsigned char net_smem_raw[];
    NetTrainSmem &S = *reinterpret_cast<NetTrainSmem *>(net_smem_raw);  // (up to recv)
    net_load_weights(S.W, a.P, a.W2b);
    net_first_tile(S, a, 0, a.first, a.nsamp, blockIdx.x);
    int buf = 0;
    for (long long tl = blockIdx.x; tl * NET_ROWS < a.nsamp; tl += gridDim.x) {
        float *out = a.partial + tl * NET_PARTIAL;
        net_cta_grad(
            S, a, buf, a.first, a.nsamp, tl + gridDim.x, a.inv_batch,
            [out](int k, float v0, float v1) { *reinterpret_cast<float2 *>(out + k) = make_float2(v0, v1); },
            [out](int k, float v) { out[k] = v; });
        __syncthreads();
    }
}

// One Adam step (Kingma & Ba) of a parameter; bc1, bc2 the bias corrections.
__device__ __forceinline__ float net_adam(float p, float &m, float &v, float grad, float lr, float bc1, float bc2)
{
    m = 0.9f * m + 0.1f * grad;
    v = 0.999f * v + 0.001f * grad * grad;
    return p - lr * (m / bc1) / (sqrtf(v / bc2) + 1e-8f);
}

// Sum the tiles' gradients in order, 64 tiles at a time: eight threads per parameter load
// them, one adds them up while the next 64 are on their way.  Optionally one Adam step, which
// also refreshes the BF16 copy of W2.
constexpr int NET_SLICES = 8, NET_AHEAD = 8;

__global__ void __launch_bounds__(32 * NET_SLICES) k_net_reduce(const float *partial, long long tiles, float *grad,
                                                                float *P, float *m, float *v, __nv_bfloat16 *W2b,
                                                                float lr, float bc1, float bc2, int adam,
                                                                float *loss_acc, float loss_scale)
{
    constexpr int ROWS = NET_SLICES * NET_AHEAD;
    __shared__ float sq[2][ROWS][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    float q[NET_AHEAD], s = 0.0f;
    auto load = [&](long long b) {
#pragma unroll
        for (int i = 0; i < NET_AHEAD; ++i) {
            const long long r = b + sl + NET_SLICES * i;
            q[i] = k <= NET_PARAMS && r < tiles ? partial[r * NET_PARTIAL + k] : 0.0f;
        }
    };
    load(0);
    int buf = 0;
    for (long long b = 0; b < tiles; b += ROWS, buf ^= 1) {
#pragma unroll
        for (int i = 0; i < NET_AHEAD; ++i) sq[buf][sl + NET_SLICES * i][lane] = q[i];
        __syncthreads();  // (also: the sum two rounds back, of the same buffer, is done)
        load(b + ROWS);
        if (sl == 0) {
            const int n = tiles - b < ROWS ? (int)(tiles - b) : ROWS;
#pragma unroll 16
            for (int r = 0; r < n; ++r) s += sq[buf][r][lane];
        }
    }
    if (sl != 0 || k > NET_PARAMS) return;
    if (k == NET_PARAMS) {
        if (loss_acc) *loss_acc += s * loss_scale;
        return;
    }
    if (grad) grad[k] = s;
    if (!adam) return;
    float mk = m[k], vk = v[k];
    const float pk = net_adam(P[k], mk, vk, s, lr, bc1, bc2);
    m[k] = mk;
    v[k] = vk;
    P[k] = pk;
    if (k >= OFF_W2 && k < OFF_W2 + 4096) W2b[k - OFF_W2] = __float2bfloat16_rn(pk);
}

// An epoch (or NET_LAUNCH_BATCHES mini-batches of it) in one launch, by one cluster of CTAs
// that keep the weights in shared memory: per mini-batch CTA r takes tile r and writes its
// gradient into the owners' shared memory (CTA r owns the parameters [r NET_OWN, (r + 1)
// NET_OWN)), a cluster barrier, every owner sums its parameters' gradients in the order of the
// tiles, takes the Adam step and writes the new values into every CTA's copy of the weights,
// a second barrier.
//
// Bound by the serial chain of a mini-batch (a tile's forward and backward, two
// barriers and the exchange).  Launched per mini-batch, the same work is two launches
// that use a fraction of the chip for a few microseconds each: 14.5 us per mini-batch
// of 4096 against 8.2 us here for 2048 (39 us before both).
constexpr int NET_LAUNCH_BATCHES = 448;  // mini-batches of a launch, so that its arguments stay below 4 KB

struct NetEpochArgs {
    NetTileArgs a;
    float *P, *m, *v;
    int batch;
    long long begin, end;  // the samples of this launch (begin a multiple of batch)
    float lr;
    float *loss;           // the epoch's mean loss, added to, or nullptr
    float loss_scale;
    float2 bc[NET_LAUNCH_BATCHES];  // Adam's bias corrections of every mini-batch
};

__global__ void __launch_bounds__(NET_THREADS, 1) k_net_epoch(const __grid_constant__ NetEpochArgs e)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char net_smem_raw[];
    NetTrainSmem &S = *reinterpret_cast<NetTrainSmem *>(net_smem_raw);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const NetTileArgs &a = e.a;
    net_load_weights(S.W, e.P, a.W2b);
    // the parameter this thread owns, with its Adam moments (the loss counts as one)
    const int k = threadIdx.x < NET_OWN && rank * NET_OWN + (int)threadIdx.x < NET_PARTIAL ? rank * NET_OWN + threadIdx.x : -1;
    const bool par = k >= 0 && k < NET_PARAMS;
    float pk = par ? e.P[k] : 0.0f, mk = par ? e.m[k] : 0.0f, vk = par ? e.v[k] : 0.0f;
    float loss = k == NET_PARAMS && e.loss ? *e.loss : 0.0f;
    net_first_tile(S, a, 0, e.begin, e.end - e.begin < e.batch ? e.end - e.begin : e.batch, rank);
    cl.sync();  // (every CTA of the cluster runs before its shared memory is written)
    int buf = 0, mb = 0;
    for (long long base = e.begin; base < e.end; base += e.batch, ++mb) {
        const long long ns = e.end - base < e.batch ? e.end - base : e.batch;
        const long long nb = base + e.batch, left = e.end - nb;
        const int tiles = (int)((ns + NET_ROWS - 1) / NET_ROWS);  // CTA r takes tile r, if there is one
        if (rank < tiles)
            net_cta_grad(
                S, a, buf, left > 0 ? nb : 0, left > e.batch ? e.batch : left > 0 ? left : 0, rank, 1.0f / (float)ns,
                [&](int q, float v0, float v1) {
                    float *d = cl.map_shared_rank(&S.recv[rank][q % NET_OWN], q / NET_OWN);
                    *reinterpret_cast<float2 *>(d) = make_float2(v0, v1);
                },
                [&](int q, float v) { *cl.map_shared_rank(&S.recv[rank][q % NET_OWN], q / NET_OWN) = v; });
        cl.sync();
        if (k >= 0) {
            float s = 0.0f;
            if (tiles == NET_CLUSTER) {
#pragma unroll
                for (int r = 0; r < NET_CLUSTER; ++r) s += S.recv[r][threadIdx.x];
            } else {
                for (int r = 0; r < tiles; ++r) s += S.recv[r][threadIdx.x];
            }
            if (k == NET_PARAMS) {
                loss += s * e.loss_scale;
            } else {
                pk = net_adam(pk, mk, vk, s, e.lr, e.bc[mb].x, e.bc[mb].y);
                if (k < OFF_B1) reinterpret_cast<float *>(&S.W.W1b1[k / 3])[k % 3] = pk;
                else if (k < OFF_W2) S.W.W1b1[k - OFF_B1].w = pk;
                else if (k < OFF_B2) S.W.W2[(k - OFF_W2) / 64][(k - OFF_W2) % 64] = __float2bfloat16_rn(pk);
                else if (k < OFF_W3) S.W.b2[k - OFF_B2] = pk;
                else if (k < OFF_B3) S.W.W3[k - OFF_W3] = pk;
                else S.W.b3 = pk;
            }
        }
        __syncthreads();
        // the owned part of the weights, updated in this CTA's copy, to the other CTAs in
        // 16-byte pieces: W2's (8 parameters each), then W1 and b1 (rank 0), b2, W3 and b3
        // (contiguous, the rank that owns them)
        {
            const int k0 = rank * NET_OWN, k1 = k0 + NET_OWN;
            const int w0 = k0 > OFF_W2 ? k0 : OFF_W2, w1 = k1 < OFF_B2 ? k1 : OFF_B2;
            const int nw = w1 > w0 ? (w1 - w0) / 8 : 0;
            const bool head = rank == 0, tail = rank == NET_CLUSTER - 1;
            static_assert(OFF_W2 <= NET_OWN && OFF_B2 >= (NET_CLUSTER - 1) * NET_OWN, "W1, b1 and b2, W3, b3 have one owner");
            const int pieces = nw + (head ? 64 : 0) + (tail ? 33 : 0);
            for (int i = threadIdx.x; i < pieces * NET_CLUSTER; i += NET_THREADS) {
                const int r = i / pieces, c = i - r * pieces;
                if (r == rank) continue;
                float4 *src;
                if (c < nw) {
                    const int q = w0 + 8 * c - OFF_W2;
                    src = reinterpret_cast<float4 *>(&S.W.W2[q / 64][q % 64]);
                } else if (head) {
                    src = &S.W.W1b1[c - nw];
                } else {
                    src = reinterpret_cast<float4 *>(S.W.b2) + (c - nw);
                }
                *cl.map_shared_rank(src, r) = *src;
            }
        }
        cl.sync();
    }
    if (par) {
        e.P[k] = pk;
        e.m[k] = mk;
        e.v[k] = vk;
    } else if (k == NET_PARAMS && e.loss) {
        *e.loss = loss;
    }
}

__global__ void k_net_bf16(const float *P, __nv_bfloat16 *W2b)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < 4096) W2b[k] = __float2bfloat16_rn(P[OFF_W2 + k]);
}

// The shared-memory image of the weights for in-kernel inference (NetWeightsSmem)
// from the FP32 parameters: W2 in BF16 with padded rows; W1, b1, W2, b2 halved.
__global__ void k_net_image(const float *P, NetWeightsSmem *img)
{
    for (int k = threadIdx.x; k < 64 * NET_W2_LD; k += blockDim.x) {
        const int j = k / NET_W2_LD, i = k % NET_W2_LD;
        img->W2h[j][i] = __float2bfloat16_rn(i < 64 ? 0.5f * P[OFF_W2 + j * 64 + i] : 0.0f);
    }
    for (int j = threadIdx.x; j < 64; j += blockDim.x) {
        img->W1b1h[j] = make_float4(__uint_as_float(to_tf32(0.5f * P[OFF_W1 + 3 * j])),
                                    __uint_as_float(to_tf32(0.5f * P[OFF_W1 + 3 * j + 1])),
                                    __uint_as_float(to_tf32(0.5f * P[OFF_W1 + 3 * j + 2])),
                                    __uint_as_float(to_tf32(0.5f * P[OFF_B1 + j])));
        img->b2h[j] = 0.5f * P[OFF_B2 + j];
        img->W3[j] = P[OFF_W3 + j];
    }
    if (threadIdx.x == 0) {
        img->b3 = P[OFF_B3];
        img->pad[0] = img->pad[1] = img->pad[2] = 0.0f;
    }
}

}  // namespace dg

// ---------------------------------------------------------------------------

struct dg_c2p_net {
    int device;
    float *P, *m, *v, *grad, *partial;
    __nv_bfloat16 *W2b;
    dg::NetWeightsSmem *img;  // weights for in-kernel inference
    long long partial_blocks;
    long long step;
    float sc[6];
};

namespace dg {

dg_status set_error(dg_status st, const char *msg);

namespace {

long long net_tiles(long long nsamp) { return (nsamp + NET_ROWS - 1) / NET_ROWS; }

// Largest mini-batch an epoch runs in one cluster: a tile of 128 samples per CTA, 8.2 us a
// mini-batch of 2048.  (A mini-batch of 4096 in two launches takes 14.5 us; in one cluster, two
// tiles per CTA, it took the same.)
constexpr int kClusterBatch = NET_CLUSTER * NET_ROWS;

NetTileArgs net_args(const dg_c2p_net *n, const double *cons, const double *p, long long count)
{
    NetTileArgs a;
    std::memset(&a, 0, sizeof(a));
    a.P = n->P;
    a.W2b = n->W2b;
    a.cons = cons;
    a.p = p;
    a.partial = n->partial;
    a.count = count;
    for (int i = 0; i < 6; ++i) a.sc[i] = n->sc[i];
    return a;
}

cudaError_t launch_net_grad(const dg_c2p_net *n, const double *cons, const double *p, long long count, long long first,
                            long long nsamp, cudaStream_t s)
{
    NetTileArgs a = net_args(n, cons, p, count);
    a.first = first;
    a.nsamp = nsamp;
    a.inv_batch = 1.0f / (float)nsamp;
    constexpr size_t smem = offsetof(NetTrainSmem, recv);
    const cudaError_t e = cudaFuncSetAttribute(k_net_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long tiles = net_tiles(nsamp);
    k_net_grad<<<(unsigned)(tiles < kNumSMs ? tiles : kNumSMs), NET_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

// Launch configuration of k_net_epoch (one cluster).
struct EpochLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    explicit EpochLaunch(cudaStream_t s)
    {
        cfg.gridDim = dim3(NET_CLUSTER);
        cfg.blockDim = dim3(NET_THREADS);
        cfg.dynamicSmemBytes = sizeof(NetTrainSmem);
        cfg.stream = s;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = NET_CLUSTER;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};

// Whether the device (or the part of it this context has) can hold the cluster.
bool net_cluster_fits()
{
    if (cudaFuncSetAttribute(k_net_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NetTrainSmem)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_net_epoch, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    EpochLaunch l(nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_net_epoch, &l.cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

// Adam's bias corrections of step `step`, on the host for both training paths: 1 - powf(0.999f, 1)
// multiplies a rounding error of powf by a thousand, and the device's powf is another function.
float2 net_bias(long long step)
{
    return make_float2(1.0f - powf(0.9f, (float)step), 1.0f - powf(0.999f, (float)step));
}

// The samples [begin, end) of an epoch, at most NET_LAUNCH_BATCHES mini-batches.
cudaError_t launch_net_epoch(const dg_c2p_net *n, const double *cons, const double *p, long long count, long long begin,
                             long long end, int batch, float lr, float *loss, cudaStream_t s)
{
    NetEpochArgs e;
    std::memset(&e, 0, sizeof(e));
    e.a = net_args(n, cons, p, count);
    e.P = n->P;
    e.m = n->m;
    e.v = n->v;
    e.batch = batch;
    e.begin = begin;
    e.end = end;
    for (long long b = 0; begin + b * batch < end; ++b) e.bc[b] = net_bias(n->step + 1 + b);
    e.lr = lr;
    e.loss = loss;
    e.loss_scale = 1.0f / (float)count;
    EpochLaunch l(s);
    const cudaError_t r = cudaLaunchKernelEx(&l.cfg, k_net_epoch, e);
    return r == cudaSuccess ? cudaGetLastError() : r;
}

}  // namespace

}  // namespace dg

namespace dg {

void net_device_view(const dg_c2p_net *n, const void **img, float sc[6])
{
    *img = n->img;
    for (int i = 0; i < 6; ++i) sc[i] = n->sc[i];
}

}  // namespace dg

using namespace dg;

#define NET_CUDA(expr)                                                                                   \
    do {                                                                                                 \
        cudaError_t e_ = (expr);                                                                         \
        if (e_ != cudaSuccess) return set_error(DG_ERR_CUDA, cudaGetErrorString(e_));                    \
    } while (0)

extern "C" {

dg_status dg_c2p_net_create(const float *params, const double *scales, dg_c2p_net **out)
{
    if (!params || !scales || !out) return set_error(DG_ERR_ARG, "params, scales and out must not be NULL");
    *out = nullptr;
    if (!(scales[1] > scales[0]) || !(scales[3] > scales[2]) || !(scales[5] != 0.0))
        return set_error(DG_ERR_ARG, "invalid feature scales");
    dg_c2p_net *n = new dg_c2p_net;
    std::memset(n, 0, sizeof(*n));
    cudaGetDevice(&n->device);
    for (int i = 0; i < 6; ++i) n->sc[i] = (float)scales[i];
    cudaError_t e = cudaSuccess;
    e = e ? e : cudaMalloc(&n->P, sizeof(float) * NET_PARAMS);
    e = e ? e : cudaMalloc(&n->m, sizeof(float) * NET_PARAMS);
    e = e ? e : cudaMalloc(&n->v, sizeof(float) * NET_PARAMS);
    e = e ? e : cudaMalloc(&n->grad, sizeof(float) * NET_PARAMS);
    e = e ? e : cudaMalloc(&n->W2b, sizeof(__nv_bfloat16) * 4096);
    e = e ? e : cudaMalloc(&n->img, sizeof(NetWeightsSmem));
    if (e == cudaSuccess) e = cudaMemcpy(n->P, params, sizeof(float) * NET_PARAMS, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, sizeof(float) * NET_PARAMS);
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, sizeof(float) * NET_PARAMS);
    if (e == cudaSuccess) {
        k_net_bf16<<<16, 256>>>(n->P, n->W2b);
        k_net_image<<<1, 256>>>(n->P, n->img);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) {
        dg_c2p_net_destroy(n);
        return set_error(e == cudaErrorMemoryAllocation ? DG_ERR_NOMEM : DG_ERR_CUDA, cudaGetErrorString(e));
    }
    *out = n;
    return DG_OK;
}

void dg_c2p_net_destroy(dg_c2p_net *n)
{
    if (!n) return;
    cudaDeviceSynchronize();
    cudaFree(n->P);
    cudaFree(n->m);
    cudaFree(n->v);
    cudaFree(n->grad);
    cudaFree(n->partial);
    cudaFree(n->W2b);
    cudaFree(n->img);
    delete n;
}

dg_status dg_c2p_net_get_params(const dg_c2p_net *n, float *params)
{
    if (!n || !params) return set_error(DG_ERR_ARG, "net and params must not be NULL");
    NET_CUDA(cudaDeviceSynchronize());
    NET_CUDA(cudaMemcpy(params, n->P, sizeof(float) * NET_PARAMS, cudaMemcpyDeviceToHost));
    return DG_OK;
}

dg_status dg_c2p_net_guess(dg_c2p_net *n, long long count, double gamma, const double *cons, double *p_guess,
                           void *stream)
{
    if (!n || count < 0) return set_error(DG_ERR_ARG, "net must not be NULL and count >= 0");
    if (count == 0) return DG_OK;
    if (!cons || !p_guess) return set_error(DG_ERR_ARG, "cons and p_guess must not be NULL");
    NetTileArgs a = net_args(n, cons, nullptr, count);
    a.guess = p_guess;
    a.nsamp = count;
    a.gamma = (float)gamma;
    const long long blocks = (count + NET_GUESS_THREADS - 1) / NET_GUESS_THREADS;
    k_net_guess<<<(unsigned)(blocks < 2 * kNumSMs ? blocks : 2 * kNumSMs), NET_GUESS_THREADS, 0, (cudaStream_t)stream>>>(a);
    NET_CUDA(cudaGetLastError());
    return DG_OK;
}

static dg_status ensure_partial(dg_c2p_net *n, long long blocks)
{
    if (blocks <= n->partial_blocks) return DG_OK;
    cudaFree(n->partial);
    n->partial = nullptr;
    NET_CUDA(cudaMalloc(&n->partial, sizeof(float) * NET_PARTIAL * blocks));
    n->partial_blocks = blocks;
    return DG_OK;
}

dg_status dg_c2p_net_grad(dg_c2p_net *n, long long count, const double *cons, const double *p, float *grad,
                          float *loss, void *stream)
{
    if (!n || count <= 0 || !cons || !p || !grad || !loss)
        return set_error(DG_ERR_ARG, "net, cons, p, grad, loss must not be NULL and count > 0");
    const long long tiles = net_tiles(count);
    if (dg_status st = ensure_partial(n, tiles)) return st;
    cudaStream_t s = (cudaStream_t)stream;
    NET_CUDA(cudaMemsetAsync(loss, 0, sizeof(float), s));
    NET_CUDA(launch_net_grad(n, cons, p, count, 0, count, s));
    k_net_reduce<<<(NET_PARTIAL + 31) / 32, 32 * NET_SLICES, 0, s>>>(n->partial, tiles, grad, n->P, n->m, n->v, n->W2b,
                                                                      0.0f, 1.0f, 1.0f, 0, loss, 1.0f / (float)count);
    NET_CUDA(cudaGetLastError());
    return DG_OK;
}

dg_status dg_c2p_net_train(dg_c2p_net *n, long long count, const double *cons, const double *p, int epochs,
                           int batch, float lr, float *loss_per_epoch, void *stream)
{
    if (!n || count <= 0 || !cons || !p || epochs <= 0 || batch <= 0 || !(lr > 0.0f))
        return set_error(DG_ERR_ARG, "invalid training arguments");
    cudaStream_t s = (cudaStream_t)stream;
    const long long nb = (count + batch - 1) / batch;
    const bool cluster = batch <= kClusterBatch && net_cluster_fits();
    if (!cluster)
        if (dg_status st = ensure_partial(n, net_tiles(batch))) return st;
    if (loss_per_epoch) NET_CUDA(cudaMemsetAsync(loss_per_epoch, 0, sizeof(float) * epochs, s));
    for (int ep = 0; ep < epochs; ++ep) {
        float *loss = loss_per_epoch ? loss_per_epoch + ep : nullptr;
        if (cluster) {
            for (long long b = 0; b < nb; b += NET_LAUNCH_BATCHES) {
                const long long m = nb - b < NET_LAUNCH_BATCHES ? nb - b : NET_LAUNCH_BATCHES;
                const long long end = b + m == nb ? count : (b + m) * batch;
                NET_CUDA(launch_net_epoch(n, cons, p, count, b * batch, end, batch, lr, loss, s));
                n->step += m;
                k_net_bf16<<<16, 256, 0, s>>>(n->P, n->W2b);
                NET_CUDA(cudaGetLastError());
            }
            continue;
        }
        for (long long b = 0; b < nb; ++b) {
            const long long first = b * batch;
            const long long ns = (first + batch <= count) ? batch : count - first;
            NET_CUDA(launch_net_grad(n, cons, p, count, first, ns, s));
            n->step += 1;
            const float2 bc = net_bias(n->step);
            k_net_reduce<<<(NET_PARTIAL + 31) / 32, 32 * NET_SLICES, 0, s>>>(n->partial, net_tiles(ns), nullptr, n->P, n->m, n->v,
                                                                              n->W2b, lr, bc.x, bc.y, 1, loss,
                                                                              1.0f / (float)count);
            NET_CUDA(cudaGetLastError());
        }
    }
    k_net_image<<<1, 256, 0, s>>>(n->P, n->img);
    NET_CUDA(cudaGetLastError());
    return DG_OK;
}

}  // extern "C"
