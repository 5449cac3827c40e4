// dg_mlp.cuh -- learned viscosity sensor: a per-cell network
//   y = W3 . gelu(W2 gelu(W1 x + b1) + b2) + b3,   gelu(z) = z/2 (1 + erf(z/sqrt 2))
// predicting y = log(nu / (cs h/p)) from x = (rho_l/rho_0, |v|hat_l/cs), the
// normalised modal coefficients of the cell (D = 2b inputs, 64 hidden units).
// Training runs in FP32 on the CUDA cores (forward, backward and the gradient sums
// of a block of samples in one kernel, a reduction in a fixed order, Adam); inference is
// one fused kernel with BF16 tensor-core products and FP32 accumulation, the
// accumulator fragments of a layer feeding the next layer's operand fragments
// directly in registers.
//
// Parameter layout (FP32): W1 [64][D], b1 [64], W2 [64][64], b2 [64], W3 [64], b3.
#pragma once

#include <cuda_bf16.h>

#include "dg_tile.cuh"

namespace dg {

constexpr int MLP_BMAX = 4096;  // largest training batch

struct MlpLayout {
    int D, P, oW1, ob1, oW2, ob2, oW3, ob3;
    __host__ __device__ static constexpr MlpLayout make(int D)
    {
        MlpLayout L{};
        L.D = D;
        L.oW1 = 0;
        L.ob1 = MLP_H * D;
        L.oW2 = L.ob1 + MLP_H;
        L.ob2 = L.oW2 + MLP_H * MLP_H;
        L.oW3 = L.ob2 + MLP_H;
        L.ob3 = L.oW3 + MLP_H;
        L.P = L.ob3 + 1;
        return L;
    }
};

// training work: the gradient sums of every block of MLP_SB samples, [block][P + 1]
// pairs of floats (the last one: the sum of squared errors)
constexpr int MLP_SB = 32;
constexpr size_t mlp_work_floats() { return (size_t)(MLP_BMAX / MLP_SB) * 2 * (MlpLayout::make(40).P + 1); }

__device__ __forceinline__ float gelu_prime_f(float z)
{
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// a sum carried as an unevaluated pair of floats: the rounding error of every
// product (FMA) and of every addition (Knuth's two-sum) goes into the second
// float, so the sum is good to about 2^-46 of its terms.  FP64 sums would be no
// better once rounded to the FP32 gradient, and run at a sixty-fourth of the rate.
struct Pair {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float p, float e)
    {
        const float t = __fadd_rn(s, p), z = __fadd_rn(t, -s);
        const float err = __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -z)), __fadd_rn(p, -z));
        s = t;
        c = __fadd_rn(c, __fadd_rn(err, e));
    }
    __device__ __forceinline__ void add_prod(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        add(p, __fmaf_rn(a, b, -p));
    }
};

// One training pass over MLP_SB samples per block, lane = sample, warp w = hidden
// units 4w .. 4w+3: forward (activations in shared memory, pre-activations in
// registers), backward, and the block's sums of the parameter gradients
//   dz2 = (2 r / n) W3 gelu'(z2),  dz1 = (W2^T dz2) gelu'(z1),
//   dW1 = dz1 x^T, dW2 = dz2 a1^T, dW3 = (2/n) sum r a2.
// The products of a gradient entry are summed as pairs over the block's samples
// and over the blocks (k_mlp_reduce) in a fixed order.
// Bound: instruction issue of the 10-instruction pair products (6.8 thousand per
// sample), with four warps per scheduler in flight; half of the warps sum dW2, the
// others dW1 and the rest.  4096 samples at D = 40: forward, backward and gradients
// took 27 + 44 + 2088 us as separate passes with one thread per sample and one per
// parameter in FP64 over 27 blocks, 29 us here with 8 warps that summed dW2 and dW1 in
// turn, 25 us with 16.
constexpr int MLP_NT = 512, MLP_HW = MLP_H / (MLP_NT / 32);  // threads, hidden units per warp
template <int D>
struct MlpPass {
    static constexpr MlpLayout L = MlpLayout::make(D);
    static constexpr int SP = MLP_SB + 4;  // row stride of the transposed arrays (conflict-free 16-byte loads)
    static constexpr int oX = (L.P + 3) / 4 * 4, oA1 = oX + D * SP, oA2 = oA1 + MLP_H * SP, oD1 = oA2 + MLP_H * SP;
    static constexpr int oD2 = oD1 + MLP_H * SP, oR = oD2 + MLP_H * SP, total = oR + MLP_SB;
    // thread tiles of dW1 [64][D]: TR x TC entries
    static constexpr int TC = D % 5 == 0 ? 5 : 2, CG = D / TC, TR = MLP_H * CG / 256;
    static_assert(D % 4 == 0 && TR * 256 == MLP_H * CG, "tiles cover dW1");
    static_assert(MLP_HW == 4 && L.oW2 % 4 == 0, "a warp's weights of a row are one 16-byte load");
};

template <int D>
__global__ void __launch_bounds__(MLP_NT) k_mlp_pass(const float* __restrict__ W, const float* __restrict__ X,
                                                  const float* __restrict__ Y, int n, float2* __restrict__ part)
{
    using M = MlpPass<D>;
    constexpr MlpLayout L = M::L;
    constexpr int SP = M::SP, HW = MLP_HW;
    extern __shared__ __align__(16) float sm[];
    float* sX = sm + M::oX;
    float* sA1 = sm + M::oA1;
    float* sA2 = sm + M::oA2;
    float* sD1 = sm + M::oD1;
    float* sD2 = sm + M::oD2;
    float* sR = sm + M::oR;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int i0 = blockIdx.x * MLP_SB, ns = min(MLP_SB, n - i0);
    for (int e = tid; e < L.P / 4; e += MLP_NT)
        reinterpret_cast<float4*>(sm)[e] = __ldg(reinterpret_cast<const float4*>(W) + e);
    if (tid < L.P % 4) sm[L.P / 4 * 4 + tid] = W[L.P / 4 * 4 + tid];
    for (int e = tid; e < MLP_SB * D; e += MLP_NT) {
        const int s = e / D, d = e - s * D;
        sX[d * SP + s] = s < ns ? X[(size_t)i0 * D + e] : 0.f;
    }
    __syncthreads();
    float z1[HW], z2[HW];
#pragma unroll
    for (int j = 0; j < HW; ++j) z1[j] = sm[L.ob1 + HW * w + j];
#pragma unroll 2
    for (int d = 0; d < D; d += 4) {
        const float x[4] = {sX[d * SP + lane], sX[(d + 1) * SP + lane], sX[(d + 2) * SP + lane], sX[(d + 3) * SP + lane]};
#pragma unroll
        for (int j = 0; j < HW; ++j) {
            const float4 q = *reinterpret_cast<const float4*>(sm + L.oW1 + (HW * w + j) * D + d);
            z1[j] += q.x * x[0];
            z1[j] += q.y * x[1];
            z1[j] += q.z * x[2];
            z1[j] += q.w * x[3];
        }
    }
#pragma unroll
    for (int j = 0; j < HW; ++j) sA1[(HW * w + j) * SP + lane] = gelu_f(z1[j]);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < HW; ++j) z2[j] = sm[L.ob2 + HW * w + j];
#pragma unroll 2
    for (int k = 0; k < MLP_H; k += 4) {
        const float x[4] = {sA1[k * SP + lane], sA1[(k + 1) * SP + lane], sA1[(k + 2) * SP + lane],
                            sA1[(k + 3) * SP + lane]};
#pragma unroll
        for (int j = 0; j < HW; ++j) {
            const float4 q = *reinterpret_cast<const float4*>(sm + L.oW2 + (HW * w + j) * MLP_H + k);
            z2[j] += q.x * x[0];
            z2[j] += q.y * x[1];
            z2[j] += q.z * x[2];
            z2[j] += q.w * x[3];
        }
    }
#pragma unroll
    for (int j = 0; j < HW; ++j) sA2[(HW * w + j) * SP + lane] = gelu_f(z2[j]);
    __syncthreads();
    if (w == 0) {
        float y = sm[L.ob3];
#pragma unroll 8
        for (int j = 0; j < MLP_H; ++j) y += sm[L.oW3 + j] * sA2[j * SP + lane];
        sR[lane] = lane < ns ? y - Y[i0 + lane] : 0.f;
    }
    __syncthreads();
    const float d3 = 2.0f * sR[lane] / (float)n;
#pragma unroll
    for (int j = 0; j < HW; ++j)
        sD2[(HW * w + j) * SP + lane] = d3 * sm[L.oW3 + HW * w + j] * gelu_prime_f(z2[j]);
    __syncthreads();
    {
        float s[HW];
#pragma unroll
        for (int k = 0; k < HW; ++k) s[k] = 0.f;
#pragma unroll 4
        for (int j = 0; j < MLP_H; ++j) {
            const float dz = sD2[j * SP + lane];
            const float4 q = *reinterpret_cast<const float4*>(sm + L.oW2 + j * MLP_H + HW * w);
            s[0] += q.x * dz;
            s[1] += q.y * dz;
            s[2] += q.z * dz;
            s[3] += q.w * dz;
        }
#pragma unroll
        for (int k = 0; k < HW; ++k) sD1[(HW * w + k) * SP + lane] = s[k] * gelu_prime_f(z1[k]);
    }
    __syncthreads();
    float2* out = part + (size_t)blockIdx.x * (L.P + 1);
    auto row4 = [](const float* p, float* o) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    };
    // sums over the samples of the products of rows i0 + i IS of A and j0 + j JS of B
    // (interleaved rows: consecutive threads read consecutive rows)
    auto tile = [&](auto R_, auto C_, auto IS_, auto JS_, const float* A, const float* B, float2* o, int ldo) {
        constexpr int R = decltype(R_)::value, C = decltype(C_)::value, IS = decltype(IS_)::value,
                      JS = decltype(JS_)::value;
        Pair acc[R][C];
#pragma unroll 1
        for (int s = 0; s < MLP_SB; s += 4) {
            float a[R][4], b[C][4];
#pragma unroll
            for (int i = 0; i < R; ++i) row4(A + i * IS * SP + s, a[i]);
#pragma unroll
            for (int j = 0; j < C; ++j) row4(B + j * JS * SP + s, b[j]);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < C; ++j) acc[i][j].add_prod(a[i][q], b[j][q]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) o[i * IS * ldo + j * JS] = make_float2(acc[i][j].s, acc[i][j].c);
    };
    using std::integral_constant;
    if (tid < 256) {
        const int j = tid >> 4, k = tid & 15;
        tile(integral_constant<int, 4>{}, integral_constant<int, 4>{}, integral_constant<int, 16>{},
             integral_constant<int, 16>{}, sD2 + j * SP, sA1 + k * SP, out + L.oW2 + j * MLP_H + k, MLP_H);
        return;
    }
    const int t2 = tid - 256;
    {
        const int j = t2 / M::CG, d = t2 % M::CG;
        tile(integral_constant<int, M::TR>{}, integral_constant<int, M::TC>{}, integral_constant<int, 256 / M::CG>{},
             integral_constant<int, M::CG>{}, sD1 + j * SP, sX + d * SP, out + L.oW1 + j * D + d, D);
    }
    // biases, the last layer and the loss: one entry per thread
    if (t2 < 3 * MLP_H + 2) {
        const int j = t2 & (MLP_H - 1), g = t2 / MLP_H;
        const float* a = g == 0 ? sD1 + j * SP : g == 1 ? sD2 + j * SP : g == 2 ? sA2 + j * SP : sR;
        Pair acc;
        for (int s = 0; s < MLP_SB; ++s) {
            if (g < 2 || t2 == 3 * MLP_H)
                acc.add(a[s], 0.f);
            else
                acc.add_prod(a[s], sR[s]);
        }
        const int p = g == 0 ? L.ob1 + j : g == 1 ? L.ob2 + j : g == 2 ? L.oW3 + j : t2 == 3 * MLP_H ? L.ob3 : L.P;
        out[p] = make_float2(acc.s, acc.c);
    }
}

// gradient and loss from the blocks' sums: four threads per entry take the blocks
// in quarters, added in order
template <int D>
__global__ void __launch_bounds__(256) k_mlp_reduce(const float2* part, int nb, int n,
                                                    float* G, double* loss)
{
    grid_dependency();
    constexpr MlpLayout L = MlpLayout::make(D);
    __shared__ float2 s[4][64];
    const int e = threadIdx.x & 63, q = threadIdx.x >> 6, p = blockIdx.x * 64 + e;
    const int len = (nb + 3) / 4, b0 = q * len, b1 = min(nb, b0 + len);
    Pair acc;
    if (p <= L.P) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) {
            const float2 v = __ldcg(part + (size_t)b * (L.P + 1) + p);
            acc.add(v.x, v.y);
        }
    }
    s[q][e] = make_float2(acc.s, acc.c);
    __syncthreads();
    if (q == 0 && p <= L.P) {
        for (int r = 1; r < 4; ++r) acc.add(s[r][e].x, s[r][e].y);
        const double v = (double)acc.s + (double)acc.c;
        if (p == L.P)
            *loss = v / n;
        else
            G[p] = (float)(p >= L.oW3 ? 2.0 * v / n : v);
    }
}

// Adam (Kingma & Ba 2015) with bias corrections c1 = 1/(1-b1^t), c2 = 1/(1-b2^t)
static __global__ void k_mlp_adam(float* __restrict__ W, const float* __restrict__ G, float* __restrict__ m,
                           float* __restrict__ v, int P, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    const float g = G[p];
    const float mm = b1 * m[p] + (1.0f - b1) * g;
    const float vv = b2 * v[p] + (1.0f - b2) * g * g;
    m[p] = mm;
    v[p] = vv;
    W[p] -= lr * (mm * c1) / (sqrtf(vv * c2) + eps);
}

// ---------------------------------------------------------------------------
// fused inference: one warp per 16 samples, three BF16 mma.sync layers
// packed weights: B1 = W1^T [KD][64], B2 = W2^T [64][64], B3 = W3 as [64][8]
// (column 0), each as fragments [K/16][N/8][32 lanes][2 words], then b1, b2, b3
// ---------------------------------------------------------------------------
// x(r, k): FROMSTATE reads the cell's state (rho_l/rho_0) and |v|hat/cs,
// otherwise an explicit feature matrix X [n][D]
template <typename T, int K, bool FROMSTATE>
__global__ void __launch_bounds__(256) k_mlp_infer(const T* __restrict__ u, const T* __restrict__ vabs,
                                                   const float* __restrict__ X, long n,
                                                   const uint32_t* __restrict__ packed, float cs, float ref,
                                                   float gate, float* __restrict__ nu_out, float* __restrict__ y_out)
{
    constexpr int b = Dims<K>::b, D = 2 * b;
    using PK = MlpPack<D>;
    __shared__ uint32_t sP[PK::words];
    __shared__ float sF[FROMSTATE ? 8 * 16 * D : 1];  // a warp's 16 feature rows (state input)
    for (int e = threadIdx.x; e < PK::words; e += blockDim.x) sP[e] = packed[e];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const float inv_cs = 1.0f / cs;
    const long nwarps = (long)gridDim.x * (blockDim.x >> 5);
    for (long base = ((long)blockIdx.x * (blockDim.x >> 5) + warp) * 16; base < n; base += nwarps * 16) {
        float* sf = sF + (FROMSTATE ? warp * 16 * D : 0);
        if constexpr (FROMSTATE) {
            // the 16 rows: lane 2 rl + h loads row rl's rho coefficients (h = 0) or its
            // |v| projection (h = 1), all b loads in flight
            __syncwarp();
            const int rl = lane >> 1, h = lane & 1;
            const long r = base + rl;
            T x[b];
#pragma unroll
            for (int l = 0; l < b; ++l) x[l] = T(0);
            if (r < n) {
                const T* src = h == 0 ? u + r * 4 * b : vabs + r * b;
                if constexpr (sizeof(T) == 4 && b % 4 == 0) {
#pragma unroll
                    for (int l = 0; l < b; l += 4) {
                        const float4 q = __ldg(reinterpret_cast<const float4*>(src + l));
                        x[l] = q.x;
                        x[l + 1] = q.y;
                        x[l + 2] = q.z;
                        x[l + 3] = q.w;
                    }
                } else {
#pragma unroll
                    for (int l = 0; l < b; ++l) x[l] = src[l];
                }
            }
            float* dst = sf + rl * D + h * b;
#pragma unroll
            for (int l = 0; l < b; ++l)
                dst[l] = r >= n ? 0.0f : (h == 0 ? (float)(x[l] / x[0]) : (float)x[l] * inv_cs);
            __syncwarp();
        }
        auto feat = [&](int rl, int k) -> float {
            if constexpr (FROMSTATE) {
                return k < D ? sf[rl * D + k] : 0.0f;
            } else {
                const long r = base + rl;
                if (r >= n || k >= D) return 0.0f;
                return X[r * D + k];
            }
        };
        float y0, y1;
        mlp_infer_warp<D>(feat, sP, y0, y1);
        const long r0 = base + g, r1 = base + g + 8;
        if (t == 0) {
            if (r0 < n) {
                if (nu_out) nu_out[r0] = expf(y0) < gate ? 0.f : ref * expf(y0);
                if (y_out) y_out[r0] = y0;
            }
            if (r1 < n) {
                if (nu_out) nu_out[r1] = expf(y1) < gate ? 0.f : ref * expf(y1);
                if (y_out) y_out[r1] = y1;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// features and labels of the learned sensor for every cell (thread per
// (cell, point)): x = (rho_l/rho_0, |v|hat_l/cs), y = log(max(nu_cell,
// nu_f)/ref), nu_cell = the Gauss-weighted mean of Pi_vNR/(rho |div v|) over
// the compressive points (summed in a fixed order), nu_f = max(beta, 0.05) ref
// the coefficient of the linear term
// ---------------------------------------------------------------------------
template <typename T, int K>
__global__ void __launch_bounds__(Tile<K>::NT) k_features(const T* __restrict__ u, const T* __restrict__ vabs,
                                                          const T* __restrict__ phiv, const T* __restrict__ wq,
                                                          long ncell, Phys ph, double dt, float* __restrict__ X,
                                                          float* __restrict__ Y)
{
    using Dm = Dims<K>;
    constexpr int b = Dm::b, nq = Dm::nq, TC = Tile<K>::TC, NT = Tile<K>::NT, EC = 12;
    __shared__ T s_u[TC][4][b];
    __shared__ T s_ec[TC][b][EC];
    __shared__ T s_phi[b * nq];  // basis at the volume points [b][nq]
    __shared__ T s_nw[TC][nq], s_w[TC][nq];  // w_q nu_q and w_q at compressive points, else 0
    const int tid = threadIdx.x;
    for (int e = tid; e < b * nq; e += NT) s_phi[e] = phiv[e];
    const T two_h = T(2.0 / ph.h);
    const float ref = (float)(ph.cs * ph.hp);
    const long ntile = (ncell + TC - 1) / TC;
    for (long tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const long c0 = tile * TC;
        for (int e = tid; e < TC * 4 * b; e += NT) {
            const long c = c0 + e / (4 * b);
            (&s_u[0][0][0])[e] = (c < ncell) ? u[c0 * 4 * b + e] : ((e % (4 * b)) == 0 ? T(1) : T(0));
        }
        __syncthreads();
        for (int e = tid; e < TC * 5; e += NT) {
            const int lc = e / 5, g = e % 5;
            const T* uu = &s_u[lc][0][0];
            T out[b];
            if (g == 0) {
                for (int l = 0; l < b; ++l)
                    for (int v = 0; v < 4; ++v) s_ec[lc][l][v] = uu[v * b + l];
                continue;
            }
            if (g == 1) modal_grad<T, K, 0>(uu, out, two_h);
            if (g == 2) modal_grad<T, K, 1>(uu, out, two_h);
            if (g == 3) modal_grad<T, K, 2>(uu, out, two_h);
            if (g == 4) {
                T t2[b];
                modal_grad<T, K, 0>(uu + b, out, two_h);
                modal_grad<T, K, 1>(uu + 2 * b, t2, two_h);
                for (int l = 0; l < b; ++l) out[l] += t2[l];
                modal_grad<T, K, 2>(uu + 3 * b, t2, two_h);
                for (int l = 0; l < b; ++l) out[l] += t2[l];
            }
            for (int l = 0; l < b; ++l) s_ec[lc][l][3 + g] = out[l];
        }
        __syncthreads();
        static_assert(TC * nq <= NT, "one thread per (cell, point)");
        if (tid < TC * nq) {
            const int lc = tid / nq, q = tid % nq;
            T f[8];
            for (int i = 0; i < 8; ++i) f[i] = T(0);
            for (int l = 0; l < b; ++l) {
                const T p = s_phi[l * nq + q];
                for (int i = 0; i < 8; ++i) f[i] += s_ec[lc][l][i] * p;
            }
            const T rho = f[0], vx = f[1] / rho, vy = f[2] / rho, vz = f[3] / rho;
            const T divv = (f[7] - (vx * f[4] + vy * f[5] + vz * f[6])) / rho;
            T nw = T(0), w = T(0);
            if (divv < T(0)) {
                const T Pi = vnr_pressure<T>(ph, rho, divv, T(dt));
                w = wq[q];
                nw = w * (Pi / (rho * (-divv)));
            }
            s_nw[lc][q] = nw;
            s_w[lc][q] = w;
        }
        __syncthreads();
        for (int e = tid; e < TC * 2 * b; e += NT) {
            const int lc = e / (2 * b), k = e % (2 * b);
            const long c = c0 + lc;
            if (c >= ncell) continue;
            X[c * 2 * b + k] = (k < b) ? (float)(s_u[lc][0][k] / s_u[lc][0][0])
                                       : (float)(vabs[c * b + (k - b)] / T(ph.cs));
        }
        for (int lc = tid; lc < TC; lc += NT) {
            const long c = c0 + lc;
            if (c >= ncell) continue;
            T sn = T(0), sw = T(0);
            for (int q = 0; q < nq; ++q) {
                sn += s_nw[lc][q];
                sw += s_w[lc][q];
            }
            const float nu = sw > T(0) ? (float)(sn / sw) : 0.f;
            const float fl = fmaxf((float)ph.beta, 0.05f) * ref;
            Y[c] = logf(fmaxf(nu, fl) / ref);
        }
        __syncthreads();
    }
}

}  // namespace dg
