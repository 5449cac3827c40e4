// dg_adi.cuh -- physics of the adiabatic system (Sec. 2.1): five conserved
// variables u = (rho, m, e) per cell with the ideal-gas equation of state
// p = (gamma - 1)(e - |m|^2 / (2 rho)) and the flux
//   F_d = (m_d, m v_d + p e_d, (e + p) v_d).
// Pointwise physics (fluxes, pressure, the positivity root) and the diagnostics;
// the right-hand side's kernels are in dg_sf_adi.cuh.
#pragma once

#include "../../include/dg.h"
#include "dg_launch.cuh"
#include "dg_tile.cuh"

namespace dg {

// gas constants in the element type, each rounded once from its double value on
// the host: near gamma = 1 the difference gamma - 1 formed in single precision
// would carry the rounding of gamma (float(1.0001) - 1 = 1.000166e-4).
// Energy offset: the fifth variable is stored as e_s = e - kap rho (kap = cs^2 /
// (gamma - 1) in reset mode, 0 otherwise), so that the thermal energy of the
// isothermal reference, 1/(gamma - 1) times larger than the kinetic energy, is
// not carried in the state: p = (gamma - 1)(e_s - |m|^2/(2 rho)) + c0 rho with
// c0 = (gamma - 1) kap, the energy flux (e_s + p) v, and the projected pressure
// is the deviation p - c0 rho.  The scheme is linear in the state, so this is
// the same discretisation in other variables.
template <typename T>
struct AdiGas {
    T gamma;   // gamma
    T g1;      // gamma - 1
    T ig1;     // 1 / (gamma - 1)
    T cth;     // reset mode: cs^2 / (gamma - 1), the thermal energy per unit mass
    T kap;     // energy offset per unit mass
    T c0;      // (gamma - 1) kap: the pressure of the offset per unit density
    T cres;    // cth - kap: the thermal energy per unit mass the reset leaves in e_s
};

constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Rusanov flux along Dd from primitive face states W = (rho, v_x, v_y, v_z, p - c0 rho):
// 1/2 (F(U_L) + F(U_R)) - 1/2 lambda (U_R - U_L), lambda = max(|v_n| + c)
template <typename T, int Dd>
__device__ __forceinline__ void adi_rusanov(const AdiGas<T>& G, const T* WL, const T* WR, T* F)
{
    const T g1 = G.g1, gamma = G.gamma;
    T UL[5], UR[5], FL[5], FR[5], ls[2];
    const T* W[2] = {WL, WR};
    T* U[2] = {UL, UR};
    T* Fx[2] = {FL, FR};
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const T* w = W[s];
        const T rho = w[0], vn = w[1 + Dd], p = w[4] + G.c0 * rho;  // w[4]: the pressure deviation
        U[s][0] = rho;
        U[s][1] = rho * w[1];
        U[s][2] = rho * w[2];
        U[s][3] = rho * w[3];
        U[s][4] = w[4] / g1 + T(0.5) * rho * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
        Fx[s][0] = U[s][1 + Dd];
        Fx[s][1] = U[s][1] * vn;
        Fx[s][2] = U[s][2] * vn;
        Fx[s][3] = U[s][3] * vn;
        Fx[s][1 + Dd] += p;
        Fx[s][4] = (U[s][4] + p) * vn;
        ls[s] = fabs(vn) + sqrt(gamma * p / rho);
    }
    // the larger of the two (a NaN of the right state propagates, as in the oracle)
    const T lam = ls[0] > ls[1] ? ls[0] : ls[1];
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = T(0.5) * (FL[v] + FR[v]) - T(0.5) * lam * (UR[v] - UL[v]);
}

// HLLC flux along Dd from primitive face states (the contact wave restored in
// the two-wave model): Davis bounds S_L = min(u - c), S_R = max(u + c) over the
// two states, the contact speed S* from the pressures and the mass fluxes
// relative to the bounds, star states U*_K = rho_K (S_K - u_K)/(S_K - S*)
// (1, S* along Dd, the tangential velocities, E_K/rho_K + (S* - u_K)(S* +
// p_K/(rho_K (S_K - u_K)))), and the flux of the region x/t = 0 falls in
template <typename T, int Dd>
__device__ __forceinline__ void adi_hllc(const AdiGas<T>& G, const T* WL, const T* WR, T* F)
{
    const T g1 = G.g1, gamma = G.gamma;
    T U[2][5], Fx[2][5], c[2], un[2], pp[2];
    const T* W[2] = {WL, WR};
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const T* w = W[s];
        const T rho = w[0], p = w[4] + G.c0 * rho;  // w[4]: the pressure deviation
        pp[s] = p;
        un[s] = w[1 + Dd];
        U[s][0] = rho;
        U[s][1] = rho * w[1];
        U[s][2] = rho * w[2];
        U[s][3] = rho * w[3];
        U[s][4] = w[4] / g1 + T(0.5) * rho * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
        Fx[s][0] = U[s][1 + Dd];
        Fx[s][1] = U[s][1] * un[s];
        Fx[s][2] = U[s][2] * un[s];
        Fx[s][3] = U[s][3] * un[s];
        Fx[s][1 + Dd] += p;
        Fx[s][4] = (U[s][4] + p) * un[s];
        c[s] = sqrt(gamma * p / rho);
    }
    const T a0 = un[0] - c[0], a1 = un[1] - c[1], b0 = un[0] + c[0], b1 = un[1] + c[1];
    const T SL = a0 < a1 ? a0 : a1, SR = b0 > b1 ? b0 : b1;
    if (SL >= T(0)) {
#pragma unroll
        for (int v = 0; v < 5; ++v) F[v] = Fx[0][v];
        return;
    }
    if (SR <= T(0)) {
#pragma unroll
        for (int v = 0; v < 5; ++v) F[v] = Fx[1][v];
        return;
    }
    const T qL = WL[0] * (SL - un[0]), qR = WR[0] * (SR - un[1]);
    const T Ss = (pp[1] - pp[0] + un[0] * qL - un[1] * qR) / (qL - qR);
    // the side of the contact x/t = 0 lies on (selects keep everything in registers)
    const bool lft = Ss >= T(0);
    const T SK = lft ? SL : SR, qK = lft ? qL : qR, uK = lft ? un[0] : un[1], pK = lft ? pp[0] : pp[1];
    T wK[5], UK[5], FK[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        wK[v] = lft ? WL[v] : WR[v];
        UK[v] = lft ? U[0][v] : U[1][v];
        FK[v] = lft ? Fx[0][v] : Fx[1][v];
    }
    const T f = qK / (SK - Ss);
    T Us[5];
    Us[0] = f;
#pragma unroll
    for (int i = 0; i < 3; ++i) Us[1 + i] = f * (i == Dd ? Ss : wK[1 + i]);
    Us[4] = f * (UK[4] / wK[0] + (Ss - uK) * (Ss + pK / qK));
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = FK[v] + SK * (Us[v] - UK[v]);
}

// smallest t in [0, 1] with p(ub + t d) = eps (p(ub) > eps > p(ub + d)): the
// root of rho p - eps rho = (gamma-1)(rho e_s - |m|^2/2) + c0 rho^2 - eps rho,
// quadratic in t
template <typename T>
__device__ __forceinline__ T adi_pressure_root(const AdiGas<T>& G, T eps, const T* ub, const T* dv)
{
    const T g1 = G.g1, c0 = G.c0;
    const T A = g1 * (dv[0] * dv[4] - T(0.5) * (dv[1] * dv[1] + dv[2] * dv[2] + dv[3] * dv[3])) + c0 * dv[0] * dv[0];
    const T B = g1 * (ub[0] * dv[4] + dv[0] * ub[4] - (ub[1] * dv[1] + ub[2] * dv[2] + ub[3] * dv[3])) +
                T(2) * c0 * ub[0] * dv[0] - eps * dv[0];
    const T C = g1 * (ub[0] * ub[4] - T(0.5) * (ub[1] * ub[1] + ub[2] * ub[2] + ub[3] * ub[3])) + c0 * ub[0] * ub[0] -
                eps * ub[0];
    T t;
    if (fabs(A) <= T(1e-14) * (fabs(B) + fabs(C))) {
        t = -C / B;
    } else {
        T disc = B * B - T(4) * A * C;
        disc = disc < T(0) ? T(0) : disc;
        const T sq = sqrt(disc);
        const T r1 = (-B - sq) / (T(2) * A), r2 = (-B + sq) / (T(2) * A);
        const T lo = r1 < r2 ? r1 : r2, hi = r1 < r2 ? r2 : r1;
        t = (lo >= T(0) && lo <= T(1)) ? lo : hi;
    }
    t = t < T(0) ? T(0) : t;
    return t > T(1) ? T(1) : t;
}

// pressure from the stored variables (e: the offset energy e_s), and its
// deviation p - c0 rho
template <typename T>
__device__ __forceinline__ T adi_pdev(const AdiGas<T>& G, T rho, T mx, T my, T mz, T e)
{
    return G.g1 * (e - T(0.5) * (mx * mx + my * my + mz * mz) / rho);
}
template <typename T>
__device__ __forceinline__ T adi_p(const AdiGas<T>& G, T rho, T mx, T my, T mz, T e)
{
    return adi_pdev<T>(G, rho, mx, my, mz, e) + G.c0 * rho;
}

// FP64 totals for the diagnostics: per block [mass, m_x, m_y, m_z, energy of
// the stored variable (offset energy e_s), kinetic energy (volume quadrature of
// |m|^2/(2 rho)), min rho, min p at the volume points], summed over blocks on the
// host in block order.  Point values in the state's precision, sums in FP64; c0 =
// (gamma - 1) kap the pressure of the energy offset per unit density.
template <typename T, int K>
__global__ void __launch_bounds__(256) k_adi_totals(const T* __restrict__ u, const T* __restrict__ tab, long ncell,
                                                   double gamma, double c0, double* __restrict__ partials)
{
    using TT = TileTab<K, BK_FMA>;
    constexpr int b = Dims<K>::b, nq = Dims<K>::nq, n = K + 1;
    __shared__ double s_red[256];
    __shared__ double s_w[nq];
    // Gauss weights (per-point volume weights w_q / 8) from the mass identity: the
    // projection weights are the phi_0 = 1 row of the weighted transpose table
    if (threadIdx.x < nq) s_w[threadIdx.x] = (double)tab[TileCfg<K, BK_FMA>::oWPhi + threadIdx.x * TileCfg<K, BK_FMA>::NP];
    __syncthreads();
    (void)n;
    double acc[6] = {0, 0, 0, 0, 0, 0}, rmin = 1e300, pmin = 1e300;
    for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < ncell; c += (long)gridDim.x * blockDim.x) {
        const T* uc = u + c * 5 * b;
        for (int v = 0; v < 5; ++v) acc[v] += (double)uc[v * b];  // mode 0: the cell mean
        for (int q = 0; q < nq; ++q) {
            T w[5];
            for (int v = 0; v < 5; ++v) {
                T s = T(0);
                for (int l = 0; l < b; ++l) s += uc[v * b + l] * tab[TT::phiv + l * nq + q];
                w[v] = s;
            }
            const double ke = 0.5 * ((double)w[1] * w[1] + (double)w[2] * w[2] + (double)w[3] * w[3]) / (double)w[0];
            acc[5] += s_w[q] * ke;
            const double p = (gamma - 1.0) * ((double)w[4] - ke) + c0 * (double)w[0];
            rmin = (double)w[0] < rmin ? (double)w[0] : rmin;
            pmin = p < pmin ? p : pmin;
        }
    }
    double vals[8] = {acc[0], acc[1], acc[2], acc[3], acc[4], acc[5], rmin, pmin};
    for (int i = 0; i < 8; ++i) {
        s_red[threadIdx.x] = vals[i];
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = i < 6 ? 0.0 : 1e300;
            for (int j = 0; j < (int)blockDim.x; ++j) t = i < 6 ? t + s_red[j] : (s_red[j] < t ? s_red[j] : t);
            partials[blockIdx.x * 8 + i] = t;
        }
        __syncthreads();
    }
}

}  // namespace dg
