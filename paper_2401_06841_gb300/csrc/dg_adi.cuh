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
    T kap;     // energy offset per unit mass
    T c0;      // (gamma - 1) kap: the pressure of the offset per unit density
    T cres;    // reset mode: cs^2 / (gamma - 1) - kap, the thermal energy per unit mass it leaves in e_s
};

constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Face fluxes along the normal (component 1) from primitive face states W = (rho, v_n,
// v_t1, v_t2, p - c0 rho).  Rusanov, (F_L + F_R)/2 - lambda (U_R - U_L)/2 with lambda =
// max(|v_n| + c): the momentum carried by q_L = rho_L (v_n,L + lambda)/2 and q_R = rho_R
// (v_n,R - lambda)/2, mass and energy from the differences of rho and e (slow flows would
// lose them between terms of the size rho c)
template <typename T>
__device__ __forceinline__ void adi_rusanov(const AdiGas<T>& G, const T* WL, const T* WR, T* F)
{
    const T pL = WL[4] + G.c0 * WL[0], pR = WR[4] + G.c0 * WR[0];  // W[4]: the pressure deviation
    const T aL = fabs(WL[1]) + fast_sqrt<T>(G.gamma * pL * rcp<T>(WL[0]));
    const T aR = fabs(WR[1]) + fast_sqrt<T>(G.gamma * pR * rcp<T>(WR[0]));
    // the larger of the two (a NaN of the right state propagates, as in the oracle)
    const T hl = T(0.5) * (aL > aR ? aL : aR);
    const T hL = T(0.5) * WL[1], hR = T(0.5) * WR[1];
    const T mL = WL[0] * hL, mR = WR[0] * hR;
    const T qL = mL + hl * WL[0], qR = mR - hl * WR[0];
    const T eL = WL[4] * G.ig1 + T(0.5) * WL[0] * (WL[1] * WL[1] + WL[2] * WL[2] + WL[3] * WL[3]);
    const T eR = WR[4] * G.ig1 + T(0.5) * WR[0] * (WR[1] * WR[1] + WR[2] * WR[2] + WR[3] * WR[3]);
    F[0] = (mL + mR) - hl * (WR[0] - WL[0]);
    F[1] = T(0.5) * (pL + pR) + (qL * WL[1] + qR * WR[1]);
    F[2] = qL * WL[2] + qR * WR[2];
    F[3] = qL * WL[3] + qR * WR[3];
    F[4] = ((eL + pL) * hL + (eR + pR) * hR) - hl * (eR - eL);
}

// HLLC (the contact wave restored in the two-wave model): Davis bounds S_L = min(u - c),
// S_R = max(u + c) over the two states, the contact speed S* from the pressures and the
// mass fluxes q_K = rho_K (S_K - u_K) relative to the bounds; behind the contact, on the
// side K that x/t = 0 lies on, rho* = q_K/(S_K - S*), p* = p_K + q_K (S* - u_K), E* =
// (E_K (S_K - u_K) - p_K u_K + p* S*)/(S_K - S*), and the flux is that of this state at
// the normal velocity S* (outside the bounds: of the state K itself)
template <typename T>
__device__ __forceinline__ void adi_hllc(const AdiGas<T>& G, const T* WL, const T* WR, T* F)
{
    const T pL = WL[4] + G.c0 * WL[0], pR = WR[4] + G.c0 * WR[0];
    const T cL = fast_sqrt<T>(G.gamma * pL * rcp<T>(WL[0])), cR = fast_sqrt<T>(G.gamma * pR * rcp<T>(WR[0]));
    const T a0 = WL[1] - cL, a1 = WR[1] - cR, b0 = WL[1] + cL, b1 = WR[1] + cR;
    const T SL = a0 < a1 ? a0 : a1, SR = b0 > b1 ? b0 : b1;
    const T qL = WL[0] * (SL - WL[1]), qR = WR[0] * (SR - WR[1]);
    const T Ss = (pR - pL + WL[1] * qL - WR[1] * qR) * rcp<T>(qL - qR);
    // selects keep everything in registers
    const bool outer = SL >= T(0) || SR <= T(0);
    const bool lft = SL >= T(0) || (!(SR <= T(0)) && Ss >= T(0));
    const T SK = lft ? SL : SR, qK = lft ? qL : qR, pK = lft ? pL : pR;
    T w[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) w[v] = lft ? WL[v] : WR[v];
    const T e = w[4] * G.ig1 + T(0.5) * w[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
    const T r = rcp<T>(SK - Ss);
    const T us = outer ? w[1] : Ss, ps = outer ? pK : pK + qK * (Ss - w[1]), rs = outer ? w[0] : qK * r;
    const T es = outer ? e : (e * (SK - w[1]) - pK * w[1] + ps * Ss) * r;
    F[0] = rs * us;
    F[1] = F[0] * us + ps;
    F[2] = F[0] * w[2];
    F[3] = F[0] * w[3];
    F[4] = (es + ps) * us;
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
