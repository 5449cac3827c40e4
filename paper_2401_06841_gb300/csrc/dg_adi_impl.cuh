// dg_adi_impl.cuh -- launchers of the adiabatic-system kernels (k = 1..3);
// instantiated per element type in dg_adi_f32.cu and dg_adi_f64.cu.
#pragma once

#include "dg_adi.cuh"
#include "dg_launch.cuh"
#include "dg_sf_adi.cuh"

namespace dg {

namespace sf {

template <typename T, int K, int MODE, bool FORCE, bool PROJ>
cudaError_t adi_vol(const Launch& L, const AArgs<T>& a)
{
    using C = AVolCfg<T, K, MODE, FORCE, PROJ>;
    constexpr size_t sm = sizeof(T) * C::total;
    static const int occ = [] {
        int o = 0;
        cudaFuncSetAttribute(k_sfa_vol<T, K, MODE, FORCE, PROJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_sfa_vol<T, K, MODE, FORCE, PROJ>, C::NT, sm) !=
            cudaSuccess)
            o = 1;
        return o < 1 ? 1 : o;
    }();
    const long ntile = (L.ncell + TCELL - 1) / TCELL;
    long g = (long)occ * L.nsm;
    if (g > ntile) g = ntile;
    if (g > kMaxGrid) g = kMaxGrid;
    return launch_dependent(k_sfa_vol<T, K, MODE, FORCE, PROJ>, (unsigned)g, C::NT, sm, L.st, a);
}

template <typename T, int K, int RS, bool STAGE>
cudaError_t adi_faces(const Launch& L, const AArgs<T>& a)
{
    constexpr size_t sm = sizeof(T) * AFaceCfg<T, K>::total;
    static const cudaError_t ready = cudaFuncSetAttribute(k_sfa_faces<T, K, RS, STAGE>,
                                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (ready != cudaSuccess) return ready;
    const int g = Brick::count(L.N);
    return launch_dependent(k_sfa_faces<T, K, RS, STAGE>, g, 128, sm, L.st, a);
}

template <typename T, int K>
cudaError_t adi_k(const Launch& L, double gamma, const AdiLaunch& t)
{
    using TT = TileTab<K, BK_FMA>;
    AArgs<T> a{};
    const bool driven = (t.flags & F_FORCE) != 0;
    if (driven && !t.ahat) return cudaErrorInvalidValue;
    a.u_in = static_cast<const T*>(t.u_in);
    a.u_n = static_cast<const T*>(t.u_n);
    a.out = static_cast<T*>(t.out);
    a.pr_in = static_cast<const T*>(t.pr_in);
    a.pr_out = static_cast<T*>(t.pr_out);
    a.ahat = driven ? static_cast<const T*>(t.ahat) : nullptr;
    a.phiv = static_cast<const T*>(L.ttab) + TT::phiv;
    a.phif = static_cast<const T*>(L.ttab) + TT::phif;
    a.ctl = L.ctl;
    a.partials = L.partials;
    a.ncell = L.ncell;
    a.N = L.N;
    a.av_mode = L.ph.av_mode;
    a.stage = t.mode == ADI_STAGE;
    a.dtf = (t.flags & F_DT) ? 1 : 0;
    a.abar_in = t.abar_in;
    a.abar_out = t.abar_out;
    fill_rows<T, K>(a.rows);
    a.gas.gamma = T(gamma);
    a.gas.g1 = T(gamma - 1.0);
    a.gas.ig1 = T(1.0 / (gamma - 1.0));
    a.gas.kap = T(t.kap);
    a.gas.c0 = T((gamma - 1.0) * t.kap);
    a.gas.cres = T(t.cs_reset * t.cs_reset / (gamma - 1.0) - t.kap);
    a.two_h = T(2.0 / L.ph.h);
    a.inv_h = T(1.0 / L.ph.h);
    a.eps = T(L.ph.floor_);
    a.a2 = T(L.ph.alpha * L.ph.hp * L.ph.hp);
    a.bh = T(L.ph.beta * L.ph.hp);
    a.rk_a = T(t.rk_a);
    a.rk_b = T(t.rk_b);
    a.hp = L.ph.hp;
    a.h3 = L.ph.h * L.ph.h * L.ph.h;
    a.dt_pimax = t.dt_pimax;
    a.beta = t.beta;
    for (int i = 0; i < 3; ++i) a.bc[i] = t.bc[i];
    for (int i = 0; i < 4; ++i) a.inflow[i] = T(t.inflow[i]);
    a.inflow[4] = T(t.inflow[4] - (double)a.gas.c0 * t.inflow[0]);
    if (t.mode == ADI_PROJECT)
        return driven ? adi_vol<T, K, SFA_PROJECT, true, true>(L, a) : adi_vol<T, K, SFA_PROJECT, false, true>(L, a);
    if (t.mode == ADI_RESET) return adi_vol<T, K, SFA_RESET, false, false>(L, a);
    cudaError_t e;
    if (t.flags & F_SELFPROJ) {
        a.pr_out = const_cast<T*>(a.pr_in);
        a.abar_out = t.abar_in;
        e = driven ? adi_vol<T, K, SFA_VOLUME, true, true>(L, a) : adi_vol<T, K, SFA_VOLUME, false, true>(L, a);
    } else {
        e = driven ? adi_vol<T, K, SFA_VOLUME, true, false>(L, a) : adi_vol<T, K, SFA_VOLUME, false, false>(L, a);
    }
    if (e != cudaSuccess) return e;
    if (a.stage)
        return L.ph.riemann == 2 ? adi_faces<T, K, 2, true>(L, a) : adi_faces<T, K, 0, true>(L, a);
    return L.ph.riemann == 2 ? adi_faces<T, K, 2, false>(L, a) : adi_faces<T, K, 0, false>(L, a);
}

}  // namespace sf

// the degree-3 launcher compiles in a translation unit of its own
#define DG_ADI_K3_EXTERN(T) \
    extern template cudaError_t sf::adi_k<T, 3>(const Launch&, double, const AdiLaunch&);
#define DG_ADI_K3_INSTANTIATE(T) template cudaError_t sf::adi_k<T, 3>(const Launch&, double, const AdiLaunch&);

namespace {

template <typename T, int K>
cudaError_t adi_totals_k(const Launch& L, double gamma, double kap, const void* u, double* partials, int* nblocks)
{
    long g = (L.ncell + 255) / 256;
    if (g > 4L * L.nsm) g = 4L * L.nsm;
    if (g > kMaxGrid) g = kMaxGrid;
    if (g < 1) g = 1;
    *nblocks = (int)g;
    k_adi_totals<T, K><<<(int)g, 256, 0, L.st>>>(static_cast<const T*>(u), static_cast<const T*>(L.ttab), L.ncell,
                                                 gamma, (gamma - 1.0) * kap, partials);
    return cudaGetLastError();
}

}  // namespace

template <typename T>
cudaError_t launch_adi(const Launch& L, double gamma, const AdiLaunch& t)
{
    if (L.K == 1) return sf::adi_k<T, 1>(L, gamma, t);
    if (L.K == 2) return sf::adi_k<T, 2>(L, gamma, t);
    return sf::adi_k<T, 3>(L, gamma, t);
}

template <typename T>
cudaError_t launch_adi_totals(const Launch& L, double gamma, double kap, const void* u, double* partials, int* nblocks)
{
    if (L.K == 1) return adi_totals_k<T, 1>(L, gamma, kap, u, partials, nblocks);
    if (L.K == 2) return adi_totals_k<T, 2>(L, gamma, kap, u, partials, nblocks);
    return adi_totals_k<T, 3>(L, gamma, kap, u, partials, nblocks);
}

// e_s += d rho, coefficient by coefficient (a change of the energy offset)
template <typename T>
__global__ void k_adi_shift(T* u, long ncell, int b, T d)
{
    const long n = ncell * b;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const long c = i / b;
        const int l = (int)(i % b);
        u[(c * 5 + 4) * b + l] += d * u[c * 5 * b + l];
    }
}

template <typename T>
cudaError_t launch_adi_shift(const Launch& L, void* u, double d)
{
    const int b = (L.K + 1) * (L.K + 2) * (L.K + 3) / 6;
    long g = (L.ncell * b + 255) / 256;
    if (g > 8L * L.nsm) g = 8L * L.nsm;
    if (g < 1) g = 1;
    k_adi_shift<T><<<(int)g, 256, 0, L.st>>>(static_cast<T*>(u), L.ncell, b, T(d));
    return cudaGetLastError();
}

}  // namespace dg
