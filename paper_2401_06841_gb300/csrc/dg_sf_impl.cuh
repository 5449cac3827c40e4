// dg_sf_impl.cuh -- launchers of the sum-factorised kernels (dg_sf.cuh), one
// explicit instantiation per element type and degree (dg_sf_*.cu).
#pragma once

#include "dg_launch.cuh"
#include "dg_sf.cuh"

namespace dg {
namespace sf {

template <typename T, int K>
struct Occ {
    static int vol[8];  // resident blocks per SM: FORCE (1), PROJ (2) of the volume kernels; 4 + FORCE (1), VABS (2)
};
template <typename T, int K>
int Occ<T, K>::vol[8] = {};

template <typename F>
static cudaError_t prepare(F* fn, size_t smem, int nt, int* occ)
{
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess || !occ) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, fn, nt, smem);
}

template <typename T, int K, bool VOL, bool FORCE, bool PROJ, bool VABS>
static cudaError_t prepare_vol(int* occ)
{
    using C = VolCfg<T, K, VOL, FORCE, PROJ, VABS>;
    return prepare(k_sf_vol<T, K, VOL, FORCE, PROJ, VABS>, sizeof(T) * C::total, C::NT, occ);
}

template <typename T, int K>
cudaError_t setup()
{
    int* o = Occ<T, K>::vol;
    cudaError_t e;
    if ((e = prepare_vol<T, K, true, false, false, false>(o + 0))) return e;
    if ((e = prepare_vol<T, K, true, true, false, false>(o + 1))) return e;
    if ((e = prepare_vol<T, K, true, false, true, false>(o + 2))) return e;
    if ((e = prepare_vol<T, K, true, true, true, false>(o + 3))) return e;
    if ((e = prepare_vol<T, K, false, false, true, false>(o + 4))) return e;
    if ((e = prepare_vol<T, K, false, true, true, false>(o + 5))) return e;
    if ((e = prepare_vol<T, K, false, false, true, true>(o + 6))) return e;
    if ((e = prepare_vol<T, K, false, true, true, true>(o + 7))) return e;
    const size_t sm = sizeof(T) * FaceCfg<T, K>::total;
    if ((e = prepare(k_sf_faces<T, K, 0, true>, sm, 128, nullptr))) return e;
    if ((e = prepare(k_sf_faces<T, K, 1, true>, sm, 128, nullptr))) return e;
    if ((e = prepare(k_sf_faces<T, K, 2, true>, sm, 128, nullptr))) return e;
    if ((e = prepare(k_sf_faces<T, K, 0, false>, sm, 128, nullptr))) return e;
    if ((e = prepare(k_sf_faces<T, K, 1, false>, sm, 128, nullptr))) return e;
    return prepare(k_sf_faces<T, K, 2, false>, sm, 128, nullptr);
}

template <typename T, int K, bool VOL, bool FORCE, bool PROJ, bool VABS>
static cudaError_t go_vol(const Launch& L, const Args<T>& a, int occ)
{
    using C = VolCfg<T, K, VOL, FORCE, PROJ, VABS>;
    const long ntile = (L.ncell + TCELL - 1) / TCELL;
    long g = (long)(occ < 1 ? 1 : occ) * L.nsm;
    if (g > ntile) g = ntile;
    if (g > kMaxGrid) g = kMaxGrid;
    return launch_dependent(k_sf_vol<T, K, VOL, FORCE, PROJ, VABS>, (unsigned)g, C::NT, sizeof(T) * C::total, L.st, a);
}

template <typename T, int K, bool STAGE>
static cudaError_t go_faces(const Launch& L, const Args<T>& a)
{
    const size_t sm = sizeof(T) * FaceCfg<T, K>::total;
    const int g = Brick::count(L.N);
    if (L.ph.riemann == 2)
        return launch_dependent(k_sf_faces<T, K, 2, STAGE>, g, 128, sm, L.st, a);
    if (L.ph.riemann == 1) return launch_dependent(k_sf_faces<T, K, 1, STAGE>, g, 128, sm, L.st, a);
    return launch_dependent(k_sf_faces<T, K, 0, STAGE>, g, 128, sm, L.st, a);
}

// the projection launch (mode 0), or the volume and face launches of a
// right-hand side / stage; a stage's F_NEXTPROJ is the caller's (a projection
// launch of its output), F_SELFPROJ projects the stage's input in its volume kernel
template <typename T, int K>
cudaError_t launch(const Launch& L, const TileLaunch& t)
{
    using TT = TileTab<K, BK_FMA>;
    Args<T> a{};
    const bool force = (t.flags & F_FORCE) != 0;
    a.u_in = static_cast<const T*>(t.u_in);
    a.u_n = static_cast<const T*>(t.u_n);
    a.out = static_cast<T*>(t.out);
    a.vh_in = static_cast<const T*>(t.vh_in);
    a.ahat = force ? static_cast<const T*>(t.ahat) : nullptr;
    a.phiv = static_cast<const T*>(L.ttab) + TT::phiv;
    a.phif = static_cast<const T*>(L.ttab) + TT::phif;
    a.nu = t.nu;
    a.ctl = L.ctl;
    a.partials = L.partials;
    a.ncell = L.ncell;
    a.N = L.N;
    a.av_mode = L.ph.av_mode;
    a.tcount = TileCfg<K, BK_FMA>::TC;
    fill_rows<T, K>(a.rows);
    a.two_h = T(2.0 / L.ph.h);
    a.inv_h = T(1.0 / L.ph.h);
    a.cs = T(L.ph.cs);
    a.cs2 = T(L.ph.cs2);
    a.eps = T(L.ph.floor_);
    a.a2 = T(L.ph.alpha * L.ph.hp * L.ph.hp);
    a.b1 = T(L.ph.beta * L.ph.cs * L.ph.hp);
    a.rk_a = T(t.rk_a);
    a.rk_b = T(t.rk_b);
    a.cs_d = L.ph.cs;
    a.hp = L.ph.hp;
    a.dt_pimax = t.dt_pimax;
    a.trouble = t.mode == TM_RHS ? nullptr : t.trouble;
    a.abar_in = t.abar_in;
    a.abar_out = t.abar_out;
    const int* o = Occ<T, K>::vol;
    if (t.mode == TM_PROJECT) {
        a.vh_out = static_cast<T*>(t.vh_out);
        a.vabs_out = static_cast<T*>(t.vabs_out);
        a.dtf = (t.flags & F_DT) ? 1 : 0;
        if (t.vabs_out)
            return force ? go_vol<T, K, false, true, true, true>(L, a, o[7])
                         : go_vol<T, K, false, false, true, true>(L, a, o[6]);
        return force ? go_vol<T, K, false, true, true, false>(L, a, o[5])
                     : go_vol<T, K, false, false, true, false>(L, a, o[4]);
    }
    a.stage = t.mode != TM_RHS;
    cudaError_t e;
    if (t.flags & F_SELFPROJ) {
        a.vh_out = const_cast<T*>(a.vh_in);
        a.abar_out = t.abar_in;
        e = force ? go_vol<T, K, true, true, true, false>(L, a, o[3]) : go_vol<T, K, true, false, true, false>(L, a, o[2]);
    } else {
        e = force ? go_vol<T, K, true, true, false, false>(L, a, o[1])
                  : go_vol<T, K, true, false, false, false>(L, a, o[0]);
    }
    if (e != cudaSuccess) return e;
    return a.stage ? go_faces<T, K, true>(L, a) : go_faces<T, K, false>(L, a);
}

}  // namespace sf

#define DG_SF_INSTANTIATE(T, K)                                            \
    template cudaError_t sf::launch<T, K>(const Launch&, const TileLaunch&); \
    template cudaError_t sf::setup<T, K>();

}  // namespace dg
