// dg_sf_adi.cuh -- sum-factorised kernels of the adiabatic system (Sec. 2.1): five
// conserved variables u = (rho, m, e) per cell with the ideal-gas equation of state
// p = (gamma - 1)(e - |m|^2 / (2 rho)) and the flux
//   F_d = (m_d, m v_d + p e_d, (e + p) v_d),
// on the layout of dg_sf.cuh: a warp per plane of Gauss points in the volume
// kernel, a thread per face of a 4 x 4 x 2 brick in the face kernel.
//
//   k_sfa_vol MODE  SFA_PROJECT  projections of v and p (Sec. 3.2) -> pr_out, with the
//                                CFL bound max sum_d(|v_d| + c) (a.dtf) and, driven,
//                                the mean acceleration <rho a_h>/<rho>
//                   SFA_VOLUME   volume term -> out; driven: with the source rho a_h
//                                and its work m.a_h (the mean acceleration's part,
//                                -abar rho_l and -abar.m_l, is the face kernel's: the
//                                quadrature of these products is exact); PROJ: also
//                                the projections of its input, and the mean acceleration
//                   SFA_RESET    uniform temperature restored in place (Sec. 4.2): e
//                                becomes the projection of rho cs^2/(gamma-1) +
//                                |m|^2/(2 rho)
//   k_sfa_faces     face traces, Riemann fluxes, surface term + volume term, SSP-RK
//                   combine, positivity of density and pressure (Sec. 3.1)
// FP64 accumulators in ctl->work: [0] injected energy (beta_s dt times the volume
// integral of the energy source), [1] dissipated energy (the thermal energy the
// reset takes out).
// Bound as in dg_sf.cuh.  64^3 of degree 3 FP32: an SSP-RK3 step takes 1.27 ms (volume
// 107 to 148, faces 236 us a stage, projection 79), on dense products 5.4; 48^3 of degree
// 2, driven with HLLC and the reset, 0.40 ms for 2.1.
#pragma once

#include "dg_adi.cuh"
#include "dg_sf.cuh"

namespace dg {
namespace sf {

enum { SFA_PROJECT = 0, SFA_VOLUME = 1, SFA_RESET = 2 };

template <typename T>
struct AArgs {
    const T* u_in;   // [c][5][b]
    const T* u_n;
    T* out;          // volume kernel: volume term; face kernel: volume term in, result out
    const T* pr_in;  // face kernel: projections of v and p of u_in [c][4][b]
    T* pr_out;       // volume kernel: the same, written
    const T* ahat;   // driving or nullptr
    const T* phiv;   // [b][nq], [b][nf]: exact positivity check
    const T* phif;
    Ctl* ctl;
    double* partials;
    long ncell;
    int N;
    int av_mode;
    int stage;       // 1: the step's dt, 0: dt_pimax
    int dtf;
    int abar_in, abar_out;
    Rows<T> rows;
    AdiGas<T> gas;
    T two_h, inv_h, eps, a2, bh;  // a2 = alpha (h/p)^2, bh = beta h/p
    T rk_a, rk_b;
    double hp, h3, dt_pimax, beta;
    int bc[3];
    T inflow[5];     // rho, v, p - c0 rho at the face at coordinate 0
};

template <typename T, int K, int MODE, bool FORCE, bool PROJ>
struct AVolCfg {
    static constexpr int b = Dims<K>::b, n = K + 1, NT = 32 * n;
    static constexpr int NP = npair(K), NPD = npair(K - 1);
    static constexpr bool VOL = MODE == SFA_VOLUME, SRC = VOL && FORCE;
    static constexpr int NC = VOL ? 9 : 0, NV = MODE == SFA_RESET ? 1 : (PROJ ? 4 : 0);
    static constexpr int LDU = padded<T>(5 * b), LDA = padded<T>(3 * b), LDH = padded<T>(b);
    static constexpr int NX = cmax(cmax(NC * NPD, NV * NP), SRC ? 4 * NP : 0);
    static constexpr int oU = 0;                                // [2][32][LDU]
    static constexpr int oAh = oU + 2 * TCELL * LDU;            // [32][LDA]
    static constexpr int oR = oAh + (FORCE ? TCELL * LDA : 0);  // [32][LDU]
    static constexpr int oX = oR + (VOL ? TCELL * LDU : 0);     // [NX][n][32]
    static constexpr int total = oX + NX * n * 32;
    // the momentum components v = v0, v0 + n.. of warp w, as in the isothermal kernel
    __device__ static constexpr int v0(int w) { return K == 3 ? (w == 0 ? 4 : w) : w + 1; }
    static_assert(NP * n * 32 >= TCELL * LDH, "a projected row fits its entries");
    static_assert(total * (int)sizeof(T) >= NT * 8, "reduction buffer");
};

// Bound: instruction issue.  Fluxes, source and projections are separate passes over
// the plane's rows: together their 94 (134 driven) partial sums would not fit the
// registers at three blocks per SM.
template <typename T, int K, int MODE, bool FORCE, bool PROJ>
__global__ void __launch_bounds__(32 * (K + 1), sizeof(T) == 4 ? (K == 3 ? 3 : K == 2 ? 4 : 8) : 1)
    k_sfa_vol(const __grid_constant__ AArgs<T> a)
{
    grid_dependency();
    using C = AVolCfg<T, K, MODE, FORCE, PROJ>;
    constexpr bool VOL = C::VOL, SRC = C::SRC;
    constexpr int b = C::b, n = C::n, NT = C::NT, NP = C::NP, NPD = C::NPD, LDU = C::LDU, LDA = C::LDA, LDH = C::LDH;
    constexpr G1<K> G{};
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    T* sAh = sm + C::oAh;
    T* sR = sm + C::oR;
    T* sX = sm + C::oX;
    __shared__ T s_dt;
    __shared__ unsigned long long s_smax;
    __shared__ double s_tot[8];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const long ntile = (a.ncell + TCELL - 1) / TCELL;
    const T g1 = a.gas.g1, c0g = a.gas.c0;
    auto fetch = [&](long tile, int buf) {
        tile_async<T, 5 * b, LDU, NT, chunk<T, 5 * b>()>(sm + C::oU + buf * TCELL * LDU, a.u_in, tile * TCELL, a.ncell);
        cp_async_commit();
    };
    if (blockIdx.x < ntile) fetch(blockIdx.x, 0);
    double dtd = a.dt_pimax;  // (thread 0)
    if (tid == 0) {
        s_smax = 0ull;
        if constexpr (VOL) {
            if (a.stage) {
                // the step's dt: CFL bound of u^n, prescribed dt, retry factor
                const double smax = __longlong_as_double((long long)a.ctl->smax);
                dtd = (a.ctl->fixed_dt > 0.0 ? a.ctl->fixed_dt : a.ctl->dt_num / smax) * a.ctl->dt_scale;
                if (blockIdx.x == 0) a.ctl->dt = dtd;
            }
            s_dt = dtd > 0.0 ? T(0.5 * a.hp * a.hp / dtd) : T(-1);
        }
    }
    T pz[n], dz[n];
#pragma unroll
    for (int l = 0; l < n; ++l) pz[l] = dz[l] = T(0);
    static_for<0, n>([&](auto C_) {
        constexpr int c = decltype(C_)::value;
        if (w == c) {
            static_for<0, n>([&](auto L) {
                constexpr int l = decltype(L)::value;
                pz[l] = T(G.P[l][c]);
                dz[l] = T(G.D[l][c]);
            });
        }
    });
    T smax = T(0);
    // FP64 sums of the thread's cells: warp w < 3: <rho a_h>_w and <m_w> (fewer warps:
    // component 2 in the second set); warp 0: <rho>, <m.a_h>; reset: thermal energy taken out
    double sa = 0.0, sm0 = 0.0, sa2 = 0.0, sm2 = 0.0, srho = 0.0, swork = 0.0, diss = 0.0;
    __syncthreads();
    const T cap = VOL ? s_dt : T(0);
    int cur = 0;
    for (long tile = blockIdx.x; tile < ntile; tile += gridDim.x, cur ^= 1) {
        const long c0 = tile * TCELL;
        const int nvalid = (int)((a.ncell - c0) < TCELL ? (a.ncell - c0) : TCELL);
        const bool valid = lane < nvalid;
        cp_async_wait<0>();
        __syncthreads();
        if constexpr (FORCE) {
            tile_async<T, 3 * b, LDA, NT, chunk<T, 3 * b>()>(sAh, a.ahat, c0, a.ncell);
            cp_async_commit();
        }
        if (tile + gridDim.x < ntile)
            fetch(tile + gridDim.x, cur ^ 1);
        else
            cp_async_commit();
        const T* sU = sm + C::oU + cur * TCELL * LDU + lane * LDU;
        constexpr int NF = MODE == SFA_RESET ? 4 : 5;
        T A[NF][NP];
        static_for<0, NF>([&](auto F) {
            constexpr int f = decltype(F)::value;
            T uu[b];
            ld_row<T, b>(sU + f * b, uu);
            plane_eval<T, K>(uu, pz, A[f]);
        });
        auto store_sums = [&](auto N_, auto M_, const T* S, int e0) {
            constexpr int nn = decltype(N_)::value, m = decltype(M_)::value;
#pragma unroll
            for (int f = 0; f < nn; ++f)
#pragma unroll
                for (int e = 0; e < m; ++e) sX[((e0 + f * m + e) * n + w) * 32 + lane] = S[f * m + e];
        };
        if constexpr (FORCE) {
            cp_async_wait<1>();
            __syncthreads();
            const T* ah = sAh + lane * LDA;
            auto dot = [&](int i) {
                T s = T(0), x[b], y[b];
                ld_row<T, b>(sU, x);
                ld_row<T, b>(ah + i * b, y);
#pragma unroll
                for (int l = 0; l < b; ++l) s += x[l] * y[l];
                return (double)s;
            };
            if (valid) {
                if (PROJ && w < 3) sa += dot(w);
                if (PROJ && n < 3 && w == 0) sa2 += dot(2);
                if (PROJ && w == 0) srho += (double)sU[0];
                if (VOL && w < 3) sm0 += (double)sU[(1 + w) * b];
                if (VOL && n < 3 && w == 0) sm2 += (double)sU[3 * b];
            }
            if constexpr (SRC) {
                // source rho a_h and its work m.a_h
                T Aa[3][NP], S[4 * NP];
                static_for<0, 3>([&](auto F) {
                    constexpr int f = decltype(F)::value;
                    T uu[b];
                    ld_row<T, b>(ah + f * b, uu);
                    plane_eval<T, K>(uu, pz, Aa[f]);
                });
#pragma unroll
                for (int e = 0; e < 4 * NP; ++e) S[e] = T(0);
#pragma unroll 1
                for (int B = 0; B < n; ++B) {
                    const T *pj = a.rows.P[B], *wj = a.rows.W[B];
                    T r[n], rho[n], wk[n], t[n];
                    row_eval<T, K>(A[0], pj, r);
                    line_eval<T, K, K, false>(r, rho);
                    static_for<0, 3>([&](auto F) {
                        constexpr int f = decltype(F)::value;
                        T v[n], m[n];
                        row_eval<T, K>(Aa[f], pj, r);
                        line_eval<T, K, K, false>(r, v);
                        row_eval<T, K>(A[1 + f], pj, r);
                        line_eval<T, K, K, false>(r, m);
#pragma unroll
                        for (int i = 0; i < n; ++i) {
                            wk[i] = f == 0 ? m[i] * v[i] : wk[i] + m[i] * v[i];
                            v[i] *= rho[i];
                        }
                        line_proj<T, K, K>(v, t);
                        row_acc<T, K>(t, wj, S + f * NP);
                    });
                    line_proj<T, K, K>(wk, t);
                    row_acc<T, K>(t, wj, S + 3 * NP);
                }
                store_sums(std::integral_constant<int, 4>{}, std::integral_constant<int, NP>{}, S, 0);
                __syncthreads();
                // the threads that add the flux part to these rows below
#pragma unroll 1
                for (int v = C::v0(w); v < 4; v += n) {
                    T q[b];
                    z_project<T, K, K>(sX + (v - 1) * NP * n * 32, lane, q);
                    st_row<T, b>(sR + lane * LDU + v * b, q);
                }
                if (w == 0) {
                    T q[b];
                    z_project<T, K, K>(sX + 3 * NP * n * 32, lane, q);
                    st_row<T, b>(sR + lane * LDU + 4 * b, q);
                    if (valid) swork += (double)q[0];  // cell mean of m.a_h
                }
                __syncthreads();
            }
        }
        // ---- fluxes ----
        if constexpr (VOL) {
            T Fx[9 * NPD];  // sums of xx, yy, zz, xy, xz, yz and the energy flux x, y, z
#pragma unroll
            for (int e = 0; e < 9 * NPD; ++e) Fx[e] = T(0);
            T Az[NPD], Mz[NPD];
            {
                T uu[b];
                ld_row<T, b>(sU, uu);
                plane_deriv<T, K>(uu, dz, Az);
                ld_row<T, b>(sU + 3 * b, uu);
                plane_deriv<T, K>(uu, dz, Mz);
            }
#pragma unroll 1
            for (int B = 0; B < n; ++B) {
                const T *pj = a.rows.P[B], *dj = a.rows.D[B], *wj = a.rows.W[B];
                T f[5][n];
                T gx[n], gy[n], gz[n], dm[n];
                static_for<0, 5>([&](auto F) {
                    constexpr int v = decltype(F)::value;
                    T r[n];
                    row_eval<T, K>(A[v], pj, r);
                    line_eval<T, K, K, false>(r, f[v]);
                    if constexpr (v == 0) line_eval<T, K, K, true>(r, gx);
                    if constexpr (v == 1) line_eval<T, K, K, true>(r, dm);
                });
                {
                    T r[n], s[n], t[n];
                    row_deriv<T, K>(A[0], dj, r);
                    line_eval<T, K, K - 1, false>(r, gy);
                    row_eval<T, K - 1>(Az, pj, r);
                    line_eval<T, K, K - 1, false>(r, gz);
                    row_deriv<T, K>(A[2], dj, r);
                    row_eval<T, K - 1>(Mz, pj, s);
#pragma unroll
                    for (int i = 0; i < K; ++i) r[i] += s[i];
                    line_eval<T, K, K - 1, false>(r, t);
#pragma unroll
                    for (int i = 0; i < n; ++i) dm[i] += t[i];
                }
                T P[n], vx[n], vy[n], vz[n];
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const T rho = f[0][i], ir = rcp<T>(rho);
                    vx[i] = f[1][i] * ir;
                    vy[i] = f[2][i] * ir;
                    vz[i] = f[3][i] * ir;
                    const T p = g1 * (f[4][i] - T(0.5) * (f[1][i] * vx[i] + f[2][i] * vy[i] + f[3][i] * vz[i])) +
                                c0g * rho;
                    P[i] = p;
                    if (a.av_mode == 1) {
                        // viscous pressure (Sec. 3.1) with the local sound speed, A = -div v
                        const T Ad = (vx[i] * gx[i] + vy[i] * gy[i] + vz[i] * gz[i] - dm[i]) * (ir * a.two_h);
                        const T ra = rho * Ad;
                        T Pi = ra * (a.a2 * Ad + a.bh * fast_sqrt<T>(a.gas.gamma * p * ir));
                        if (cap >= T(0)) {
                            const T Pm = ra * cap;
                            Pi = Pi > Pm ? Pm : Pi;
                        }
                        P[i] += Ad > T(0) ? Pi : T(0);
                    }
                    f[4][i] += P[i];
                }
                auto comp = [&](auto G_, const T* p, const T* q, bool diag) {
                    constexpr int g = decltype(G_)::value;
                    T x[n], t[n];
#pragma unroll
                    for (int i = 0; i < n; ++i) x[i] = diag ? p[i] * q[i] + P[i] : p[i] * q[i];
                    line_proj<T, K, K - 1>(x, t);
                    row_acc<T, K - 1>(t, wj, Fx + g * NPD);
                };
                comp(std::integral_constant<int, 0>{}, f[1], vx, true);
                comp(std::integral_constant<int, 1>{}, f[2], vy, true);
                comp(std::integral_constant<int, 2>{}, f[3], vz, true);
                comp(std::integral_constant<int, 3>{}, f[1], vy, false);
                comp(std::integral_constant<int, 4>{}, f[1], vz, false);
                comp(std::integral_constant<int, 5>{}, f[2], vz, false);
                comp(std::integral_constant<int, 6>{}, f[4], vx, false);
                comp(std::integral_constant<int, 7>{}, f[4], vy, false);
                comp(std::integral_constant<int, 8>{}, f[4], vz, false);
            }
            store_sums(std::integral_constant<int, 9>{}, std::integral_constant<int, NPD>{}, Fx, 0);
            __syncthreads();
            // volume term (2/h) sum_d D_d^T Fhat_d
            auto grad3 = [&](int cx, int cy, int cz, T* r) {
                T q[b];
                z_project<T, K, K - 1>(sX + cx * NPD * n * 32, lane, q);
                modal_grad_T_acc<T, K, 0>(q, r, a.two_h);
                z_project<T, K, K - 1>(sX + cy * NPD * n * 32, lane, q);
                modal_grad_T_acc<T, K, 1>(q, r, a.two_h);
                z_project<T, K, K - 1>(sX + cz * NPD * n * 32, lane, q);
                modal_grad_T_acc<T, K, 2>(q, r, a.two_h);
            };
            // rows v of the momentum, then (warp 0) the energy and the density
#pragma unroll 1
            for (int v = K == 3 ? (w == 0 ? 4 : w) : w + 1; v < 5; v += n) {
                T r[b];
                if constexpr (SRC) {
                    // written by this thread, except the work by warp 0
                    ld_row<T, b>(sR + lane * LDU + v * b, r);
                } else {
#pragma unroll
                    for (int l = 0; l < b; ++l) r[l] = T(0);
                }
                const int cx = v == 4 ? 6 : (v == 1 ? 0 : v + 1);
                const int cy = v == 4 ? 7 : (v == 1 ? 3 : (v == 2 ? 1 : 5));
                const int cz = v == 4 ? 8 : (v == 3 ? 2 : v + 3);
                grad3(cx, cy, cz, r);
                st_row<T, b>(sR + lane * LDU + v * b, r);
            }
            if (w == n - 1) {
                T r[b], q[b];
#pragma unroll
                for (int l = 0; l < b; ++l) r[l] = T(0);
                ld_row<T, b>(sU + b, q);
                modal_grad_T_acc<T, K, 0>(q, r, a.two_h);
                ld_row<T, b>(sU + 2 * b, q);
                modal_grad_T_acc<T, K, 1>(q, r, a.two_h);
                ld_row<T, b>(sU + 3 * b, q);
                modal_grad_T_acc<T, K, 2>(q, r, a.two_h);
                st_row<T, b>(sR + lane * LDU, r);
            }
            __syncthreads();
            tile_store<T, 5 * b, LDU, NT>(a.out, sR, c0, nvalid);
        }
        // ---- projections (or the reset's energy) ----
        if constexpr (C::NV > 0) {
            T Vx[C::NV * NP];
#pragma unroll
            for (int e = 0; e < C::NV * NP; ++e) Vx[e] = T(0);
#pragma unroll 1
            for (int B = 0; B < n; ++B) {
                const T *pj = a.rows.P[B], *wj = a.rows.W[B];
                T f[NF][n], t[n];
                static_for<0, NF>([&](auto F) {
                    constexpr int v = decltype(F)::value;
                    T r[n];
                    row_eval<T, K>(A[v], pj, r);
                    line_eval<T, K, K, false>(r, f[v]);
                });
                if constexpr (MODE == SFA_RESET) {
                    T x[n];
#pragma unroll
                    for (int i = 0; i < n; ++i)
                        x[i] = f[0][i] * a.gas.cres +
                               T(0.5) * (f[1][i] * f[1][i] + f[2][i] * f[2][i] + f[3][i] * f[3][i]) * rcp<T>(f[0][i]);
                    line_proj<T, K, K>(x, t);
                    row_acc<T, K>(t, wj, Vx);
                } else {
#pragma unroll
                    for (int i = 0; i < n; ++i) {
                        const T rho = f[0][i], ir = rcp<T>(rho);
                        const T vx = f[1][i] * ir, vy = f[2][i] * ir, vz = f[3][i] * ir;
                        // projected: p - c0 rho
                        const T pd = g1 * (f[NF - 1][i] - T(0.5) * (f[1][i] * vx + f[2][i] * vy + f[3][i] * vz));
                        f[1][i] = vx;
                        f[2][i] = vy;
                        f[3][i] = vz;
                        f[NF - 1][i] = pd;
                        if (MODE == SFA_PROJECT && a.dtf && valid) {
                            const T cs = rounded_sqrt<T>(a.gas.gamma * (pd + c0g * rho) * ir);
                            const T sp = fabs(f[1][i]) + fabs(f[2][i]) + fabs(f[3][i]) + T(3) * cs;
                            smax = sp > smax ? sp : smax;
                        }
                    }
                    static_for<0, 4>([&](auto V_) {
                        constexpr int v = decltype(V_)::value;
                        line_proj<T, K, K>(f[1 + v], t);
                        row_acc<T, K>(t, wj, Vx + v * NP);
                    });
                }
            }
            // (VOL: every warp has read the flux sums at the last barrier)
            store_sums(std::integral_constant<int, C::NV>{}, std::integral_constant<int, NP>{}, Vx, 0);
            __syncthreads();
#pragma unroll 1
            for (int v = w; v < C::NV; v += n) {
                T q[b];
                T* X = sX + v * NP * n * 32;
                z_project<T, K, K>(X, lane, q);
                if constexpr (MODE == SFA_RESET) {
                    if (valid) diss += (double)sU[4 * b] - (double)q[0];
                }
                __syncwarp();
                st_row<T, b>(X + lane * LDH, q);
            }
            __syncthreads();
            // rows of component v at sX + v NP n 32
            constexpr int CS = NP * n * 32, OS = MODE == SFA_RESET ? 5 : 4, O0 = MODE == SFA_RESET ? 4 : 0;
            constexpr int CH = chunk<T, b>(), V = CH / (int)sizeof(T), NCB = b / V, NCH = C::NV * NCB;
            T* g = (MODE == SFA_RESET ? a.out : a.pr_out) + (c0 * OS + O0) * b;
            if ((reinterpret_cast<uintptr_t>(g) & (CH - 1)) == 0) {
                for (int e = tid; e < nvalid * NCH; e += NT) {
                    const int c = e / NCH, ch = e - c * NCH, i = ch / NCB, o = ch - i * NCB;
                    const T* s = sX + i * CS + c * LDH + o * V;
                    T* q = g + (c * OS + i) * b + o * V;
                    if constexpr (CH == 16)
                        *reinterpret_cast<uint4*>(q) = *reinterpret_cast<const uint4*>(s);
                    else
                        *reinterpret_cast<uint2*>(q) = *reinterpret_cast<const uint2*>(s);
                }
            } else {
                for (int e = tid; e < nvalid * C::NV * b; e += NT) {
                    const int c = e / (C::NV * b), i = (e / b) % C::NV, l = e % b;
                    g[(c * OS + i) * b + l] = sX[i * CS + c * LDH + l];
                }
            }
        }
    }
    // ---- block sums, then the last block of the launch ----
    cp_async_wait<0>();
    __syncthreads();
    double* s_buf = reinterpret_cast<double*>(smem_raw);
    if (MODE == SFA_PROJECT && a.dtf) {
        const double sp = (double)warp_max(smax);
        if (lane == 0) atomicMax(&s_smax, (unsigned long long)__double_as_longlong(sp));
        __syncthreads();
        if (tid == 0) atomicMax(&a.ctl->smax, s_smax);
    }
    if constexpr (FORCE || MODE == SFA_RESET) {
        double mine[8];
        // per warp by shuffles, the warps' sums in s_buf[0..n)
        auto reduce = [&](double v, double* dst, int cnt) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) s_buf[w] = v;
            __syncthreads();
            if (tid == 0)
                for (int j = 0; j < cnt; ++j) dst[j] = s_buf[j];
            __syncthreads();
        };
        if constexpr (MODE == SFA_RESET) {
            double d[n];
            reduce(diss, d, n);
            if (tid == 0) mine[0] = d[0];  // component 0 is warp 0's
            if (last_block_reduce<NT>(a.partials + 8 * kMaxGrid, mine, 1, &a.ctl->cnt_diag, s_tot) && tid == 0)
                a.ctl->work[1] += s_tot[0] * a.h3;
        } else {
            // 0-2 <rho a_h>, 3 <rho>, 4 <m.a_h>, 5-7 <m>
            constexpr int nc = n < 3 ? n : 3;
            for (int i = 0; i < 8; ++i) mine[i] = 0.0;
            double d[n];
            if constexpr (PROJ) {
                reduce(sa, mine, nc);
                if constexpr (n < 3) {
                    reduce(sa2, d, 1);
                    if (tid == 0) mine[2] = d[0];
                }
                reduce(srho, d, 1);
                if (tid == 0) mine[3] = d[0];
            }
            if constexpr (VOL) {
                reduce(swork, d, 1);
                if (tid == 0) mine[4] = d[0];
                reduce(sm0, mine + 5, nc);
                if constexpr (n < 3) {
                    reduce(sm2, d, 1);
                    if (tid == 0) mine[7] = d[0];
                }
            }
            if (last_block_reduce<NT>(a.partials, mine, VOL ? 8 : 4, &a.ctl->cnt_proj, s_tot) && tid == 0) {
                double ab[3];
                for (int i = 0; i < 3; ++i) ab[i] = PROJ ? s_tot[i] / s_tot[3] : a.ctl->abar2[a.abar_in][i];
                if (PROJ)
                    for (int i = 0; i < 3; ++i) a.ctl->abar2[a.abar_out][i] = ab[i];
                if (VOL && a.stage)
                    a.ctl->work[0] += a.beta * dtd * a.h3 *
                                      (s_tot[4] - ab[0] * s_tot[5] - ab[1] * s_tot[6] - ab[2] * s_tot[7]);
            }
        }
    }
}

template <typename T, int K>
struct AFaceCfg {
    static constexpr int b = Dims<K>::b, NP = npair(K), NT = 128;
    static constexpr int LD = padded<T>(5 * b);  // rows rho, v, p (operands) and rho, m, e (states)
    static constexpr int REG = TCELL * LD;
    static constexpr int oFlux = 3 * REG;  // [variable][pair][face]
    static constexpr int total = oFlux + 5 * NP * 128;
};

// The bricks of k_sf_faces, with warps 0-2 on the + faces along x, y, z and warp 3 on the
// lower faces (BrickFaces here took degree 2 with HLLC from 0.81 to 0.80 ms and degree 3
// from 2.53 to 2.60).  Boundary faces take a ghost trace: the cell's own (outflow), with
// the normal velocity negated (reflective), or the prescribed inflow
// state at the faces at coordinate 0.
// Blocks per SM in FP32: degree 1 6 (96^3: 0.440 ms a step; 5: 0.458), degree 2 4 with
// HLLC (48^3 with reset, 2 steps: 0.81 ms; 3: 0.83) and 3 with Rusanov, whose flux
// spills at 4 (88^3: 1.42 ms a step; 4: 1.45), degree 3 2 (64^3, 2 steps: 2.53 ms; 3: 2.85).
template <typename T, int K, int RS, bool STAGE>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? (K == 1 ? 6 : K == 2 ? (RS == 2 ? 4 : 3) : 2) : 1)
    k_sfa_faces(const __grid_constant__ AArgs<T> a)
{
    grid_dependency();
    using C = AFaceCfg<T, K>;
    constexpr int b = C::b, n = K + 1, NP = C::NP, LD = C::LD, nq = n * n * n, nf = 6 * n * n;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    __shared__ T s_bound[5][2][TCELL];  // mean and bound of the higher modes per variable and cell
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int N = a.N;
    const Brick brick(blockIdx.x, N);
    const int x0 = brick.x0, y0 = brick.y0, z0 = brick.z0;
    const int rs = tid >> 2, sub = tid & 3;
    const int ri = rs & 3, rj = (rs >> 2) & 3, rk = rs >> 4;
    const long rcell = brick.cell(ri, rj, rk), own = brick.own(rs);
    {
        constexpr int CH = chunk<T, b>(), V = CH / (int)sizeof(T), NB = b / V, NR = 5 * NB;
        auto copy_row = [&](T* dst, long c) {
            const T* ru = a.u_in + c * 5 * b;
            const T* rv = a.pr_in + c * 4 * b - b;  // chunk ch >= NB: v, p
#pragma unroll
            for (int k = 0; k < (NR + 3) / 4; ++k) {
                const int ch = sub + 4 * k;
                if (NR % 4 == 0 || ch < NR) cp_async<CH>(dst + ch * V, (ch < NB ? ru : rv) + ch * V);
            }
        };
        copy_row(sm + rs * LD, rcell);
        const int hs = rs >> 3, h0 = rs & 3, h1 = (rs >> 2) & 1;
        copy_row(sm + (32 + rs) * LD, hs < 2 ? brick.cell(hs ? 4 : -1, h0, h1) : brick.cell(h0, hs == 3 ? 4 : -1, h1));
        copy_row(sm + (64 + rs) * LD, brick.cell(ri, rj, rk ? 2 : -1));
        cp_async_commit();
    }
    int d, rowL, rowR;
    bool up = false;  // the face is the mesh's upper boundary along d
    {
        const int i = lane & 3, j = (lane >> 2) & 3, k = lane >> 4;
        if (w < 3) {
            d = w;
            rowL = lane;
            rowR = w == 0 ? (i < 3 ? lane + 1 : 40 + 4 * k + j)
                          : (w == 1 ? (j < 3 ? lane + 4 : 56 + 4 * k + i) : (k < 1 ? lane + 16 : 80 + 4 * j + i));
            up = (w == 0 ? x0 + i : (w == 1 ? y0 + j : z0 + k)) == N - 1;
        } else if (lane < 16) {
            d = lane >> 3;
            const int e0 = lane & 3, e1 = (lane >> 2) & 1;
            rowL = 32 + 16 * d + (lane & 7);
            rowR = d == 0 ? 16 * e1 + 4 * e0 : 16 * e1 + e0;
        } else {
            d = 2;
            rowL = 64 + lane - 16;
            rowR = lane - 16;
        }
    }
    const int bcd = d == 0 ? a.bc[0] : (d == 1 ? a.bc[1] : a.bc[2]);
    const bool down = w == 3 && (d == 0 ? x0 : (d == 1 ? y0 : z0)) == 0;
    const T dt = STAGE ? T(a.ctl->dt) : T(0);
    const bool fix = a.ahat != nullptr;
    cp_async_wait<0>();
    __syncthreads();
    T c2[10][NP];
    {
        const T* Lp = sm + rowL * LD;
        const T* Rp = sm + rowR * LD;
        auto traces = [&](auto D_) {
            constexpr int Dd = decltype(D_)::value;
            constexpr int t1 = Dd == 0 ? 1 : 0, t2 = Dd == 2 ? 1 : 2;
            constexpr int fld[5] = {0, 1 + Dd, 1 + t1, 1 + t2, 4};
            static_for<0, 5>([&](auto F) {
                constexpr int f = decltype(F)::value;
                T uu[b];
                ld_row<T, b>(Lp + fld[f] * b, uu);
                trace<T, K, Dd, 1>(uu, c2[f]);
                ld_row<T, b>(Rp + fld[f] * b, uu);
                trace<T, K, Dd, 0>(uu, c2[5 + f]);
            });
        };
        if (d == 0)
            traces(std::integral_constant<int, 0>{});
        else if (d == 1)
            traces(std::integral_constant<int, 1>{});
        else
            traces(std::integral_constant<int, 2>{});
    }
    if (bcd != DG_BC_PERIODIC && (up || down)) {
        const T sg = bcd == DG_BC_REFLECT ? T(-1) : T(1);
        const T in[5] = {a.inflow[0], d == 0 ? a.inflow[1] : (d == 1 ? a.inflow[2] : a.inflow[3]),
                         d == 0 ? a.inflow[2] : a.inflow[1], d == 2 ? a.inflow[2] : a.inflow[3], a.inflow[4]};
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            const T s = f == 1 ? sg : T(1);
#pragma unroll
            for (int e = 0; e < NP; ++e) {
                if (up)
                    c2[5 + f][e] = s * c2[f][e];
                else if (bcd == DG_BC_INFLOW)
                    c2[f][e] = e == 0 ? in[f] : T(0);
                else
                    c2[f][e] = s * c2[5 + f][e];
            }
        }
    }
    __syncthreads();
    constexpr int CHU = chunk<T, 5 * b>(), VU = CHU / (int)sizeof(T), NCU = 5 * b / VU;
    const bool out16 = (reinterpret_cast<uintptr_t>(a.out) & (CHU - 1)) == 0;
    // the rows of the brick's own cells (see k_sf_faces)
    if (own >= 0) {
        auto copy_state = [&](T* dst, const T* src) {
            const T* s = src + own * 5 * b;
            T* q = dst + rs * LD;
#pragma unroll
            for (int k = 0; k < (NCU + 3) / 4; ++k)
                if (NCU % 4 == 0 || sub + 4 * k < NCU) cp_async<CHU>(q + (sub + 4 * k) * VU, s + (sub + 4 * k) * VU);
        };
        copy_state(sm, a.u_in);
        if (out16) {
            copy_state(sm + C::REG, a.out);
        } else {
            for (int e = sub; e < 5 * b; e += 4) sm[C::REG + rs * LD + e] = a.out[own * 5 * b + e];
        }
        if (STAGE && a.rk_a != T(0)) copy_state(sm + 2 * C::REG, a.u_n);
    }
    cp_async_commit();
    {
        T fx[5][NP];
#pragma unroll
        for (int f = 0; f < 5; ++f)
#pragma unroll
            for (int e = 0; e < NP; ++e) fx[f][e] = T(0);
#pragma unroll 1
        for (int B = 0; B < n; ++B) {
            const T *pj = a.rows.P[B], *wj = a.rows.W[B];
            T W[10][n];
            static_for<0, 10>([&](auto F) {
                constexpr int f = decltype(F)::value;
                T r[n];
                row_eval<T, K>(c2[f], pj, r);
                line_eval<T, K, K, false>(r, W[f]);
            });
            T Fl[5][n];
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const T WL[5] = {W[0][i], W[1][i], W[2][i], W[3][i], W[4][i]};
                const T WR[5] = {W[5][i], W[6][i], W[7][i], W[8][i], W[9][i]};
                T F[5];
                if constexpr (RS == 2)
                    adi_hllc<T>(a.gas, WL, WR, F);
                else
                    adi_rusanov<T>(a.gas, WL, WR, F);
#pragma unroll
                for (int v = 0; v < 5; ++v) Fl[v][i] = F[v];
            }
            static_for<0, 5>([&](auto F) {
                constexpr int f = decltype(F)::value;
                T t[n];
                line_proj<T, K, K>(Fl[f], t);
                row_acc<T, K>(t, wj, fx[f]);
            });
        }
        const int v1 = 1 + d, v2 = d == 0 ? 2 : 1, v3 = d == 2 ? 2 : 3;
        T* X = sm + C::oFlux + tid;
#pragma unroll
        for (int e = 0; e < NP; ++e) {
            X[e * 128] = fx[0][e];
            X[(v1 * NP + e) * 128] = fx[1][e];
            X[(v2 * NP + e) * 128] = fx[2][e];
            X[(v3 * NP + e) * 128] = fx[3][e];
            X[(4 * NP + e) * 128] = fx[4][e];
        }
    }
    cp_async_wait<0>();
    __syncthreads();
    // ---- right-hand side of the variables v = w, w + 4: surface term + volume term ----
    unsigned int st = 0u;
    const int ci = lane & 3, cj = (lane >> 2) & 3, ck = lane >> 4;
    T ab[3] = {T(0), T(0), T(0)};
    if (fix)
        for (int i = 0; i < 3; ++i) ab[i] = T(a.ctl->abar2[a.abar_in][i]);
    T rr[2][b];
#pragma unroll
    for (int vi = 0; vi < 2; ++vi) {
        const int v = w + 4 * vi;
        if (v > 4) break;
        T* r = rr[vi];
#pragma unroll
        for (int l = 0; l < b; ++l) r[l] = T(0);
        static_for<0, 3>([&](auto D_) {
            constexpr int Dd = decltype(D_)::value;
            const T* X = sm + C::oFlux + v * NP * 128;
            const T* Xp = X + 32 * Dd + lane;
            const T* Xm = X + (Dd == 0 ? (ci > 0 ? lane - 1 : 96 + 4 * ck + cj)
                                       : (Dd == 1 ? (cj > 0 ? 32 + lane - 4 : 104 + 4 * ck + ci)
                                                  : (ck > 0 ? 64 + lane - 16 : 112 + 4 * cj + ci)));
            static_for<0, K + 1>([&](auto I) {
                constexpr int p = decltype(I)::value;
                static_for<0, K - p + 1>([&](auto J) {
                    constexpr int q = decltype(J)::value;
                    const T xm = Xm[ip(K, p, q) * 128], xp = Xp[ip(K, p, q) * 128];
                    const T ev = xm - xp, od = -(xm + xp);
                    static_for<0, K - p - q + 1>([&](auto L) {
                        constexpr int dn = decltype(L)::value;
                        constexpr int m = Dd == 0 ? im<K>(dn, p, q) : (Dd == 1 ? im<K>(p, dn, q) : im<K>(p, q, dn));
                        DG_SF_MAC(T, r[m], csqrt(2.0 * dn + 1.0), ((dn & 1) ? od : ev), false);
                    });
                });
            });
        });
        T x[b];
        ld_row<T, b>(sm + lane * LD + v * b + C::REG, x);  // volume term
#pragma unroll
        for (int l = 0; l < b; ++l) r[l] = r[l] * a.inv_h + x[l];
        if (fix && v > 0) {
            // the source's mean-acceleration part: -abar_i rho_l; its work: -abar.m_l
            if (v < 4) {
                const T s = v == 1 ? ab[0] : (v == 2 ? ab[1] : ab[2]);
                ld_row<T, b>(sm + lane * LD, x);
#pragma unroll
                for (int l = 0; l < b; ++l) r[l] -= s * x[l];
            } else {
                for (int i = 0; i < 3; ++i) {
                    ld_row<T, b>(sm + lane * LD + (1 + i) * b, x);
#pragma unroll
                    for (int l = 0; l < b; ++l) r[l] -= ab[i] * x[l];
                }
            }
        }
    }
    // every warp has read rho and m before the results replace them
    if (fix) __syncthreads();
#pragma unroll
    for (int vi = 0; vi < 2; ++vi) {
        const int v = w + 4 * vi;
        if (v > 4) break;
        T* r = rr[vi];
        T* row = sm + lane * LD + v * b;
        if constexpr (STAGE) {
            T x[b];
            ld_row<T, b>(row, x);
            if (a.rk_a != T(0)) {
                T y[b];
                ld_row<T, b>(row + 2 * C::REG, y);
#pragma unroll
                for (int l = 0; l < b; ++l) r[l] = a.rk_a * y[l] + a.rk_b * (x[l] + dt * r[l]);
            } else {
#pragma unroll
                for (int l = 0; l < b; ++l) r[l] = a.rk_b * (x[l] + dt * r[l]);
            }
            T part = T(0);
            static_for<1, b>([&](auto M) {
                constexpr int m = decltype(M)::value;
                part += T(sup_phi<K>(m)) * fabs(r[m]);
            });
            s_bound[v][0][lane] = r[0];
            s_bound[v][1][lane] = part;
        }
        st_row<T, b>(row, r);
    }
    __syncthreads();
    if constexpr (STAGE) {
        // ---- positivity of density and pressure (Sec. 3.1) ----
        const T eps = a.eps, g1 = a.gas.g1;
        const bool valid = brick.inside(ci, cj, ck);
        bool check = false;
        if (valid) {
            T ub[5], dl[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                ub[v] = s_bound[v][0][lane];
                dl[v] = s_bound[v][1][lane];
            }
            const T pbar = adi_p<T>(a.gas, ub[0], ub[1], ub[2], ub[3], ub[4]);
            if (!(ub[0] > eps) || !(pbar > eps)) {
                st |= DG_ST_FAIL_;
            } else {
                // sufficient condition on the box ubar +- delta: no point can be below a floor
                bool ok = ub[0] - dl[0] >= eps;
                if (ok) {
                    // rho p = (gamma-1)(rho e_s - |m|^2/2) + c0 rho^2 >= eps rho on the box
                    const T lr = ub[0] - dl[0], ur = ub[0] + dl[0], le = ub[4] - dl[4];
                    T mm2 = T(0);
#pragma unroll
                    for (int i = 1; i < 4; ++i) {
                        const T mi = fabs(ub[i]) + dl[i];
                        mm2 += mi * mi;
                    }
                    const T re = le >= T(0) ? lr * le : ur * le;
                    ok = g1 * (re - T(0.5) * mm2) + a.gas.c0 * lr * lr - eps * ur > T(0);
                }
                check = !ok;
            }
        }
        // exact check at every volume and face point of the cells in question, each by
        // one of the block's warps in turn
        unsigned low = __ballot_sync(0xffffffffu, check);
        for (int k = 0; low; ++k) {
            const int c = __ffs(low) - 1;
            low &= low - 1;
            if ((k & 3) != w) continue;
            T* u = sm + c * LD;
            constexpr int NPT = nq + nf, NPW = (NPT + 31) / 32;
            T ub[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) ub[v] = u[v * b];
            T val[NPW][5];
            T rmin = T(1e30);
#pragma unroll
            for (int j = 0; j < NPW; ++j) {
                const int pt = lane + 32 * j;
#pragma unroll
                for (int v = 0; v < 5; ++v) val[j][v] = ub[v];
                if (pt < NPT) {
                    const T* ph = pt < nq ? a.phiv + pt : a.phif + (pt - nq);
                    const int sp = pt < nq ? nq : nf;
                    T s[5] = {T(0), T(0), T(0), T(0), T(0)};
#pragma unroll 4
                    for (int l = 0; l < b; ++l) {
                        const T p = __ldg(ph + l * sp);
#pragma unroll
                        for (int v = 0; v < 5; ++v) s[v] += u[v * b + l] * p;
                    }
#pragma unroll
                    for (int v = 0; v < 5; ++v) val[j][v] = s[v];
                    rmin = val[j][0] < rmin ? val[j][0] : rmin;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const T other = __shfl_xor_sync(0xffffffffu, rmin, o);
                rmin = other < rmin ? other : rmin;
            }
            const T th_r = rmin < eps ? (ub[0] - eps) / (ub[0] - rmin) : T(1);
            T th_p = T(1);
#pragma unroll
            for (int j = 0; j < NPW; ++j) {
                const int pt = lane + 32 * j;
                if (pt < NPT) {
                    T uq[5], dv[5];
#pragma unroll
                    for (int v = 0; v < 5; ++v) {
                        uq[v] = ub[v] + th_r * (val[j][v] - ub[v]);
                        dv[v] = uq[v] - ub[v];
                    }
                    if (adi_p<T>(a.gas, uq[0], uq[1], uq[2], uq[3], uq[4]) < eps) {
                        const T t = adi_pressure_root<T>(a.gas, eps, ub, dv);
                        th_p = t < th_p ? t : th_p;
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const T other = __shfl_xor_sync(0xffffffffu, th_p, o);
                th_p = other < th_p ? other : th_p;
            }
            const T th = th_r * th_p;
            __syncwarp();
            if (th < T(1)) {
                st |= DG_ST_LIMITED_;
                for (int e = lane; e < 5 * b; e += 32)
                    if (e % b) u[e] *= th;
            }
        }
        __syncthreads();
        if (own >= 0) {
            bool bad = false;
            for (int e = sub; e < 5 * b; e += 4) bad |= !isfinite(sm[rs * LD + e]);
            if (bad) st |= DG_ST_NONFINITE_;
        }
        st = __reduce_or_sync(0xffffffffu, st);
        if (lane == 0 && st) atomicOr(&a.ctl->status, st);
    }
    if (own >= 0) {
        T* g = a.out + own * 5 * b;
        const T* q = sm + rs * LD;
        if (out16) {
#pragma unroll
            for (int k = 0; k < (NCU + 3) / 4; ++k)
                if (NCU % 4 == 0 || sub + 4 * k < NCU) {
                    if constexpr (CHU == 16)
                        *reinterpret_cast<uint4*>(g + (sub + 4 * k) * VU) =
                            *reinterpret_cast<const uint4*>(q + (sub + 4 * k) * VU);
                    else
                        *reinterpret_cast<uint2*>(g + (sub + 4 * k) * VU) =
                            *reinterpret_cast<const uint2*>(q + (sub + 4 * k) * VU);
                }
        } else {
            for (int e = sub; e < 5 * b; e += 4) g[e] = q[e];
        }
    }
}

}  // namespace sf
}  // namespace dg
