// dg_force.cuh -- projection of the driving acceleration of explicit Fourier modes
//   a(x) = sum_m 2 Re(A_m exp(2 pi i k_m . x))   (Sec. 4.2)
//   ahat_l = sum_q (w_q/8) phi_l(xi_q) a(x_q),  x_q = x_c + (h/2) xi_q
// The tensor Gauss rule, the product basis and the plane waves all factor over
// the axes: with the 1D factors
//   G[i_c][kap][m] = sum_a (w_a/2) Pn_m(xi_a) exp(2 pi i kap (i_c + 1/2 + xi_a/2) h)
// a mode's projection is G[ix][kx][i_l] G[iy][ky][j_l] G[iz][kz][l_l], and the sum
// over the modes contracts one axis at a time:
//   Hz[kx, ky][l]    = sum_kz A G[iz][kz][l]           once per plane iz
//   Hy[kx][(j, l)]   = sum_ky G[iy][ky][j] Hz[kx, ky][l]  once per row (iy, iz)
//   ahat[(i, j, l)]  = sum_kx Re(G[ix][kx][i] Hy[kx][(j, l)])  per cell
// For the 61 modes 1 <= |k|^2 <= 9 at degree 3 that is about 480 multiply-adds per
// cell (14.6 thousand when every mode is formed per cell), so the store of the
// coefficients bounds it.  G depends on the mesh and the rule alone: it is built
// once per context, before its first projection (k_force_axis, FP64 arithmetic,
// stored in T).
#pragma once

#include "dg_sf.cuh"

namespace dg {

constexpr int kForceKM = 8;  // |k_d| <= 8 supported
constexpr int kForceNK = 2 * kForceKM + 1;
constexpr int kForceModes = 512;

// the modes as the kernel reads them: kx >= 0 (a mode with kx < 0 stands as its
// conjugate), sorted by (kx, ky, kz); pairs of equal (kx, ky) and groups of equal
// kx as start indices.  Device layout of the 3 kForceModes ints: packed modes
// kx | (ky + 8) << 8 | (kz + 8) << 16, pair starts, group starts.
struct ForceModes {
    int nm, npair, ngroup;
};
constexpr int kForcePairs = kForceModes, kForceGroups = 2 * kForceModes;  // offsets

// sqrt(2m+1) P_m(x) by the three-term recurrence
__device__ __forceinline__ double legendre_pn(int m, double x)
{
    double p0 = 1.0, p1 = x;
    if (m == 0) return 1.0;
    for (int j = 2; j <= m; ++j) {
        const double p2 = ((2.0 * j - 1.0) * x * p1 - (j - 1.0) * p0) / j;
        p0 = p1;
        p1 = p2;
    }
    return sqrt(2.0 * m + 1.0) * p1;
}

template <typename T, int K>
__global__ void __launch_bounds__(256) k_force_axis(Rule1 r, int N, T* G)
{
    constexpr int n = K + 1;
    const int total = N * kForceNK * n;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int m = e % n, kap = (e / n) % kForceNK - kForceKM, ic = e / (n * kForceNK);
        double re = 0.0, im = 0.0;
        const double h = 1.0 / N;
        for (int a = 0; a < n; ++a) {
            const double wp = 0.5 * r.w[a] * legendre_pn(m, r.x[a]);
            double sn, cn;
            sincospi(2.0 * kap * ((ic + 0.5 + 0.5 * r.x[a]) * h), &sn, &cn);
            re += wp * cn;
            im += wp * sn;
        }
        G[2 * e] = T(re);
        G[2 * e + 1] = T(im);
    }
}

template <typename T, int K>
struct ForceCfg {
    static constexpr int b = Dims<K>::b, n = K + 1, NP = sf::npair(K), CELLS = 64, NT = 3 * CELLS;
    static constexpr int NG = kForceKM + 1, NPAIR = NG * kForceNK;  // largest numbers of kx and of (kx, ky)
    static constexpr int RB = 4;                                    // rows whose sums are formed together
    static constexpr int LD = sf::padded<T>(3 * b);
    // shared memory in elements of T, sized by the modes at hand (few of the possible
    // ones in use: several blocks per SM)
    int hz, hy, gx, out, total;
    __host__ __device__ explicit ForceCfg(const ForceModes& fm)
    {
        hz = 0;                                  // [pair][l][v] complex
        hy = hz + fm.npair * n * 3 * 2;          // [row][group][pair (j, l)][v] complex
        gx = hy + RB * fm.ngroup * NP * 3 * 2;   // [group][i][re, im][cell]
        out = (gx + fm.ngroup * n * 2 * CELLS + 3) / 4 * 4;  // [64][3][b]
        total = out + CELLS * LD;
    }
};

// block: rows iy0 .. iy0 + rpb - 1 of the plane iz = blockIdx.y, RB of them at a time
// (their sums over ky are short chains of dependent loads: several rows in flight
// cover the latency), 64 cells at a time.  128^3 cells of degree 3 in FP32, 61 modes:
// 190 us (2.7 TB/s of coefficients); 474 us row by row, 2060 us mode by mode at the
// points.
template <typename T, int K>
__global__ void __launch_bounds__(192) k_force(const T* __restrict__ G, int N, int rpb, ForceModes fm,
                                               const int* __restrict__ modes, const double* __restrict__ amp,
                                               T* __restrict__ ahat)
{
    using C = ForceCfg<T, K>;
    constexpr int b = C::b, n = C::n, NP = C::NP, NT = C::NT, LD = C::LD;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    const C lay(fm);
    T* hz = sm + lay.hz;
    T* hy = sm + lay.hy;
    T* gx = sm + lay.gx;
    T* so = sm + lay.out;
    const int HY = 2 * fm.ngroup * NP * 3;
    __shared__ int s_mode[kForceModes], s_pair[C::NPAIR + 1], s_group[C::NG + 1];
    const int tid = threadIdx.x, iz = blockIdx.y;
    for (int e = tid; e < fm.nm; e += NT) s_mode[e] = modes[e];
    for (int e = tid; e <= fm.npair; e += NT) s_pair[e] = e < fm.npair ? modes[kForcePairs + e] : fm.nm;
    for (int e = tid; e <= fm.ngroup; e += NT) s_group[e] = e < fm.ngroup ? modes[kForceGroups + e] : fm.npair;
    __syncthreads();
    const T* gz = G + (long)iz * kForceNK * n * 2;
    for (int e = tid; e < fm.npair * n * 3; e += NT) {
        const int p = e / (n * 3), l = (e / 3) % n, v = e % 3;
        T re = T(0), im = T(0);
        for (int m = s_pair[p]; m < s_pair[p + 1]; ++m) {
            const T* g = gz + ((s_mode[m] >> 16) * n + l) * 2;
            const T ar = T(2.0 * amp[(m * 3 + v) * 2]), ai = T(2.0 * amp[(m * 3 + v) * 2 + 1]);
            re += ar * g[0] - ai * g[1];
            im += ar * g[1] + ai * g[0];
        }
        hz[2 * e] = re;
        hz[2 * e + 1] = im;
    }
    const int iy1 = min(N, (int)(blockIdx.x + 1) * rpb);
    const int v = tid / C::CELLS, cl = tid % C::CELLS;
    for (int y0 = blockIdx.x * rpb; y0 < iy1; y0 += C::RB) {
        const int nr = min(C::RB, iy1 - y0);
        __syncthreads();
        const int per = fm.ngroup * NP * 3;
        for (int e = tid; e < nr * per; e += NT) {
            const int r = e / per, q = e - r * per, g = q / (NP * 3), pr = (q / 3) % NP, c = q % 3;
            // the pair (j, l) of index pr
            int j = 0, l = pr;
            while (l > K - j) l -= K - j + 1, ++j;
            const T* gy = G + ((long)(y0 + r) * kForceNK * n + j) * 2;
            T re = T(0), im = T(0);
            for (int p = s_group[g]; p < s_group[g + 1]; ++p) {
                const T* y = gy + ((s_mode[s_pair[p]] >> 8) & 255) * n * 2;
                const T hr = hz[2 * ((p * n + l) * 3 + c)], hi = hz[2 * ((p * n + l) * 3 + c) + 1];
                re += y[0] * hr - y[1] * hi;
                im += y[0] * hi + y[1] * hr;
            }
            hy[r * HY + 2 * q] = re;
            hy[r * HY + 2 * q + 1] = im;
        }
        for (int x0 = 0; x0 < N; x0 += C::CELLS) {
            const int nc = min(C::CELLS, N - x0);
            if (N > C::CELLS || y0 == (int)blockIdx.x * rpb) {
                // the chunk's factors along x
                __syncthreads();
                for (int e = tid; e < fm.ngroup * C::CELLS; e += NT) {
                    const int g = e / C::CELLS, c = e % C::CELLS;
                    const int kx = s_mode[s_pair[s_group[g]]] & 255;
                    if (c < nc) {
                        const T* x = G + ((long)((x0 + c) * kForceNK + kx + kForceKM) * n) * 2;
#pragma unroll
                        for (int i = 0; i < 2 * n; ++i) gx[(g * 2 * n + i) * C::CELLS + c] = __ldg(x + i);
                    }
                }
            }
            for (int r = 0; r < nr; ++r) {
                __syncthreads();
                if (cl < nc) {
                    T acc[b];
#pragma unroll
                    for (int l = 0; l < b; ++l) acc[l] = T(0);
                    for (int g = 0; g < fm.ngroup; ++g) {
                        T xr[n], xi[n];
#pragma unroll
                        for (int i = 0; i < n; ++i) {
                            xr[i] = gx[(g * 2 * n + 2 * i) * C::CELLS + cl];
                            xi[i] = gx[(g * 2 * n + 2 * i + 1) * C::CELLS + cl];
                        }
                        const T* H = hy + r * HY + 2 * (g * NP * 3 + v);
                        static_for<0, K + 1>([&](auto J) {
                            constexpr int j = decltype(J)::value;
                            static_for<0, K - j + 1>([&](auto L) {
                                constexpr int l = decltype(L)::value;
                                const T hr = H[sf::ip(K, j, l) * 6], hi = H[sf::ip(K, j, l) * 6 + 1];
                                static_for<0, K - j - l + 1>([&](auto I) {
                                    constexpr int i = decltype(I)::value;
                                    acc[sf::im<K>(i, j, l)] += xr[i] * hr - xi[i] * hi;
                                });
                            });
                        });
                    }
                    sf::st_row<T, b>(so + cl * LD + v * b, acc);
                }
                __syncthreads();
                sf::tile_store<T, 3 * b, LD, NT>(ahat + ((long)iz * N + y0 + r) * N * 3 * b, so, x0, nc);
            }
        }
    }
}

}  // namespace dg
