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
    static constexpr int NPAIR = (kForceKM + 1) * kForceNK;  // largest number of (kx, ky) pairs
    static constexpr int LD = sf::padded<T>(3 * b);
    static constexpr int oHz = 0;                                    // [pair][l][v] complex
    static constexpr int oHy = oHz + NPAIR * n * 3 * 2;              // [group][pair (j, l)][v] complex
    static constexpr int oOut = (oHy + (kForceKM + 1) * NP * 3 * 2 + 3) / 4 * 4;  // [64][3][b]
    static constexpr int total = oOut + CELLS * LD;
};

// block: rows iy0 .. iy0 + rpb - 1 of the plane iz = blockIdx.y
template <typename T, int K>
__global__ void __launch_bounds__(192) k_force(const T* __restrict__ G, int N, int rpb, ForceModes fm,
                                               const int* __restrict__ modes, const double* __restrict__ amp,
                                               T* __restrict__ ahat)
{
    using C = ForceCfg<T, K>;
    constexpr int b = C::b, n = C::n, NP = C::NP, NT = C::NT, LD = C::LD;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    T* hz = sm + C::oHz;
    T* hy = sm + C::oHy;
    T* so = sm + C::oOut;
    const int tid = threadIdx.x, iz = blockIdx.y;
    const int* pairs = modes + kForcePairs;
    const int* groups = modes + kForceGroups;
    const T* gz = G + (long)iz * kForceNK * n * 2;
    for (int e = tid; e < fm.npair * n * 3; e += NT) {
        const int p = e / (n * 3), l = (e / 3) % n, v = e % 3;
        const int m0 = pairs[p], m1 = p + 1 < fm.npair ? pairs[p + 1] : fm.nm;
        T re = T(0), im = T(0);
        for (int m = m0; m < m1; ++m) {
            const T* g = gz + ((modes[m] >> 16) * n + l) * 2;
            const T ar = T(2.0 * amp[(m * 3 + v) * 2]), ai = T(2.0 * amp[(m * 3 + v) * 2 + 1]);
            re += ar * g[0] - ai * g[1];
            im += ar * g[1] + ai * g[0];
        }
        hz[2 * e] = re;
        hz[2 * e + 1] = im;
    }
    const int iy1 = min(N, (int)(blockIdx.x + 1) * rpb);
    for (int iy = blockIdx.x * rpb; iy < iy1; ++iy) {
        __syncthreads();
        const T* gy = G + (long)iy * kForceNK * n * 2;
        for (int e = tid; e < fm.ngroup * NP * 3; e += NT) {
            const int g = e / (NP * 3), pr = (e / 3) % NP, v = e % 3;
            // the pair (j, l) of index pr
            int j = 0, l = pr;
            while (l > K - j) l -= K - j + 1, ++j;
            const int p0 = groups[g], p1 = g + 1 < fm.ngroup ? groups[g + 1] : fm.npair;
            T re = T(0), im = T(0);
            for (int p = p0; p < p1; ++p) {
                const T* y = gy + (((modes[pairs[p]] >> 8) & 255) * n + j) * 2;
                const T hr = hz[2 * ((p * n + l) * 3 + v)], hi = hz[2 * ((p * n + l) * 3 + v) + 1];
                re += y[0] * hr - y[1] * hi;
                im += y[0] * hi + y[1] * hr;
            }
            hy[2 * e] = re;
            hy[2 * e + 1] = im;
        }
        const int v = tid / C::CELLS, cl = tid % C::CELLS;
        T* row = ahat + ((long)iz * N + iy) * N * 3 * b;
        for (int x0 = 0; x0 < N; x0 += C::CELLS) {
            __syncthreads();
            const int ix = x0 + cl;
            if (ix < N) {
                T acc[b];
#pragma unroll
                for (int l = 0; l < b; ++l) acc[l] = T(0);
                for (int g = 0; g < fm.ngroup; ++g) {
                    const int kx = modes[pairs[groups[g]]] & 255;
                    const T* x = G + ((long)(ix * kForceNK + kx + kForceKM) * n) * 2;
                    T xr[n], xi[n];
#pragma unroll
                    for (int i = 0; i < n; ++i) {
                        xr[i] = __ldg(x + 2 * i);
                        xi[i] = __ldg(x + 2 * i + 1);
                    }
                    const T* H = hy + 2 * (g * NP * 3 + v);
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
            const int nc = min(C::CELLS, N - x0);
            sf::tile_store<T, 3 * b, LD, NT>(row, so, x0, nc);
        }
    }
}

}  // namespace dg
