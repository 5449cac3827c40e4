// dg_sf.cuh -- sum-factorised kernels of the right-hand side (FP32 and FP64,
// degrees 1..3): every basis <-> point transform runs axis by axis in the
// registers of one thread, with the 1D basis values as immediates.
//
//   k_sf_vol    volume term of a state -> rvol (Sec. 2.2, first and last terms of
//               eq. weight_evolution; Sec. 3.1 viscous pressure), and/or the
//               Gauss projection of the primitive velocity (Sec. 3.2), the CFL
//               bound and the forcing sums
//   k_sf_faces  face traces, Riemann fluxes, surface term + rvol, then the SSP-RK
//               combine and the positivity rescaling (Sec. 3.1, Sec. 7)
//
// Counts per cell at degree 3: one field to the 64 volume points takes 496
// multiply-adds axis by axis (1280 as a dense product), a flux component back
// onto the degree-2 modes that its derivative needs 328 (dense 1280), a trace on a
// face 124.
//
// Layout of the work: a block takes 32 consecutive cells, lane = cell, so that
// everything a warp branches on is uniform and shared-memory accesses of
// consecutive lanes never conflict (rows are padded to an odd number of 16-byte
// units: 8 lanes of a 16-byte load then fall on 8 distinct groups of banks).  In k_sf_vol warp c
// owns the plane c of Gauss points along z (K+1 warps): it contracts the modes
// along z with its plane's basis values, then walks the rows of points, whose
// fields, fluxes and partial sums along x and y stay in registers; the sums along
// z go through shared memory once per tile.  In k_sf_faces a thread owns a face of a
// brick of 4 x 4 x 2 cells (4 warps): the traces of both sides, the Riemann fluxes and
// their projection stay in its registers, and the faces of a cell meet in shared
// memory once per brick.
//
// A driven SSP-RK3 step of 64^3 cells of degree 3 in FP32 takes 0.96 ms (volume 112 to
// 158, faces 130 us a stage, projection 63), where the dense products of the fused stage
// kernel (dg_tile.cuh) took 5.07; 128^3 of degree 2 3.50 ms for 19.8; one FP64
// right-hand side of 24^3 of degree 3 0.56 ms for 1.79.
#pragma once

#include "dg_brick.cuh"
#include "dg_kernels.cuh"
#include "dg_tile.cuh"

namespace dg {
namespace sf {

// ---------------------------------------------------------------------------
// compile-time 1D tables: Gauss-Legendre rule with K+1 points (closed forms),
// normalised Legendre polynomials and their derivatives at the points
// ---------------------------------------------------------------------------
template <int K>
struct G1 {
    static constexpr int n = K + 1;
    double x[n], w[n], P[n][n], D[n][n];  // P[m][a], D[m][a] = Pn_m'(x_a)
    constexpr G1() : x{}, w{}, P{}, D{}
    {
        if (K == 1) {
            x[1] = csqrt(1.0 / 3.0);
            x[0] = -x[1];
            w[0] = w[1] = 1.0;
        } else if (K == 2) {
            x[2] = csqrt(0.6);
            x[1] = 0.0;
            x[0] = -x[2];
            w[0] = w[2] = 5.0 / 9.0;
            w[1] = 8.0 / 9.0;
        } else {
            const double s = 2.0 / 7.0 * csqrt(1.2), t = csqrt(30.0);
            x[3] = csqrt(3.0 / 7.0 + s);
            x[2] = csqrt(3.0 / 7.0 - s);
            x[1] = -x[2];
            x[0] = -x[3];
            w[0] = w[3] = (18.0 - t) / 36.0;
            w[1] = w[2] = (18.0 + t) / 36.0;
        }
        for (int a = 0; a < n; ++a) {
            double p[n + 1] = {}, d[n + 1] = {};
            p[0] = 1.0;
            p[1] = x[a];
            d[1] = 1.0;
            for (int m = 1; m < K; ++m) {
                p[m + 1] = ((2.0 * m + 1.0) * x[a] * p[m] - m * p[m - 1]) / (m + 1.0);
                d[m + 1] = d[m - 1] + (2.0 * m + 1.0) * p[m];
            }
            for (int m = 0; m <= K; ++m) {
                P[m][a] = csqrt(2.0 * m + 1.0) * p[m];
                D[m][a] = csqrt(2.0 * m + 1.0) * d[m];
            }
        }
    }
};

// pairs (i, j) with i + j <= M, i major
constexpr int npair(int M) { return (M + 1) * (M + 2) / 2; }
constexpr int ip(int M, int i, int j) { return i * (M + 1) - i * (i - 1) / 2 + j; }
// index of the mode (i, j, l) in the library's order
template <int K>
constexpr int im(int i, int j, int l)
{
    constexpr Modes<K> M{};
    for (int m = 0; m < Dims<K>::b; ++m)
        if (M.i[m] == i && M.j[m] == j && M.l[m] == l) return m;
    return -1;
}
constexpr bool is_zero(double v) { return v < 1e-14 && v > -1e-14; }

// acc (+)= C x with the zeros and ones of C resolved at compile time; FIRST:
// acc is not read
#define DG_SF_MAC(T, acc, C, x, FIRST)                  \
    do {                                                \
        constexpr double cc_ = (C);                     \
        if constexpr (FIRST) {                          \
            if constexpr (cc_ == 1.0)                   \
                acc = (x);                              \
            else                                        \
                acc = T(cc_) * (x);                     \
        } else if constexpr (!is_zero(cc_)) {           \
            if constexpr (cc_ == 1.0)                   \
                acc += (x);                             \
            else                                        \
                acc += T(cc_) * (x);                    \
        }                                               \
    } while (0)

// values at the K+1 points of a line from the coefficients r[0..M] of a degree-M
// polynomial (DER: of its derivative, r[0] not read): even and odd parts at a
// pair of points +-x share their products
template <typename T, int K, int M, bool DER>
__device__ __forceinline__ void line_eval(const T* r, T* out)
{
    constexpr G1<K> G{};
    constexpr int n = K + 1, m0 = DER ? 1 : 0;
    static_for<0, (n + 1) / 2>([&](auto A_) {
        constexpr int a = n - 1 - decltype(A_)::value, ma = n - 1 - a;  // a: x >= 0, ma: -x
        if constexpr (M < m0) {
            out[a] = T(0);
            if constexpr (ma != a) out[ma] = T(0);
        } else {
            T e = T(0), o = T(0);
            // even part: m of the parity of m0
            static_for<0, (M - m0) / 2 + 1>([&](auto I) {
                constexpr int i = decltype(I)::value, m = m0 + 2 * i;
                DG_SF_MAC(T, e, DER ? G.D[m][a] : G.P[m][a], r[m], i == 0);
            });
            if constexpr (ma != a && M >= m0 + 1) {
                static_for<0, (M - m0 - 1) / 2 + 1>([&](auto I) {
                    constexpr int i = decltype(I)::value, m = m0 + 1 + 2 * i;
                    DG_SF_MAC(T, o, DER ? G.D[m][a] : G.P[m][a], r[m], i == 0);
                });
                out[a] = e + o;
                out[ma] = e - o;
            } else {
                out[a] = e;
                if constexpr (ma != a) out[ma] = e;
            }
        }
    });
}

// weighted moments t[m] = sum_a (w_a/2) Pn_m(x_a) f[a], m = 0..M
template <typename T, int K, int M>
__device__ __forceinline__ void line_proj(const T* f, T* t)
{
    constexpr G1<K> G{};
    constexpr int n = K + 1;
    T s[(n + 1) / 2], d[(n + 1) / 2];
    static_for<0, (n + 1) / 2>([&](auto A_) {
        constexpr int q = decltype(A_)::value, a = n - 1 - q;
        if constexpr (a != q) {
            s[q] = f[a] + f[q];
            if constexpr (M >= 1) d[q] = f[a] - f[q];
        } else {
            s[q] = f[a];
        }
    });
    static_for<0, M + 1>([&](auto M_) {
        constexpr int m = decltype(M_)::value;
        T acc = T(0);
        static_for<0, (m & 1) ? n / 2 : (n + 1) / 2>([&](auto A_) {
            constexpr int q = decltype(A_)::value, a = n - 1 - q;
            DG_SF_MAC(T, acc, 0.5 * G.w[a] * G.P[m][a], ((m & 1) ? d[q] : s[q]), q == 0);
        });
        t[m] = acc;
    });
}

// The rows of points of a plane or face run as a rolled loop (unrolled, the
// instructions of a tile pass outgrow the instruction cache): the row's basis
// values come from the kernel arguments.
// contraction of the pairs (i, j) of a 2D expansion over j with the row's values
// c[j] (c[0] = 1): r[i], i = 0..M
template <typename T, int M>
__device__ __forceinline__ void row_eval(const T* A, const T* c, T* r)
{
    static_for<0, M + 1>([&](auto I) {
        constexpr int i = decltype(I)::value;
        T acc = A[ip(M, i, 0)];
        static_for<1, M - i + 1>([&](auto J) { acc += c[decltype(J)::value] * A[ip(M, i, decltype(J)::value)]; });
        r[i] = acc;
    });
}
// the same with the row's derivatives d[j] along j: r[i], i = 0..M-1
template <typename T, int M>
__device__ __forceinline__ void row_deriv(const T* A, const T* d, T* r)
{
    static_for<0, M>([&](auto I) {
        constexpr int i = decltype(I)::value;
        T acc = d[1] * A[ip(M, i, 1)];
        static_for<2, M - i + 1>([&](auto J) { acc += d[decltype(J)::value] * A[ip(M, i, decltype(J)::value)]; });
        r[i] = acc;
    });
}
// acc(i, j) += w[j] t[i], i + j <= M, w[j] = (w_B/2) Pn_j(x_B)
template <typename T, int M>
__device__ __forceinline__ void row_acc(const T* t, const T* w, T* acc)
{
    static_for<0, M + 1>([&](auto I) {
        constexpr int i = decltype(I)::value;
        static_for<0, M - i + 1>(
            [&](auto J) { acc[ip(M, i, decltype(J)::value)] += w[decltype(J)::value] * t[i]; });
    });
}
// the 1D tables by row: values, derivatives, weighted values
template <typename T>
struct Rows {
    T P[4][4], D[4][4], W[4][4];
};
template <typename T, int K>
inline void fill_rows(Rows<T>& r)
{
    constexpr G1<K> G{};
    for (int a = 0; a <= K; ++a)
        for (int m = 0; m <= K; ++m) {
            r.P[a][m] = T(G.P[m][a]);
            r.D[a][m] = T(G.D[m][a]);
            r.W[a][m] = T(0.5 * G.w[a] * G.P[m][a]);
        }
}

// contraction of the modes (i, j, l) over l with the plane's values pz[l]
template <typename T, int K>
__device__ __forceinline__ void plane_eval(const T* u, const T* pz, T* A)
{
    static_for<0, K + 1>([&](auto I) {
        constexpr int i = decltype(I)::value;
        static_for<0, K - i + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            T acc = u[im<K>(i, j, 0)];
            static_for<1, K - i - j + 1>([&](auto L) {
                constexpr int l = decltype(L)::value;
                acc += pz[l] * u[im<K>(i, j, l)];
            });
            A[ip(K, i, j)] = acc;
        });
    });
}
// the same with the derivative along z (pairs i + j <= K-1)
template <typename T, int K>
__device__ __forceinline__ void plane_deriv(const T* u, const T* dz, T* A)
{
    static_for<0, K>([&](auto I) {
        constexpr int i = decltype(I)::value;
        static_for<0, K - i>([&](auto J) {
            constexpr int j = decltype(J)::value;
            T acc = T(0);
            static_for<1, K - i - j + 1>([&](auto L) {
                constexpr int l = decltype(L)::value;
                if constexpr (l == 1)
                    acc = dz[l] * u[im<K>(i, j, l)];
                else
                    acc += dz[l] * u[im<K>(i, j, l)];
            });
            A[ip(K - 1, i, j)] = acc;
        });
    });
}

// coefficients f[(i, j, l)] of degree <= M from the plane sums X[(entry) n 32 +
// plane 32 + lane] of a component
template <typename T, int K, int M>
__device__ __forceinline__ void z_project(const T* X, int lane, T* f)
{
    constexpr int n = K + 1;
    static_for<0, M + 1>([&](auto I) {
        constexpr int i = decltype(I)::value;
        static_for<0, M - i + 1>([&](auto J) {
            constexpr int j = decltype(J)::value;
            T x[n], t[n];
#pragma unroll
            for (int c = 0; c < n; ++c) x[c] = X[(ip(M, i, j) * n + c) * 32 + lane];
            line_proj<T, K, M - i - j>(x, t);
            static_for<0, M - i - j + 1>([&](auto L) {
                constexpr int l = decltype(L)::value;
                f[im<K>(i, j, l)] = t[l];
            });
        });
    });
}

// ---------------------------------------------------------------------------
// row copies
// ---------------------------------------------------------------------------
// N elements of a row by the widest vector its length allows (rows start on
// 16-byte boundaries when N elements are a multiple of 16 bytes, else 8)
template <typename T, int N>
__device__ __forceinline__ void ld_row(const T* p, T* o)
{
    constexpr int bytes = N * (int)sizeof(T);
    if constexpr (bytes % 16 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int l = 0; l < N; l += 4) {
            const float4 v = *reinterpret_cast<const float4*>(p + l);
            o[l] = v.x;
            o[l + 1] = v.y;
            o[l + 2] = v.z;
            o[l + 3] = v.w;
        }
    } else if constexpr (bytes % 8 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int l = 0; l < N; l += 2) {
            const float2 v = *reinterpret_cast<const float2*>(p + l);
            o[l] = v.x;
            o[l + 1] = v.y;
        }
    } else {
        static_assert(sizeof(T) == 8 && bytes % 16 == 0, "row length");
#pragma unroll
        for (int l = 0; l < N; l += 2) {
            const double2 v = *reinterpret_cast<const double2*>(p + l);
            o[l] = v.x;
            o[l + 1] = v.y;
        }
    }
}
template <typename T, int N>
__device__ __forceinline__ void st_row(T* p, const T* o)
{
    constexpr int bytes = N * (int)sizeof(T);
    if constexpr (bytes % 16 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int l = 0; l < N; l += 4)
            *reinterpret_cast<float4*>(p + l) = make_float4(o[l], o[l + 1], o[l + 2], o[l + 3]);
    } else if constexpr (bytes % 8 == 0 && sizeof(T) == 4) {
#pragma unroll
        for (int l = 0; l < N; l += 2) *reinterpret_cast<float2*>(p + l) = make_float2(o[l], o[l + 1]);
    } else {
        static_assert(sizeof(T) == 8 && bytes % 16 == 0, "row length");
#pragma unroll
        for (int l = 0; l < N; l += 2) *reinterpret_cast<double2*>(p + l) = make_double2(o[l], o[l + 1]);
    }
}

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
template <int CH>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem)
{
    if constexpr (CH == 16)
        cp_async16(smem, gmem);
    else
        cp_async8(smem, gmem);
}
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

constexpr int TCELL = 32;  // cells per block

// row length in elements, padded to an odd number of 16-byte units (rows of
// 8-byte vectors: to a multiple of 8 bytes that is no multiple of 16)
template <typename T>
constexpr int padded(int len)
{
    int bytes = len * (int)sizeof(T);
    if (bytes % 16 == 8) return len;
    while ((bytes / 16) % 2 == 0) bytes += 16;
    return bytes / (int)sizeof(T);
}

// cell of a tile's lane: cells past the end repeat the last one (finite values,
// not stored)
__device__ __forceinline__ long clamp_cell(long c, long ncell) { return c < ncell ? c : ncell - 1; }

// asynchronous copy of the tile's rows (ROW elements per cell, consecutive in
// global memory) into shared rows of LD elements: four lanes per cell
template <typename T, int ROW, int LD, int NT, int CH>
__device__ __forceinline__ void tile_async(T* dst, const T* src, long c0, long ncell)
{
    constexpr int V = CH / (int)sizeof(T), NCH = ROW / V;
    static_assert(ROW % V == 0, "chunks");
    const int sub = threadIdx.x & 3;
#pragma unroll
    for (int cb = 0; cb < TCELL; cb += NT / 4) {
        const int c = cb + (threadIdx.x >> 2);
        if (c < TCELL) {
            const T* s = src + clamp_cell(c0 + c, ncell) * ROW;
            T* d = dst + c * LD;
#pragma unroll
            for (int k = 0; k < (NCH + 3) / 4; ++k) {
                const int ch = sub + 4 * k;
                if (NCH % 4 == 0 || ch < NCH) cp_async<CH>(d + ch * V, s + ch * V);
            }
        }
    }
}
// chunk width of rows of ROW elements
template <typename T, int ROW>
constexpr int chunk()
{
    return (ROW * (int)sizeof(T)) % 16 == 0 ? 16 : 8;
}

// coalesced store of nvalid rows of ROW elements from shared rows of LD elements;
// destinations that are not 16-byte aligned are written element by element
template <typename T, int ROW, int LD, int NT>
__device__ __forceinline__ void tile_store(T* dst, const T* src, long c0, int nvalid)
{
    constexpr int CH = chunk<T, ROW>(), V = CH / (int)sizeof(T), NCH = ROW / V;
    T* g = dst + c0 * ROW;
    if ((reinterpret_cast<uintptr_t>(g) & (CH - 1)) == 0) {
        for (int e = threadIdx.x; e < nvalid * NCH; e += NT) {
            const int c = e / NCH, ch = e - c * NCH;
            if constexpr (CH == 16)
                reinterpret_cast<uint4*>(g)[e] = *reinterpret_cast<const uint4*>(src + c * LD + ch * V);
            else
                reinterpret_cast<uint2*>(g)[e] = *reinterpret_cast<const uint2*>(src + c * LD + ch * V);
        }
    } else {
        for (int e = threadIdx.x; e < nvalid * ROW; e += NT) g[e] = src[(e / ROW) * LD + e % ROW];
    }
}

// ---------------------------------------------------------------------------
// arguments
// ---------------------------------------------------------------------------
template <typename T>
struct Args {
    const T* u_in;
    const T* u_n;
    T* out;            // volume kernel: rvol; face kernel: rvol in, u^(s+1) or dudt out
    const T* vh_in;    // face kernel: projected velocity of u_in
    T* vh_out;         // volume kernel: projected velocity of u_in
    T* vabs_out;       // projection of |v|
    const T* ahat;
    const T* phiv;     // [b][nq], [b][nf]: exact positivity check
    const T* phif;
    const float* nu;   // learned sensor: per-cell coefficient
    Ctl* ctl;
    double* partials;
    long ncell;
    int N;
    int av_mode;
    int tcount;        // cells per counted volume tile (dg_prof)
    int stage;         // 1: the step's dt, 0: dt_pimax
    int dtf;           // record the CFL bound
    int abar_in, abar_out;
    Rows<T> rows;
    T two_h, inv_h, cs, cs2, eps, a2, b1;
    T rk_a, rk_b;
    double cs_d, hp, dt_pimax;
    unsigned char* trouble;
};

// shared-memory layout of the volume kernel in elements of T
template <typename T, int K, bool VOL, bool FORCE, bool PROJ, bool VABS>
struct VolCfg {
    static constexpr int b = Dims<K>::b, n = K + 1, NT = 32 * n;
    static constexpr int NP = npair(K), NPD = npair(K - 1);
    static constexpr int NC = VOL ? 6 : 0, NV = PROJ ? (VABS ? 4 : 3) : 0;
    static constexpr int LDU = padded<T>(4 * b), LDA = padded<T>(3 * b);
    static constexpr int LDH = padded<T>(b);  // projected rows, per component
    static constexpr int NX0 = NC * NPD + NV * NP;
    static constexpr int NX = (VOL && FORCE && 3 * NP > NX0) ? 3 * NP : NX0;  // exchanged entries
    static constexpr int oU = 0;                                // [2][32][LDU]
    static constexpr int oAh = oU + 2 * TCELL * LDU;            // [32][LDA]
    static constexpr int oR = oAh + (FORCE ? TCELL * LDA : 0);  // [32][LDU] result rows
    static constexpr int oX = oR + (VOL ? TCELL * LDU : 0);     // [NX][n][32]
    static constexpr int total = oX + NX * n * 32;
    // the momentum components (and the projected velocity's) v = v0, v0 + n.. of warp w;
    // at degree 3 warp 0 takes the density and |v| instead
    __device__ static constexpr int v0(int w) { return K == 3 ? (w == 0 ? 4 : w) : w + 1; }
    static constexpr int W_RHO = K == 1 ? 1 : 0, W_ABS = K == 3 ? 0 : 1;
    static_assert(NV == 0 || NP * n * 32 >= TCELL * LDH, "a projected row fits its entries");
    static_assert(total * (int)sizeof(T) >= NT * 8, "reduction buffer");
};

// ---------------------------------------------------------------------------
// volume kernel
// ---------------------------------------------------------------------------
// VOL: volume term -> out (FORCE: with the driving source rho a_h; the mean
// acceleration, a reduction over the state, is subtracted by the face kernel:
// the quadrature of rho abar against phi_l is abar rho_l exactly); PROJ: the
// velocity projection -> vh_out (VABS: and of |v|), with the forcing sums when
// FORCE.  !VOL: the projection launch (CFL bound with a.dtf).
//
// Bound: FP32 instruction issue and its latency, with the 12 warps per SM that 168
// registers leave: at degree 3 with FORCE and PROJ 13.5 thousand instructions per cell go
// out in 60 % of the issue slots (FMA pipe 44 %, HBM 20 %), with PROJ alone in 64 %, the
// volume term alone in 70 %.  FP64 by the FP64 pipe.
// Blocks per SM in FP32: as many as the registers allow without spilling more than a few
// (degree 2: 5 blocks 128^3 7.12 ms for 2 steps, 4 blocks 7.19, 6 blocks 7.23).
template <typename T, int K, bool VOL, bool FORCE, bool PROJ, bool VABS>
__global__ void __launch_bounds__(32 * (K + 1), sizeof(T) == 4 ? (K == 3 ? (VOL ? 3 : 4) : K == 2 ? 5 : 8) : 1)
    k_sf_vol(const __grid_constant__ Args<T> a)
{
    grid_dependency();
    using C = VolCfg<T, K, VOL, FORCE, PROJ, VABS>;
    constexpr int b = C::b, n = C::n, NT = C::NT, NP = C::NP, NPD = C::NPD, LDU = C::LDU, LDA = C::LDA;
    constexpr G1<K> G{};
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    T* sAh = sm + C::oAh;
    T* sR = sm + C::oR;
    T* sX = sm + C::oX;
    __shared__ T s_cap;
    __shared__ unsigned long long s_smax;
    __shared__ double s_tot[8];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const long ntile = (a.ncell + TCELL - 1) / TCELL;
    auto fetch = [&](long tile, int buf) {
        tile_async<T, 4 * b, LDU, NT, chunk<T, 4 * b>()>(sm + C::oU + buf * TCELL * LDU, a.u_in, tile * TCELL, a.ncell);
        cp_async_commit();
    };
    if (blockIdx.x < ntile) fetch(blockIdx.x, 0);
    if (tid == 0) {
        s_smax = 0ull;
        if constexpr (VOL) {
            double dtd = a.dt_pimax;
            if (a.stage) {
                // the step's dt (Sec. 7 CFL condition), fixed for all its stages: from the
                // wave-speed bound of u^n, a prescribed dt, and the retry factor
                dtd = (a.ctl->fixed_dt > 0.0 ? a.ctl->fixed_dt : a.ctl->dt_num / a.ctl->sn) * a.ctl->dt_scale;
                if (blockIdx.x == 0) a.ctl->dt = dtd;
            }
            s_cap = dtd > 0.0 ? T(0.5 * a.hp * a.hp / dtd) : T(-1);
        }
    }
    // the plane's basis values and derivatives along z
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
    // positivity by repetition: a volume point of a stage output faster than the
    // Courant condition of its step allows marks its cell
    const T vlim = (PROJ && a.trouble) ? T(DG_REPEAT_SPEED * a.ctl->sn - 3.0 * a.cs_d) : T(0);
    T smax = T(0);
    double sum = 0.0, sum3 = 0.0;  // thread (component i = w + n.., cell): <rho a_h>_i; warp 0: <rho>
    double sumx = 0.0;             // component n + w where there are fewer than three warps
    unsigned int ntiles = 0, gated = 0;
    __syncthreads();
    const T cap = VOL ? s_cap : T(0);
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
        T a2 = a.a2, b1 = a.b1;
        bool need_div = a.av_mode == 1;
        if constexpr (VOL) {
            if (a.av_mode == 2) {
                // learned sensor: Pi = rho nu |div v|; no gradients where every cell of the
                // block has a zero coefficient
                b1 = valid ? T(a.nu[c0 + lane]) : T(0);
                a2 = T(0);
                need_div = __ballot_sync(0xffffffffu, b1 != T(0)) != 0u;
            }
            if (tid == 0) {
                // a block's cells skip together: a tile beside one that needs div v has not
                const unsigned int nt = (nvalid + a.tcount - 1) / a.tcount;
                ntiles += nt;
                gated += need_div ? 0u : nt;
            }
        }
        T A[4][NP];
        static_for<0, 4>([&](auto F) {
            constexpr int f = decltype(F)::value;
            T uu[b];
            ld_row<T, b>(sU + f * b, uu);
            plane_eval<T, K>(uu, pz, A[f]);
        });
        // ---- driving source rho a_h (Sec. 2.2), a pass of its own: its 30 sums would
        // not fit the registers next to those of the fluxes ----
        if constexpr (FORCE) {
            cp_async_wait<1>();
            __syncthreads();
            const T* ah = sAh + lane * LDA;
            // per-cell forcing sums <rho a_h> = sum_l rho_l a_l (orthonormal basis), <rho>
            if constexpr (PROJ) {
                auto dot = [&](int i) {
                    T s = T(0), x[b], y[b];
                    ld_row<T, b>(sU, x);
                    ld_row<T, b>(ah + i * b, y);
#pragma unroll
                    for (int l = 0; l < b; ++l) s += x[l] * y[l];
                    return (double)s;
                };
                if (valid) {
                    if (w < 3) sum += dot(w);
                    if (n < 3 && w == 0) sumx += dot(2);
                    if (w == 0) sum3 += (double)sU[0];
                }
            }
            if constexpr (VOL) {
                T Aa[3][NP], S[3][NP];
                static_for<0, 3>([&](auto F) {
                    constexpr int f = decltype(F)::value;
                    T uu[b];
                    ld_row<T, b>(ah + f * b, uu);
                    plane_eval<T, K>(uu, pz, Aa[f]);
                });
#pragma unroll
                for (int f = 0; f < 3; ++f)
#pragma unroll
                    for (int e = 0; e < NP; ++e) S[f][e] = T(0);
#pragma unroll 1
                for (int B = 0; B < n; ++B) {
                    const T *pj = a.rows.P[B], *wj = a.rows.W[B];
                    T r[n], rho[n];
                    row_eval<T, K>(A[0], pj, r);
                    line_eval<T, K, K, false>(r, rho);
                    static_for<0, 3>([&](auto F) {
                        constexpr int f = decltype(F)::value;
                        T q[n], v[n], t[n];
                        row_eval<T, K>(Aa[f], pj, q);
                        line_eval<T, K, K, false>(q, v);
#pragma unroll
                        for (int i = 0; i < n; ++i) v[i] *= rho[i];
                        line_proj<T, K, K>(v, t);
                        row_acc<T, K>(t, wj, S[f]);
                    });
                }
                static_for<0, 3>([&](auto F) {
                    constexpr int f = decltype(F)::value;
#pragma unroll
                    for (int e = 0; e < NP; ++e) sX[((f * NP + e) * n + w) * 32 + lane] = S[f][e];
                });
                __syncthreads();
                // the thread of the momentum component adds the flux part to these rows below
#pragma unroll 1
                for (int v = C::v0(w); v < 4; v += n) {
                    T q[b];
                    z_project<T, K, K>(sX + (v - 1) * NP * n * 32, lane, q);
                    st_row<T, b>(sR + lane * LDU + v * b, q);
                }
                __syncthreads();
            }
        }
        // ---- main pass: the plane's rows of points ----
        T Fx[VOL ? 6 : 1][VOL ? NPD : 1];  // sums of xx, yy, zz, xy, xz, yz (degree <= K-1)
        T Vx[PROJ ? C::NV : 1][PROJ ? NP : 1];  // sums of v (and |v|)
        if constexpr (VOL) {
#pragma unroll
            for (int f = 0; f < 6; ++f)
#pragma unroll
                for (int e = 0; e < NPD; ++e) Fx[f][e] = T(0);
        }
        if constexpr (PROJ) {
#pragma unroll
            for (int f = 0; f < C::NV; ++f)
#pragma unroll
                for (int e = 0; e < NP; ++e) Vx[f][e] = T(0);
        }
        auto rows = [&](auto DIV_) {
            constexpr bool DIV = decltype(DIV_)::value;
            T Az[DIV ? NPD : 1], Mz[DIV ? NPD : 1];  // d rho/dz, d m_z/dz
            if constexpr (DIV) {
                T uu[b];
                ld_row<T, b>(sU, uu);
                plane_deriv<T, K>(uu, dz, Az);
                ld_row<T, b>(sU + 3 * b, uu);
                plane_deriv<T, K>(uu, dz, Mz);
            }
#pragma unroll 1
            for (int B = 0; B < n; ++B) {
                const T *pj = a.rows.P[B], *dj = a.rows.D[B], *wj = a.rows.W[B];
                T f[4][n];
                T gx[n], gy[n], gz[n], dm[n];
                static_for<0, 4>([&](auto F) {
                    constexpr int v = decltype(F)::value;
                    T r[n];
                    row_eval<T, K>(A[v], pj, r);
                    line_eval<T, K, K, false>(r, f[v]);
                    if constexpr (DIV && v == 0) line_eval<T, K, K, true>(r, gx);
                    if constexpr (DIV && v == 1) line_eval<T, K, K, true>(r, dm);
                });
                if constexpr (DIV) {
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
                // pointwise (Sec. 3.1: Pi at the volume points)
                T P[n], vx[n], vy[n], vz[n];
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const T rho = f[0][i], ir = rcp<T>(rho);
                    vx[i] = f[1][i] * ir;
                    vy[i] = f[2][i] * ir;
                    vz[i] = f[3][i] * ir;
                    if constexpr (VOL) {
                        P[i] = a.cs2 * rho;
                        if constexpr (DIV) {
                            // A = -div v
                            const T Ad = (vx[i] * gx[i] + vy[i] * gy[i] + vz[i] * gz[i] - dm[i]) * (ir * a.two_h);
                            const T ra = rho * Ad;
                            T Pi = ra * (a2 * Ad + b1);
                            if (cap >= T(0)) {
                                const T Pm = ra * cap;
                                Pi = Pi < Pm ? Pi : Pm;
                            }
                            P[i] += Ad > T(0) ? Pi : T(0);
                        }
                    }
                    if constexpr (PROJ) {
                        const T sp = fabs(vx[i]) + fabs(vy[i]) + fabs(vz[i]);
                        if constexpr (!VOL) {
                            if (a.dtf && valid) smax = sp > smax ? sp : smax;
                        }
                        if (a.trouble && valid && sp > vlim) {
                            a.trouble[c0 + lane] |= DG_MARK_FAST;
                            atomicOr(&a.ctl->status, DG_ST_TROUBLED_);
                        }
                    }
                }
                if constexpr (VOL) {
                    auto comp = [&](auto G_, const T* p, const T* q, bool diag) {
                        constexpr int g = decltype(G_)::value;
                        T x[n], t[n];
#pragma unroll
                        for (int i = 0; i < n; ++i) x[i] = diag ? p[i] * q[i] + P[i] : p[i] * q[i];
                        line_proj<T, K, K - 1>(x, t);
                        row_acc<T, K - 1>(t, wj, Fx[g]);
                    };
                    comp(std::integral_constant<int, 0>{}, f[1], vx, true);
                    comp(std::integral_constant<int, 1>{}, f[2], vy, true);
                    comp(std::integral_constant<int, 2>{}, f[3], vz, true);
                    comp(std::integral_constant<int, 3>{}, f[1], vy, false);
                    comp(std::integral_constant<int, 4>{}, f[1], vz, false);
                    comp(std::integral_constant<int, 5>{}, f[2], vz, false);
                }
                if constexpr (PROJ) {
                    T t[n];
                    if constexpr (VABS) {
                        T x[n];
#pragma unroll
                        for (int i = 0; i < n; ++i) x[i] = sqrt(vx[i] * vx[i] + vy[i] * vy[i] + vz[i] * vz[i]);
                        line_proj<T, K, K>(x, t);
                        row_acc<T, K>(t, wj, Vx[C::NV - 1]);
                    }
                    line_proj<T, K, K>(vx, t);
                    row_acc<T, K>(t, wj, Vx[0]);
                    line_proj<T, K, K>(vy, t);
                    row_acc<T, K>(t, wj, Vx[1]);
                    line_proj<T, K, K>(vz, t);
                    row_acc<T, K>(t, wj, Vx[2]);
                }
            }
        };
        if (VOL && need_div)
            rows(std::integral_constant<bool, VOL>{});
        else
            rows(std::integral_constant<bool, false>{});
        // ---- exchange along z ----
        if constexpr (VOL) {
            static_for<0, 6>([&](auto F) {
                constexpr int f = decltype(F)::value;
#pragma unroll
                for (int e = 0; e < NPD; ++e) sX[((f * NPD + e) * n + w) * 32 + lane] = Fx[f][e];
            });
        }
        if constexpr (PROJ) {
            static_for<0, C::NV>([&](auto F) {
                constexpr int f = decltype(F)::value;
#pragma unroll
                for (int e = 0; e < NP; ++e) sX[((C::NC * NPD + f * NP + e) * n + w) * 32 + lane] = Vx[f][e];
            });
        }
        __syncthreads();
        // ---- volume term (2/h) sum_d D_d^T Fhat_d of a variable, and the projected
        // components ----
        if constexpr (VOL) {
            if (w == C::W_RHO) {
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
        }
#pragma unroll 1
        for (int v = C::v0(w); v < 4; v += n) {
            T q[b];
            if constexpr (VOL) {
                T r[b];
                const int cx = v == 1 ? 0 : v + 1, cy = v == 1 ? 3 : (v == 2 ? 1 : 5), cz = v == 3 ? 2 : v + 3;
                if constexpr (FORCE) {
                    ld_row<T, b>(sR + lane * LDU + v * b, r);
                } else {
#pragma unroll
                    for (int l = 0; l < b; ++l) r[l] = T(0);
                }
                z_project<T, K, K - 1>(sX + cx * NPD * n * 32, lane, q);
                modal_grad_T_acc<T, K, 0>(q, r, a.two_h);
                z_project<T, K, K - 1>(sX + cy * NPD * n * 32, lane, q);
                modal_grad_T_acc<T, K, 1>(q, r, a.two_h);
                z_project<T, K, K - 1>(sX + cz * NPD * n * 32, lane, q);
                modal_grad_T_acc<T, K, 2>(q, r, a.two_h);
                st_row<T, b>(sR + lane * LDU + v * b, r);
            }
            if constexpr (PROJ) {
                // the rows replace the component's entries, which only this warp reads
                T* X = sX + (C::NC * NPD + (v - 1) * NP) * n * 32;
                z_project<T, K, K>(X, lane, q);
                __syncwarp();
                st_row<T, b>(X + lane * C::LDH, q);
            }
        }
        if constexpr (VABS) {
            if (w == C::W_ABS) {
                T q[b];
                T* X = sX + (C::NC * NPD + 3 * NP) * n * 32;
                z_project<T, K, K>(X, lane, q);
                __syncwarp();
                st_row<T, b>(X + lane * C::LDH, q);
            }
        }
        __syncthreads();
        // ---- coalesced stores ----
        if constexpr (VOL) tile_store<T, 4 * b, LDU, NT>(a.out, sR, c0, nvalid);
        if constexpr (PROJ) {
            const T* X = sX + C::NC * NPD * n * 32;
            constexpr int CS = NP * n * 32;  // components apart
            constexpr int CH = chunk<T, b>(), V = CH / (int)sizeof(T), NCH = 3 * b / V, NCB = b / V;
            T* g = a.vh_out + c0 * 3 * b;
            if ((reinterpret_cast<uintptr_t>(g) & (CH - 1)) == 0) {
                for (int e = tid; e < nvalid * NCH; e += NT) {
                    const int c = e / NCH, ch = e - c * NCH, i = ch / NCB, o = ch - i * NCB;
                    const T* s = X + i * CS + c * C::LDH + o * V;
                    if constexpr (CH == 16)
                        reinterpret_cast<uint4*>(g)[e] = *reinterpret_cast<const uint4*>(s);
                    else
                        reinterpret_cast<uint2*>(g)[e] = *reinterpret_cast<const uint2*>(s);
                }
            } else {
                for (int e = tid; e < nvalid * 3 * b; e += NT) {
                    const int c = e / (3 * b), i = (e / b) % 3, l = e % b;
                    g[e] = X[i * CS + c * C::LDH + l];
                }
            }
            if constexpr (VABS) {
                if (a.vabs_out) tile_store<T, b, C::LDH, NT>(a.vabs_out, X + 3 * CS, c0, nvalid);
            }
        }
    }
    // ---- block reductions ----
    if constexpr (VOL) {
        if (tid == 0 && ntiles > 0) {
            atomicAdd(&a.ctl->tiles_vol, (unsigned long long)ntiles);
            if (gated) atomicAdd(&a.ctl->tiles_gated, (unsigned long long)gated);
        }
    }
    if constexpr (PROJ && (FORCE || !VOL)) {
        cp_async_wait<0>();
        __syncthreads();
        double* s_buf = reinterpret_cast<double*>(smem_raw);
        if (!VOL && a.dtf) {
            const double sp = (double)warp_max(smax) + 3.0 * a.cs_d;
            if (lane == 0) atomicMax(&s_smax, (unsigned long long)__double_as_longlong(sp));
            __syncthreads();
            if (tid == 0) atomicMax(&a.ctl->smax, s_smax);
        }
        double mine[4] = {0.0, 0.0, 0.0, 0.0};
        if constexpr (FORCE) {
            // over the warp by shuffles, then the warps' sums in s_buf[0..n)
            auto reduce = [&](double v, double* dst) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) s_buf[w] = v;
                __syncthreads();
                if (tid == 0)
                    for (int j = 0; j < n; ++j) dst[j] = s_buf[j];
                __syncthreads();
            };
            double t4[n], x4[n];
            reduce(sum, t4);
            if (tid == 0)
                for (int i = 0; i < 3 && i < n; ++i) mine[i] = t4[i];
            if constexpr (n < 3) {
                reduce(sumx, x4);
                if (tid == 0) mine[2] = x4[0];
            }
            reduce(sum3, x4);
            if (tid == 0) mine[3] = x4[0];
        }
        if (last_block_reduce<NT>(a.partials, mine, FORCE ? 4 : 0, &a.ctl->cnt_proj, s_tot)) {
            if (tid == 0) {
                const int o = a.abar_out;
                for (int i = 0; i < 3; ++i) a.ctl->abar2[o][i] = FORCE ? s_tot[i] / s_tot[3] : 0.0;
                if (!VOL && a.dtf) {
                    const unsigned long long bits = atomicAdd(&a.ctl->smax, 0ull);
                    a.ctl->sn = __longlong_as_double((long long)bits);
                    a.ctl->smax = 0ull;
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// face kernel
// ---------------------------------------------------------------------------
// A block takes a brick of 4 x 4 x 2 cells (lane = cell, x fastest) with 4 warps, a
// thread per face (BrickFaces): 128 faces where 32 cells taken one by one have 192, and
// 96 operand rows where those would read 224.  Bricks past the end of the mesh hold the
// periodic images of its cells, which are the neighbours the last cells need.
// Bound: latency between the phases of a brick (rows in, traces and fluxes, rows of the
// stage in, combine), with the 12 warps per SM that 168 registers and 53 KB leave at
// degree 3: issue slots 47 %, FMA pipe 32 %, HBM 37 %, no pipe near its limit.  64^3 of
// degree 3 FP32: 130 us (2.3 TB/s; 212 us with the six faces of 32 consecutive cells),
// 256^3 8.3 ms.  Four blocks with the traces in shared memory were slower
// (0.83-0.9x), packed pairs of FP32 and a prefetch of the next bricks to L2 no faster.
template <typename T, int K>
struct FaceCfg {
    static constexpr int b = Dims<K>::b, NP = npair(K), NT = 128;
    static constexpr int LD = padded<T>(4 * b);  // rows rho, v (operands) and rho, m (states)
    static constexpr int REG = TCELL * LD;
    // rows 0-31: the brick's cells; 32-63: those across its -x, +x, -y, +y sides (8
    // each); 64-95: across -z, +z (16 each).  Later 0-31: u^(s) (then the new state),
    // 32-63: rvol, 64-95: u^n
    static constexpr int oFlux = 3 * REG;  // [variable][pair][face]
    static constexpr int total = oFlux + 4 * NP * 128;
};

// The faces of a brick by thread.  Warps 0 and 1 own the + faces of the cells along x
// and y; warps 2 and 3 the three layers of z faces (0 below the brick, 1 between its
// planes, 2 above) and the 8 + 8 faces of its lower x and y sides:
//   warp 2 layer 1 of cells 0-7, lower x, layer 2; warp 3 lower y, layer 1 of cells 8-15,
//   layer 0.
// The traces along the directions are different code: no warp runs more than two of the
// three while the others wait (with all lower faces in warp 3, 64^3 of degree 3 took 3.94
// ms for 4 steps, 3.90 so; 256^3 51.0 and 50.5).
struct BrickFaces {
    int d, rowL, rowR;  // direction, rows of the lower (L) and upper (R) cell
    __device__ __forceinline__ BrickFaces(int w, int lane)
    {
        const int i = lane & 3, j = (lane >> 2) & 3, k = lane >> 4, k8 = j & 1;
        if (w < 2) {
            d = w;
            rowL = lane;
            rowR = w == 0 ? (i < 3 ? lane + 1 : 40 + 4 * k + j) : (j < 3 ? lane + 4 : 56 + 4 * k + i);
        } else if (k == 0 && (lane >= 8) == (w == 2)) {  // lower x of (j, k) = (i, k8), lower y of (i, k8)
            d = w - 2;
            rowL = 32 + 16 * d + (lane & 7);
            rowR = d == 0 ? 16 * k8 + 4 * i : 16 * k8 + i;
        } else {
            const bool low = w == 3 && k == 1;
            d = 2;
            rowL = low ? 64 + lane - 16 : lane;
            rowR = low ? lane - 16 : (k < 1 ? lane + 16 : 80 + 4 * j + i);
        }
    }
    // the face of cell c of the brick on its + / - side along Dd
    template <int Dd>
    __device__ static __forceinline__ int above(int c)
    {
        return 32 * Dd + c + (Dd == 2 && (c & 24) == 8 ? 32 : 0);
    }
    template <int Dd>
    __device__ static __forceinline__ int below(int c)
    {
        const int i = c & 3, j = (c >> 2) & 3, k = c >> 4;
        if constexpr (Dd == 0) return i > 0 ? c - 1 : 72 + 4 * k + j;
        if constexpr (Dd == 1) return j > 0 ? 32 + c - 4 : 96 + 4 * k + i;
        return k > 0 ? above<2>(c - 16) : 112 + c;
    }
};

// 2D coefficients of a field's trace on the + (SIDE 1) or - face along Dd
template <typename T, int K, int Dd, int SIDE>
__device__ __forceinline__ void trace(const T* c, T* c2)
{
    static_for<0, K + 1>([&](auto I) {
        constexpr int p = decltype(I)::value;
        static_for<0, K - p + 1>([&](auto J) {
            constexpr int q = decltype(J)::value;
            T acc = T(0);
            static_for<0, K - p - q + 1>([&](auto L) {
                constexpr int d = decltype(L)::value;
                constexpr int m = Dd == 0 ? im<K>(d, p, q) : (Dd == 1 ? im<K>(p, d, q) : im<K>(p, q, d));
                DG_SF_MAC(T, acc, ((SIDE || !(d & 1)) ? 1.0 : -1.0) * csqrt(2.0 * d + 1.0), c[m], d == 0);
            });
            c2[ip(K, p, q)] = acc;
        });
    });
}

// Face fluxes along the normal (component 1) from left/right primitive states (rho, v_n,
// v_t1, v_t2).  The momentum crosses with a left and a right mass flux,
//   F_m = q_L v_L + q_R v_R + p* e_n;
// the mass flux itself, q_L + q_R, is formed from the density difference instead, so
// that slow flows do not lose it between two terms of the size rho cs.
// Rusanov, F = (F_L + F_R)/2 - lambda (U_R - U_L)/2, lambda = max |v_n| + cs:
//   q_L = rho_L (v_n,L + lambda)/2, q_R = rho_R (v_n,R - lambda)/2, p* = cs^2 (rho_L + rho_R)/2
// (19 instructions where the states and fluxes written out take 33)
template <typename T>
__device__ __forceinline__ void rusanov_normal(T cs, T cs2, const T* WL, const T* WR, T* F)
{
    const T hl = T(0.5) * fmax(fabs(WL[1]), fabs(WR[1])) + T(0.5) * cs;
    const T mL = WL[0] * (T(0.5) * WL[1]), mR = WR[0] * (T(0.5) * WR[1]);
    const T qL = mL + hl * WL[0], qR = mR - hl * WR[0];
    F[0] = (mL + mR) - hl * (WR[0] - WL[0]);
    F[1] = T(0.5) * cs2 * (WL[0] + WR[0]) + (qL * WL[1] + qR * WR[1]);
    F[2] = qL * WL[2] + qR * WR[2];
    F[3] = qL * WL[3] + qR * WR[3];
}
// HLL, F = (S_R F_L - S_L F_R + S_L S_R (U_R - U_L))/(S_R - S_L) with the Davis bounds,
// clamped at zero where both have one sign:
//   w_L = S_R/(S_R - S_L), w_R = -S_L/(S_R - S_L), q_L = w_L rho_L (v_n,L - S_L),
//   q_R = w_R rho_R (v_n,R - S_R), p* = cs^2 (w_L rho_L + w_R rho_R).
// The smaller weight is formed from its own bound and the larger one as the rest: a clamped
// bound then leaves the upwind flux exactly, on either side, and a bound near zero lets no
// rounding of the other weight carry a dense side's flux into a thin one.  Outside the bounds
// the upwind state stands on both sides: a downwind vacuum or NaN does not enter.
// CONTACT (HLLC for p = cs^2 rho): the tangential momenta cross with the mass flux at the
// tangential velocity of the side the contact S_M = m*/rho* leaves behind
template <typename T, bool CONTACT>
__device__ __forceinline__ void hll_normal(T cs, T cs2, const T* L, const T* R, T* F)
{
    const T SL = fmin(L[1], R[1]) - cs, SR = fmax(L[1], R[1]) + cs;
    T WL[4], WR[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        WL[v] = SR <= T(0) ? R[v] : L[v];
        WR[v] = SL >= T(0) ? L[v] : R[v];
    }
    const T vl = WL[1], vr = WR[1];
    const T sl = fmin(SL, T(0)), sr = fmax(SR, T(0));
    const bool nearer = sr < -sl;  // of the two bounds S_R
    const T ws = (nearer ? sr : -sl) * rcp<T>(sr - sl), wb = T(1) - ws;
    const T wl = nearer ? ws : wb, wr = nearer ? wb : ws;
    const T rl = wl * WL[0], rr = wr * WR[0];
    const T qL = rl * (vl - sl), qR = rr * (vr - sr);
    F[0] = (rl * vl + rr * vr) - wr * sr * (WR[0] - WL[0]);
    F[1] = cs2 * (rl + rr) + (qL * vl + qR * vr);
    if constexpr (CONTACT) {
        // signs of rho* and m* (times S_R - S_L > 0)
        const T aL = WL[0] * (SL - vl), aR = WR[0] * (SR - vr);
        const T ms = aR * vr - aL * vl - cs2 * (WR[0] - WL[0]);
        const bool left = (aR - aL > T(0)) == (ms >= T(0));
        F[2] = F[0] * (left ? WL[2] : WR[2]);
        F[3] = F[0] * (left ? WL[3] : WR[3]);
    } else {
        F[2] = qL * WL[2] + qR * WR[2];
        F[3] = qL * WL[3] + qR * WR[3];
    }
}

// 9.1 thousand instructions per cell at degree 3, bound as above.
// Blocks per SM in FP32: degree 1 8 blocks (96^3: 0.377 ms a step; 6: 0.394),
// degree 2 4 (128^3, 2 steps: 7.19 ms; 5: 7.28), degree 3 3.
template <typename T, int K, int RS, bool STAGE>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? (K == 1 ? 8 : K == 2 ? 4 : 3) : 1)
    k_sf_faces(const __grid_constant__ Args<T> a)
{
    grid_dependency();
    using C = FaceCfg<T, K>;
    constexpr int b = C::b, n = K + 1, NP = C::NP, NT = C::NT, LD = C::LD, nq = n * n * n, nf = 6 * n * n;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sm = reinterpret_cast<T*>(smem_raw);
    __shared__ T s_th[TCELL];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const Brick brick(blockIdx.x, a.N);
    // ---- operand rows (rho, v), four lanes per row ----
    const int rs = tid >> 2, sub = tid & 3;  // row within a group of 32, lane of it
    const int ri = rs & 3, rj = (rs >> 2) & 3, rk = rs >> 4;
    const long rcell = brick.cell(ri, rj, rk), own = brick.own(rs);
    {
        constexpr int CH = chunk<T, b>(), V = CH / (int)sizeof(T), NB = b / V;  // chunks of rho; 3 NB of v
        auto copy_row = [&](T* dst, long c) {
            const T* ru = a.u_in + c * 4 * b;
            const T* rv = a.vh_in + c * 3 * b - b;  // chunk ch >= NB: v
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const int ch = sub + 4 * k;
                cp_async<CH>(dst + ch * V, (ch < NB ? ru : rv) + ch * V);
            }
        };
        copy_row(sm + rs * LD, rcell);
        // -x, +x: (j, k) = (rs & 3, (rs >> 2) & 1); -y, +y: (i, k) the same
        const int hs = rs >> 3, h0 = rs & 3, h1 = (rs >> 2) & 1;
        copy_row(sm + (32 + rs) * LD, hs < 2 ? brick.cell(hs ? 4 : -1, h0, h1) : brick.cell(h0, hs == 3 ? 4 : -1, h1));
        copy_row(sm + (64 + rs) * LD, brick.cell(ri, rj, rk ? 2 : -1));
        cp_async_commit();
    }
    const BrickFaces face(w, lane);
    const int d = face.d;
    const T dt = STAGE ? T(a.ctl->dt) : T(0);
    const bool fix = a.ahat != nullptr;
    cp_async_wait<0>();
    __syncthreads();
    // ---- traces: left state (the lower cell's + face), right state (- face); fields
    // rho, v_n, v_t1, v_t2 ----
    T c2[8][NP];
    {
        const T* Lp = sm + face.rowL * LD;
        const T* Rp = sm + face.rowR * LD;
        auto traces = [&](auto D_) {
            constexpr int Dd = decltype(D_)::value;
            constexpr int t1 = Dd == 0 ? 1 : 0, t2 = Dd == 2 ? 1 : 2;
            constexpr int fld[4] = {0, 1 + Dd, 1 + t1, 1 + t2};
            static_for<0, 4>([&](auto F) {
                constexpr int f = decltype(F)::value;
                T uu[b];
                ld_row<T, b>(Lp + fld[f] * b, uu);
                trace<T, K, Dd, 1>(uu, c2[f]);
                ld_row<T, b>(Rp + fld[f] * b, uu);
                trace<T, K, Dd, 0>(uu, c2[4 + f]);
            });
        };
        if (d == 0)
            traces(std::integral_constant<int, 0>{});
        else if (d == 1)
            traces(std::integral_constant<int, 1>{});
        else
            traces(std::integral_constant<int, 2>{});
    }
    __syncthreads();
    // the operand rows are free: the epilogue's inputs arrive during the fluxes, those of
    // the brick's own cells alone (rows past the end of the mesh keep what they hold: no
    // result uses them)
    constexpr int CHU = chunk<T, 4 * b>(), VU = CHU / (int)sizeof(T), NCU = 4 * b / VU;
    static_assert(CHU == 16, "state rows in 16-byte chunks");
    const bool out16 = (reinterpret_cast<uintptr_t>(a.out) & 15u) == 0;
    if (own >= 0) {
        auto copy_state = [&](T* dst, const T* src) {
            const T* s = src + own * 4 * b;
            T* q = dst + rs * LD;
#pragma unroll
            for (int k = 0; k < (NCU + 3) / 4; ++k)
                if (NCU % 4 == 0 || sub + 4 * k < NCU) cp_async<16>(q + (sub + 4 * k) * VU, s + (sub + 4 * k) * VU);
        };
        copy_state(sm, a.u_in);
        if (out16) {
            copy_state(sm + C::REG, a.out);
        } else {
            for (int e = sub; e < 4 * b; e += 4) sm[C::REG + rs * LD + e] = a.out[own * 4 * b + e];
        }
        if (STAGE && a.rk_a != T(0)) copy_state(sm + 2 * C::REG, a.u_n);
    }
    cp_async_commit();
    // ---- Riemann fluxes at the face points, lifted row by row ----
    {
        T fx[4][NP];
#pragma unroll
        for (int f = 0; f < 4; ++f)
#pragma unroll
            for (int e = 0; e < NP; ++e) fx[f][e] = T(0);
#pragma unroll 1
        for (int B = 0; B < n; ++B) {
            const T *pj = a.rows.P[B], *wj = a.rows.W[B];
            T W[8][n];
            static_for<0, 8>([&](auto F) {
                constexpr int f = decltype(F)::value;
                T r[n];
                row_eval<T, K>(c2[f], pj, r);
                line_eval<T, K, K, false>(r, W[f]);
            });
            T Fl[4][n];
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const T WL[4] = {W[0][i], W[1][i], W[2][i], W[3][i]};
                const T WR[4] = {W[4][i], W[5][i], W[6][i], W[7][i]};
                T F[4];
                if constexpr (RS == 0)
                    rusanov_normal<T>(a.cs, a.cs2, WL, WR, F);
                else
                    hll_normal<T, RS == 2>(a.cs, a.cs2, WL, WR, F);
#pragma unroll
                for (int v = 0; v < 4; ++v) Fl[v][i] = F[v];
            }
            static_for<0, 4>([&](auto F) {
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
        }
    }
    cp_async_wait<0>();
    __syncthreads();
    // ---- right-hand side of variable w: surface term + rvol ----
    T r[b];
    unsigned int st = 0u;
    const int ci = lane & 3, cj = (lane >> 2) & 3, ck = lane >> 4;
    const bool valid = brick.inside(ci, cj, ck);
    T* const row = sm + lane * LD + w * b;  // u^(s), later the result
#pragma unroll
    for (int l = 0; l < b; ++l) r[l] = T(0);
    static_for<0, 3>([&](auto D_) {
        constexpr int Dd = decltype(D_)::value;
        const T* X = sm + C::oFlux + w * NP * 128;
        const T *Xp = X + BrickFaces::above<Dd>(lane), *Xm = X + BrickFaces::below<Dd>(lane);
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
    {
        T x[b];
        ld_row<T, b>(row + C::REG, x);  // rvol
#pragma unroll
        for (int l = 0; l < b; ++l) r[l] = r[l] * a.inv_h + x[l];
        if (fix && w > 0) {
            // the source's mean-acceleration part: -abar_i rho_l
            const T ab = T(a.ctl->abar2[a.abar_in][w - 1]);
            ld_row<T, b>(sm + lane * LD, x);
#pragma unroll
            for (int l = 0; l < b; ++l) r[l] -= ab * x[l];
        }
    }
    // every warp has read rho before warp 0 replaces it
    if (fix) __syncthreads();
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
        if (w == 0) {
            // positivity (Sec. 3.1): a cell passes when rho_0 - sum_l |rho_l| sup|phi_l| >= eps;
            // otherwise rho is evaluated at every volume and face Gauss point (the warp
            // takes one such cell at a time) and the modes l > 0 are scaled by theta
            T part = T(0);
            static_for<1, b>([&](auto M) {
                constexpr int m = decltype(M)::value;
                part += T(sup_phi<K>(m)) * fabs(r[m]);
            });
            T th = T(1);
            unsigned low = __ballot_sync(0xffffffffu, valid && r[0] - part < a.eps);
            if (low) {
                st_row<T, b>(row, r);
                __syncwarp();
                while (low) {
                    const int c = __ffs(low) - 1;
                    low &= low - 1;
                    T rr[b];
                    ld_row<T, b>(sm + c * LD, rr);
                    T mn = T(1e30);
                    for (int pt = lane; pt < nq + nf; pt += 32) {
                        const T* ph = pt < nq ? a.phiv + pt : a.phif + (pt - nq);
                        const int sp = pt < nq ? nq : nf;
                        T rho = T(0);
#pragma unroll
                        for (int l = 0; l < b; ++l) rho += rr[l] * __ldg(ph + l * sp);
                        mn = rho < mn ? rho : mn;
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const T other = __shfl_xor_sync(0xffffffffu, mn, o);
                        mn = other < mn ? other : mn;
                    }
                    if (a.trouble && mn < T(0)) {
                        if (lane == c) a.trouble[brick.own(lane)] |= DG_MARK_NEGATIVE;
                        st |= DG_ST_TROUBLED_;
                    }
                    if (mn < a.eps) {
                        if (rr[0] > a.eps) {
                            if (lane == c) th = (rr[0] - a.eps) / (rr[0] - mn);
                            st |= DG_ST_LIMITED_;
                        } else if (!a.trouble || !(rr[0] > T(0))) {
                            // positivity by repetition: a mean in (0, eps] stands
                            st |= DG_ST_FAIL_;
                        }
                    }
                }
            }
            s_th[lane] = th;
        }
        __syncthreads();
        const T th = s_th[lane];
        bool bad = !isfinite(r[0]);
#pragma unroll
        for (int l = 1; l < b; ++l) {
            r[l] *= th;
            bad |= !isfinite(r[l]);
        }
        if (bad && valid) st |= DG_ST_NONFINITE_;
        st = __reduce_or_sync(0xffffffffu, st);
        if (lane == 0 && st) atomicOr(&a.ctl->status, st);
    }
    st_row<T, b>(row, r);
    __syncthreads();
    if (own >= 0) {
        T* g = a.out + own * 4 * b;
        const T* q = sm + rs * LD;
        if (out16) {
#pragma unroll
            for (int k = 0; k < (NCU + 3) / 4; ++k)
                if (NCU % 4 == 0 || sub + 4 * k < NCU)
                    *reinterpret_cast<uint4*>(g + (sub + 4 * k) * VU) =
                        *reinterpret_cast<const uint4*>(q + (sub + 4 * k) * VU);
        } else {
            for (int e = sub; e < 4 * b; e += 4) g[e] = q[e];
        }
    }
}

}  // namespace sf
}  // namespace dg
