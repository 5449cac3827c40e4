// dg_analysis.cu -- turbulence statistics of a state (Sec. 4.1 definitions,
// Sec. 4.3 measurement): the volume-weighted density PDF, the second-order
// velocity structure function, and the velocity sampled on the (k+1)N Fourier
// grid with the shell sums of its power spectrum.  All evaluation in FP64
// from the state's coefficients (FP64 or FP32), accumulation in FP64.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "dg_launch.cuh"
#include "dg_launch_impl.cuh"
#include "dg_sf.cuh"

namespace dg {

// All of these kernels are bound by the FP64 pipe (2 lanes per clock and SM, a
// sixty-fourth of FP32's): they evaluate the expansions axis by axis, and keep
// divisions, roots and logarithms out of FP64 where single precision decides, and
// conversions out of its pipe (widen_row, narrow).  On 64^3 cells of degree 3, FP32,
// the pipe 84-90 % busy, before and after the conversions went and the sums changed:
// 2 M pairs of the structure function 2.07 -> 1.15 ms, a sampled component 0.52 -> 0.38,
// its shell sums 0.36 -> 0.13.

// A thread's part of a cell's (K+1)^3 points: all of them, or one row along x
// (rows: item = (cell, z, y)), whose expansion along z the n threads of a plane repeat.
template <int K>
struct CellPart {
    long c;
    int z0, z1, y0, y1;
    __device__ __forceinline__ CellPart(long it, bool rows)
    {
        constexpr int n = K + 1;
        c = rows ? it / (n * n) : it;
        const int q = rows ? (int)(it - c * n * n) : 0;
        z0 = rows ? q / n : 0;
        z1 = rows ? z0 + 1 : n;
        y0 = rows ? q - z0 * n : 0;
        y1 = rows ? y0 + 1 : n;
    }
};
// Rows on meshes whose cells are too few to fill the multiprocessors: there a thread's
// chain through its whole cell is the kernel's time.  Below 64 cells per multiprocessor
// (21^3): degree 3, 200 bins, rows against cells 8^3 44 and 69 us, 16^3 53 and 77, 28^3 78
// and 78, 40^3 128 and 114; spectrum 8^3 242 and 319 us, 16^3 300 and 351, 32^3 1103 and
// 1074; degree 1 8^3 194 and 204, 24^3 226 and 218.
constexpr long kRowCells = 64;
static bool cell_rows(const Launch& L) { return L.ncell < kRowCells * (long)L.nsm; }

// sqrt(2m+1) P_m(x), m = 0..K (K <= 3)
template <int K>
__device__ __forceinline__ void pnorm_all(double x, double* p)
{
    constexpr double r3 = csqrt(3.0), r5 = csqrt(5.0), r7 = csqrt(7.0);
    p[0] = 1.0;
    if constexpr (K >= 1) p[1] = r3 * x;
    const double x2 = x * x;
    if constexpr (K >= 2) p[2] = (1.5 * r5) * x2 - 0.5 * r5;
    if constexpr (K >= 3) p[3] = x * ((2.5 * r7) * x2 - 1.5 * r7);
}

// b coefficients: 16-byte loads where the row starts on a 16-byte boundary
template <typename T, int b>
__device__ __forceinline__ void load_row(const T* __restrict__ p, T* o)
{
    constexpr int V = 16 / (int)sizeof(T);
    if (b % V == 0 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
#pragma unroll
        for (int l = 0; l + V <= b; l += V) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(p + l));
            memcpy(o + l, &q, 16);
        }
    } else {
#pragma unroll
        for (int l = 0; l < b; ++l) o[l] = __ldg(p + l);
    }
}

// the fields (rho, m_x, m_y, m_z) of one cell at reference point xi, summed along
// x, y, z in turn
template <typename T, int K>
__device__ __forceinline__ void eval_point(const T* __restrict__ uc, const double xi[3], double f[4])
{
    constexpr int b = Dims<K>::b;
    double px[K + 1], py[K + 1], pz[K + 1];
    pnorm_all<K>(xi[0], px);
    pnorm_all<K>(xi[1], py);
    pnorm_all<K>(xi[2], pz);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        T x[b];
        load_row<T, b>(uc + v * b, x);
        double u[b];
        widen_row<b>(x, u);
        double fz = 0.0;
        static_for<0, K + 1>([&](auto L) {
            constexpr int l = decltype(L)::value;
            double fy = 0.0;
            static_for<0, K - l + 1>([&](auto J) {
                constexpr int j = decltype(J)::value;
                double fx = u[sf::im<K>(0, j, l)];
                static_for<1, K - l - j + 1>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    fx += px[i] * u[sf::im<K>(i, j, l)];
                });
                fy = j == 0 ? fx : fy + py[j] * fx;
            });
            fz = l == 0 ? fy : fz + pz[l] * fy;
        });
        f[v] = fz;
    }
}

// values of the normalised Legendre polynomials at n points of an axis, symmetric
// about 0: P[a][m]
struct Line {
    double P[4][4];
};
// the n values of a line from the coefficients r[0..K] (even and odd parts of the
// mirrored points share their products)
template <int K>
__device__ __forceinline__ void line_values(const Line& t, const double* r, double* out)
{
    constexpr int n = K + 1;
#pragma unroll
    for (int q = 0; q < (n + 1) / 2; ++q) {
        const int a = n - 1 - q;
        double e = r[0], o = 0.0;
#pragma unroll
        for (int m = 2; m <= K; m += 2) e += t.P[a][m] * r[m];
#pragma unroll
        for (int m = 1; m <= K; m += 2) o = m == 1 ? t.P[a][m] * r[m] : o + t.P[a][m] * r[m];
        out[a] = e + o;
        if (a != q) out[q] = e - o;
    }
}

// the coefficients of field v of a cell in FP64
template <typename T, int K>
__device__ __forceinline__ void load_field(const T* __restrict__ uc, int v, double* o)
{
    constexpr int b = Dims<K>::b;
    T x[b];
    load_row<T, b>(uc + v * b, x);
    widen_row<b>(x, o);
}

// velocity m/rho at a point x of the periodic unit box, -1 < x_d < 2.  Floors by
// comparison and by an addition that rounds down onto the integers (the sum with
// 3 2^51 keeps them in its low word): no conversions on the FP64 pipe
template <typename T, int K>
__device__ __forceinline__ void velocity_at(const T* __restrict__ u, int N, double dN, const double x[3], double v[3])
{
    int ic[3];
    double xi[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        constexpr double big = 6755399441055744.0;
        const int hx = __double2hiint(x[d]);
        const double y = hx < 0 ? x[d] + 1.0 : (hx >= 0x3ff00000 ? x[d] - 1.0 : x[d]);
        const double s = y * dN, t = __dadd_rd(s, big);
        int i = __double2loint(t);
        double fi = t - big;
        if (i >= N) {
            i = N - 1;
            fi = dN - 1.0;
        }
        ic[d] = i;
        xi[d] = 2.0 * (s - fi) - 1.0;
    }
    const long c = ((long)ic[2] * N + ic[1]) * N + ic[0];
    double f[4];
    eval_point<T, K>(u + c * 4 * Dims<K>::b, xi, f);
    const double ir = inverse(f[0]);
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = f[1 + d] * ir;
}

// SplitMix64: the n-th output of the sequence started from `seed`, as a
// uniform double in [0, 1) from its top 53 bits
__device__ __forceinline__ double splitmix_u01(unsigned long long seed, unsigned long long n)
{
    unsigned long long z = seed + (n + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

// mean density (cell means, unit box) -> *mean (accumulated with atomics)
template <typename T, int K>
__global__ void __launch_bounds__(256) k_mean_rho(const T* __restrict__ u, long ncell, double* mean)
{
    constexpr int b = Dims<K>::b;
    __shared__ double s[256];
    double acc = 0.0;
    for (long c = blockIdx.x * 256L + threadIdx.x; c < ncell; c += (long)gridDim.x * 256)
        acc += (double)u[c * 4 * b];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(mean, s[0] / (double)ncell);
}

// volume-weighted histogram of log10(rho / mean) over the Gauss points of every
// cell.  The weights w_a w_b w_c take four values (the number of inner points among
// a, b, c: two distinct 1D weights), so the samples are counted per bin and weight
// class in integers, cnt[bin][class], and weighted once at the end.  The bin
// floor((log10(rho/mean) - lo)/ds) comes from single precision, and from FP64 where
// that lands within tol of a bin edge (tol above its error: same bins).
// One thread per cell (64 points of degree 3: 16 M points in 6.2 ms with a thread
// and a full evaluation per point) or per row of points, see cell_rows.  A block whose
// samples are fewer than the bins adds to the counters in global memory.  The last
// block to finish weights the counts and leaves the histogram in their place.
template <int K>
__host__ __device__ constexpr int inner(int a)
{
    return K == 3 ? (a == 1 || a == 2) : (K == 2 ? a == 1 : 0);
}
static __device__ __noinline__ bool positive(double x) { return x > 0.0; }
struct ClassWeights {
    double w[4];
};

template <typename T, int K>
__global__ void __launch_bounds__(128) k_density_pdf(const T* __restrict__ u, long ncell,
                                                     const __grid_constant__ Line t, const double* mean, double lo,
                                                     double ds, float tol, int nbins, bool rows, bool shared,
                                                     ClassWeights weight, unsigned int* counter, double* acc)
{
    constexpr int n = K + 1, b = Dims<K>::b, NP = sf::npair(K);
    extern __shared__ unsigned int s_cnt[];
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(acc);  // [nbins][4]
    if (shared) {
        for (int i = threadIdx.x; i < 4 * nbins; i += blockDim.x) s_cnt[i] = 0u;
        __syncthreads();
    }
    const double rm = *mean;
    const float irm = (float)(1.0 / rm), lof = (float)lo, ids = (float)(1.0 / ds);
    const long items = rows ? ncell * n * n : ncell;
    for (long it = blockIdx.x * (long)blockDim.x + threadIdx.x; it < items; it += (long)gridDim.x * blockDim.x) {
        const CellPart<K> part(it, rows);
        double r[b], A[NP];
        load_field<T, K>(u + part.c * 4 * b, 0, r);
#pragma unroll 1
        for (int z = part.z0; z < part.z1; ++z) {
            sf::plane_eval<double, K>(r, t.P[z], A);
#pragma unroll 1
            for (int y = part.y0; y < part.y1; ++y) {
                double q[n], f[n];
                sf::row_eval<double, K>(A, t.P[y], q);
                line_values<K>(t, q, f);
                const int c2 = inner<K>(z) + inner<K>(y);
#pragma unroll
                for (int x = 0; x < n; ++x) {
                    const float fs = narrow(f[x]);
                    if (!(fs > 0.0f) && !positive(f[x])) continue;  // (a density below FP32's range counts)
                    const float g = fs * irm;
                    const float s = (log10f(g) - lof) * ids, fl = floorf(s), fr = s - fl;
                    int bin = -1;
                    if (!(g > 1e-30f && g < 1e30f) || !(fr > tol && fr < 1.0f - tol)) {
                        const double e = floor((log10(f[x] / rm) - lo) / ds);
                        if (e >= 0.0 && e < (double)nbins) bin = (int)e;
                    } else if (fl >= 0.0f && fl < (float)nbins) {
                        bin = (int)fl;
                    }
                    if (bin < 0) continue;
                    const int at = 4 * bin + c2 + inner<K>(x);
                    if (shared)
                        atomicAdd(&s_cnt[at], 1u);
                    else
                        atomicAdd(&cnt[at], 1ull);
                }
            }
        }
    }
    if (shared) {
        __syncthreads();
        for (int i = threadIdx.x; i < 4 * nbins; i += blockDim.x)
            if (s_cnt[i]) atomicAdd(&cnt[i], (unsigned long long)s_cnt[i]);
    }
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // bin i is written over the counts of bin i / 4, which its own pass or an earlier one
    // has read; eight bins of a thread at a time, their loads in flight together.  (Most of
    // many bins are empty: no FP64 conversions there.)
    constexpr int NB = 8;
    for (int i0 = 0; i0 < nbins; i0 += NB * blockDim.x) {
        ulonglong2 q[NB][2];
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int i = i0 + j * blockDim.x + threadIdx.x;
            const ulonglong2* p = reinterpret_cast<const ulonglong2*>(cnt + 4 * i);
            q[j][0] = q[j][1] = make_ulonglong2(0ull, 0ull);
            if (i < nbins) q[j][0] = __ldcg(p), q[j][1] = __ldcg(p + 1);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int i = i0 + j * blockDim.x + threadIdx.x;
            double h = 0.0;
            if (q[j][0].x | q[j][0].y | q[j][1].x | q[j][1].y) {
                h += (double)q[j][0].x * weight.w[0];
                h += (double)q[j][0].y * weight.w[1];
                h += (double)q[j][1].x * weight.w[2];
                h += (double)q[j][1].y * weight.w[3];
            }
            if (i < nbins) acc[i] = h;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *counter = 0u;
}

// structure-function pairs: item = j * npairs + p, five uniforms per item
template <typename T, int K>
__global__ void __launch_bounds__(256) k_structure(const T* __restrict__ u, int N, int nbins, long npairs,
                                                   unsigned long long seed, double lmin, double lmax,
                                                   double* __restrict__ acc)
{
    extern __shared__ double s_acc[];
    double* s_l = s_acc + nbins;  // the bins' separations
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
        s_acc[i] = 0.0;
        s_l[i] = lmin * pow(lmax / lmin, (i + 0.5) / nbins);
    }
    __syncthreads();
    const long items = (long)nbins * npairs;
    const double dN = N;
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < items; e += (long)gridDim.x * blockDim.x) {
        const int j = (int)(e / npairs);
        const double l = s_l[j];
        const unsigned long long n0 = (unsigned long long)e * 5ull;
        double x[3], y[3], va[3], vb[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) x[d] = splitmix_u01(seed, n0 + d);
        const double ct = 2.0 * splitmix_u01(seed, n0 + 3) - 1.0;
        double sp, cp;
        sincospi(2.0 * splitmix_u01(seed, n0 + 4), &sp, &cp);
        const double st = sqrt(fmax(0.0, 1.0 - ct * ct));
        const double dir[3] = {st * cp, st * sp, ct};
#pragma unroll
        for (int d = 0; d < 3; ++d) y[d] = x[d] + l * dir[d];
        velocity_at<T, K>(u, N, dN, x, va);
        velocity_at<T, K>(u, N, dN, y, vb);
        double s = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) s += (va[d] - vb[d]) * (va[d] - vb[d]);
        // one addition per warp where its pairs share the separation (an atomic addition of
        // doubles in shared memory repeats for every lane)
        const unsigned int m = __activemask();
        if (m == 0xffffffffu && __all_sync(m, j == __shfl_sync(m, j, 0))) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(m, s, o);
            if ((threadIdx.x & 31) == 0) atomicAdd(&s_acc[j], s);
        } else {
            atomicAdd(&s_acc[j], s);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nbins; i += blockDim.x)
        if (s_acc[i] != 0.0) atomicAdd(&acc[i], s_acc[i]);
}

// velocity component d on the Ng = (K+1) N grid, x_g = (g + 1/2)/Ng:
// out[(gz Ng + gy) Ng + gx]
// one thread per cell, or per row of points on small meshes: rho and m_d axis by axis at
// the cell's (K+1)^3 grid points
template <typename T, int K>
__global__ void __launch_bounds__(128) k_sample(const T* __restrict__ u, int N, int d, const __grid_constant__ Line t,
                                                bool rows, double* __restrict__ out)
{
    constexpr int p = K + 1, b = Dims<K>::b, NP = sf::npair(K);
    const long Ng = (long)p * N, ncell = (long)N * N * N, items = rows ? ncell * p * p : ncell;
    for (long it = blockIdx.x * (long)blockDim.x + threadIdx.x; it < items; it += (long)gridDim.x * blockDim.x) {
        const CellPart<K> part(it, rows);
        int ix, iy, iz;
        cell_xyz(part.c, N, ix, iy, iz);
        double r[b], m[b], A[NP], M[NP];
        load_field<T, K>(u + part.c * 4 * b, 0, r);
        load_field<T, K>(u + part.c * 4 * b, 1 + d, m);
        double* o = out + ((long)iz * p * Ng + (long)iy * p) * Ng + (long)ix * p;
#pragma unroll 1
        for (int z = part.z0; z < part.z1; ++z) {
            sf::plane_eval<double, K>(r, t.P[z], A);
            sf::plane_eval<double, K>(m, t.P[z], M);
#pragma unroll 1
            for (int y = part.y0; y < part.y1; ++y) {
                double q[p], f[p], g[p];
                sf::row_eval<double, K>(A, t.P[y], q);
                line_values<K>(t, q, f);
                sf::row_eval<double, K>(M, t.P[y], q);
                line_values<K>(t, q, g);
                double* w = o + (z * Ng + y) * Ng;
                if constexpr (p % 2 == 0) {
#pragma unroll
                    for (int x = 0; x < p; x += 2)
                        *reinterpret_cast<double2*>(w + x) = make_double2(g[x] * inverse(f[x]), g[x + 1] * inverse(f[x + 1]));
                } else {
#pragma unroll
                    for (int x = 0; x < p; ++x) w[x] = g[x] * inverse(f[x]);
                }
            }
        }
    }
}

// shell sums of |F|^2 scale^2 over the half spectrum of a real-to-complex
// transform F[gz][gy][kx] (kx = 0..Ng/2); a mode with 0 < kx < Ng/2 stands
// for itself and its conjugate partner.  Bins logarithmic in |kappa|:
// i = floor(log|kappa| / log kmax * nbins), capped at nbins - 1; from single
// precision, and from FP64 where that lands within tol of a bin edge (tol above its
// error: same bins)
// A thread takes the modes (kx, +-a, +-b), (kx, +-b, +-a), 0 <= a <= b, up to eight of
// one |kappa|: one logarithm and one root for them.  The lanes of a warp hold
// consecutive kx, whose bins rise slowly: their sums are added up along the runs of
// equal bins, and one lane of a run adds to the block's sums (an atomic addition of
// doubles in shared memory repeats for every lane that meets the same bin).
// 256^3 points, 100 bins: 0.36 ms with an atomic per mode, 0.13 ms.
__global__ void __launch_bounds__(256) k_shell(const double2* __restrict__ F, int Ng, int nbins, double scale2,
                                               int first, double* __restrict__ power, double* __restrict__ ksum,
                                               unsigned long long* __restrict__ count)
{
    extern __shared__ double s_sh[];
    double* s_pow = s_sh;
    double* s_k = s_sh + nbins;
    unsigned long long* s_cnt = reinterpret_cast<unsigned long long*>(s_sh + 2 * nbins);
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
        s_pow[i] = 0.0;
        s_k[i] = 0.0;
        s_cnt[i] = 0ull;
    }
    __syncthreads();
    const int nh = Ng / 2 + 1, lane = threadIdx.x & 31;
    const long items = (long)nh * (nh + 1) / 2 * nh;
    const double lkmax = log(sqrt(3.0) * Ng / 2.0);
    const float hb = (float)(0.5 * nbins / lkmax), tol = 1e-6f * nbins;
    for (long i0 = blockIdx.x * 256L + (threadIdx.x & ~31); i0 < items; i0 += (long)gridDim.x * 256) {
        const long it = i0 + lane;
        int bin = -1;
        double sp = 0.0, sk = 0.0;
        unsigned int sc = 0u;
        if (it < items) {
            // pair index b (b + 1)/2 + a
            const unsigned int pr = (unsigned int)(it / nh);
            const int kx = (int)(it - (long)pr * nh);
            unsigned int b = (unsigned int)(0.5f * (sqrtf(8.0f * (float)pr + 1.0f) - 1.0f));
            while (b * (b + 1u) / 2u > pr) --b;
            while ((b + 1u) * (b + 2u) / 2u <= pr) ++b;
            const unsigned int a = pr - b * (b + 1u) / 2u;
            const int k2 = kx * kx + (int)(a * a + b * b);  // Ng / 2 <= 2 kMaxN: below 2^24, exact in FP32
            if (k2 > 0) {
                const float fk = (float)k2, s = logf(fk) * hb, fl = floorf(s), fr = s - fl;
                bin = (int)fl;
                if (!(fr > tol && fr < 1.0f - tol)) bin = (int)floor(log(sqrt((double)k2)) / lkmax * nbins);
                if (bin > nbins - 1) bin = nbins - 1;
                if (bin < 0) bin = 0;
                // the grid rows of +-a and +-b
                const unsigned int n = (unsigned int)Ng;
                const unsigned int ra[2] = {a, n - a}, rb[2] = {b, n - b};
                const int na = a == 0u || 2u * a == n ? 1 : 2, nb = b == 0u || 2u * b == n ? 1 : 2;
                const double2* f = F + kx;
                double2 z[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool in = (i & 1) < na && (i >> 1) < nb;
                    const unsigned int p = ra[i & 1], q = rb[i >> 1];
                    z[i] = in ? f[(long)(q * n + p) * nh] : make_double2(0.0, 0.0);
                    z[4 + i] = in && a != b ? f[(long)(p * n + q) * nh] : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) sp = fma(z[i].y, z[i].y, fma(z[i].x, z[i].x, sp));
                // the conjugate modes -kx
                const unsigned int w = kx == 0 || 2 * kx == Ng ? 1u : 2u;
                sp *= w == 1u ? 1.0 : 2.0;
                if (first) {
                    sc = w * (unsigned int)(na * nb * (a != b ? 2 : 1));
                    // the root in single precision and two Newton steps
                    const float sf = fast_sqrt<float>(fk), g[4] = {fk, sf, 0.5f * rcp<float>(sf), (float)sc};
                    double d[4];
                    widen_row<4>(g, d);
                    double dk = d[1] + d[2] * (d[0] - d[1] * d[1]);
                    dk += d[2] * (d[0] - dk * dk);
                    sk = d[3] * dk;
                }
            }
        }
        const int before = __shfl_up_sync(0xffffffffu, bin, 1);
        const unsigned int heads = __ballot_sync(0xffffffffu, lane == 0 || before != bin);
        // heads of the lanes above; bit o - 1 set: lane + o starts another run
        const unsigned int above = lane == 31 ? 0xffffffffu : (heads >> (lane + 1)) | ~(0xffffffffu >> (lane + 1));
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const bool same = (above & ((1u << o) - 1u)) == 0u;
            const double v = __shfl_down_sync(0xffffffffu, sp, o);
            if (same) sp += v;
            if (first) {
                const double y = __shfl_down_sync(0xffffffffu, sk, o);
                const unsigned int c = __shfl_down_sync(0xffffffffu, sc, o);
                if (same) {
                    sk += y;
                    sc += c;
                }
            }
        }
        if ((heads >> lane & 1u) && bin >= 0) {
            atomicAdd(&s_pow[bin], sp * scale2);
            if (first) {
                atomicAdd(&s_k[bin], sk);
                atomicAdd(&s_cnt[bin], (unsigned long long)sc);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
        if (s_pow[i] != 0.0) atomicAdd(&power[i], s_pow[i]);
        if (first && s_cnt[i]) {
            atomicAdd(&ksum[i], s_k[i]);
            atomicAdd(&count[i], s_cnt[i]);
        }
    }
}

static int grid_of(long items, int nsm)
{
    long g = (items + 255) / 256;
    if (g > 16L * nsm) g = 16L * nsm;
    return g < 1 ? 1 : (int)g;
}

// values of the normalised Legendre polynomials at the points x[0..n)
static Line line_of(const double* x, int n)
{
    Line t{};
    for (int a = 0; a < n; ++a) {
        const double y = x[a];
        const double p[4] = {1.0, y, 1.5 * y * y - 0.5, y * (2.5 * y * y - 1.5)};
        for (int m = 0; m < n; ++m) t.P[a][m] = std::sqrt(2.0 * m + 1.0) * p[m];
    }
    return t;
}

// acc: zeroed room of [nbins][4] counts (samples per bin and weight class), the histogram
// [nbins] when the kernel is through; a class's weight: a product of three 1D weights / 8,
// over the cells
template <typename T, int K>
static cudaError_t pdf_k(const Launch& L, const T* u, double lo, double hi, int nbins, double* mean, double* acc)
{
    k_mean_rho<T, K><<<grid_of(L.ncell, L.nsm), 256, 0, L.st>>>(u, L.ncell, mean);
    const double ds = (hi - lo) / nbins;
    // error of the single-precision bin coordinate: the logarithm's (below 1e-6 of
    // its size) over ds and the rounding of the coordinate
    const double tol = 1e-6 * (2.0 + std::fabs(lo) + std::fabs(hi)) / ds + 1e-6 * nbins;
    constexpr int n = K + 1;
    const bool rows = cell_rows(L);
    const long items = rows ? L.ncell * n * n : L.ncell;
    long g = (items + 127) / 128;
    if (g > 16L * L.nsm) g = 16L * L.nsm;
    const double wo = L.r1.w[0], wi = K >= 2 ? L.r1.w[1] : wo;
    ClassWeights w;
    for (int c = 0; c < 4; ++c) w.w[c] = std::pow(wi, c) * std::pow(wo, 3 - c) / 8.0 / (double)L.ncell;
    // counters of the block's own where its samples are no fewer than the bins: 16^3 of degree
    // 3 by rows, 200 bins 53 us so, 109 on the common ones; 8^3, 2000 bins 54 us on the common
    // ones, 108 by cells on the block's own
    const bool shared = (items + g - 1) / g * (rows ? n : n * n * n) >= nbins;
    const size_t sm = shared ? sizeof(unsigned int) * 4 * nbins : 0;
    k_density_pdf<T, K><<<(int)g, 128, sm, L.st>>>(u, L.ncell, line_of(L.r1.x, n), mean, lo, ds,
                                                   (float)std::min(tol, 1.0), nbins, rows, shared,
                                                   w, &L.ctl->cnt_diag, acc);
    return cudaGetLastError();
}

template <typename T, int K>
static cudaError_t sfunc_k(const Launch& L, const T* u, int nbins, long npairs, unsigned long long seed, double* acc)
{
    const double lmin = 1.0 / ((K + 1) * (double)L.N), lmax = 0.5;
    k_structure<T, K><<<grid_of((long)nbins * npairs, L.nsm), 256, 2 * sizeof(double) * nbins, L.st>>>(
        u, L.N, nbins, npairs, seed, lmin, lmax, acc);
    return cudaGetLastError();
}

template <typename T, int K>
static cudaError_t sample_k(const Launch& L, const T* u, int d, double* out)
{
    double x[4];
    for (int a = 0; a <= K; ++a) x[a] = (2.0 * a + 1.0) / (K + 1) - 1.0;
    const bool rows = cell_rows(L);
    long g = (L.ncell * (rows ? (K + 1) * (K + 1) : 1) + 127) / 128;
    if (g > 16L * L.nsm) g = 16L * L.nsm;
    k_sample<T, K><<<(int)g, 128, 0, L.st>>>(u, L.N, d, line_of(x, K + 1), rows, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_density_pdf(const Launch& L, const T* u, double lo, double hi, int nbins, double* mean, double* acc)
{
    DG_DISPATCH(pdf_k, u, lo, hi, nbins, mean, acc);
}

template <typename T>
cudaError_t launch_structure(const Launch& L, const T* u, int nbins, long npairs, unsigned long long seed, double* acc)
{
    DG_DISPATCH(sfunc_k, u, nbins, npairs, seed, acc);
}

template <typename T>
cudaError_t launch_sample(const Launch& L, const T* u, int d, double* out)
{
    DG_DISPATCH(sample_k, u, d, out);
}

cudaError_t launch_shell(const Launch& L, const void* F, int Ng, int nbins, double scale2, int first, double* power,
                         double* ksum, unsigned long long* count)
{
    const long nh = Ng / 2 + 1, total = nh * (nh + 1) / 2 * nh;
    const size_t sm = (sizeof(double) * 2 + sizeof(unsigned long long)) * nbins;
    k_shell<<<grid_of(total, L.nsm), 256, sm, L.st>>>(static_cast<const double2*>(F), Ng, nbins, scale2, first,
                                                       power, ksum, count);
    return cudaGetLastError();
}

#define DG_ANALYSIS_INSTANTIATE(T)                                                                               \
    template cudaError_t launch_density_pdf<T>(const Launch&, const T*, double, double, int, double*, double*);  \
    template cudaError_t launch_structure<T>(const Launch&, const T*, int, long, unsigned long long, double*);   \
    template cudaError_t launch_sample<T>(const Launch&, const T*, int, double*);
DG_ANALYSIS_INSTANTIATE(float)
DG_ANALYSIS_INSTANTIATE(double)

}  // namespace dg
