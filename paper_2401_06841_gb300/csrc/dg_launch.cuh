// dg_launch.cuh -- internal launch interface between the host API and the
// kernel translation units (one per element type).
#pragma once

#include <cuda_runtime.h>

#include "dg_common.cuh"

namespace dg {

struct Launch {
    cudaStream_t st;
    int K;
    int N;
    long ncell;
    Phys ph;
    const void* tab;     // tables of the element type in use (auxiliary kernels)
    const void* ttab;    // tables of the tile kernels
    Ctl* ctl;
    double* partials;    // [16][kMaxGrid]
    int nsm;             // multiprocessors on the device
    int bk;              // 0: CUDA-core products, 1: split-BF16 x3 tensor-core products
    Rule1 r1;            // the 1D Gauss rule
    void* gtab;          // forcing: 1D factors [N][17][k+1][2] of the element type
};

template <typename T>
cudaError_t setup_kernels(int K);
// tile kernel modes: 0 projection only (velocity projection, forcing sums,
// CFL dt with F_DT), 1 right-hand side only, 2 right-hand side + SSP-RK stage
// (+ the next stage's projection with F_NEXTPROJ), 3 as 2 with the projection
// of |v| (vabs_out) for the learned sensor
struct TileLaunch {
    int mode;
    const void* u_in;
    const void* u_n;
    void* out;
    const void* vh_in;
    void* vh_out;
    const void* ahat;
    double rk_a, rk_b;
    double dt_pimax;
    int flags;
    int abar_in, abar_out;
    const float* nu;     // learned sensor: per-cell coefficient
    void* vabs_out;      // learned sensor: projection of |v|
    float* nu_next;      // learned sensor: coefficient of the output, evaluated in the kernel (mode 3)
    const uint32_t* mlp; // learned sensor: packed network for nu_next
    unsigned char* trouble;  // positivity by repetition: per-cell marks of the stage (or nullptr)
};
template <typename T>
cudaError_t launch_tile(const Launch& L, const TileLaunch& t);
// forcing projection (dg_force.cuh): the 1D factors L.gtab of a mesh, once per
// context, and the projection of a list of modes
struct ForceModes;
template <typename T>
cudaError_t launch_force_axis(const Launch& L);
template <typename T>
cudaError_t launch_force(const Launch& L, const ForceModes& fm, const int* modes, const double* amp, T* ahat);
template <typename T>
cudaError_t launch_diag(const Launch& L, const T* u, const T* ahat, double dt_pimax, int flags);
template <typename T>
cudaError_t launch_l1(const Launch& L, const T* uA, const T* uB);
// positivity by repetition: every marked cell of u [c][4][b] is unmarked and its
// modes l > 0 scaled by 1/2 (level 0, 1) or 0 (level 2), its level incremented;
// a marked cell whose modes l > 0 are all zero sets DG_ST_FLAT_ instead
template <typename T>
cudaError_t launch_flatten(const Launch& L, T* u, unsigned char* trouble, unsigned char* level);

// adiabatic system (dg_sf_adi.cuh): mode 0 projection of v and p (+ CFL bound
// with F_DT, forcing sums with F_FORCE), 1 right-hand side, 2 stage
// (right-hand side, SSP-RK combine, positivity of density and pressure; with
// F_SELFPROJ the projections of its input are written to pr_in first), 3 isothermal
// reset of the thermal energy (in place)
enum { ADI_PROJECT = 0, ADI_RHS = 1, ADI_STAGE = 2, ADI_RESET = 3 };
struct AdiLaunch {
    int mode;
    const void* u_in;
    const void* u_n;
    void* out;
    const void* pr_in;
    void* pr_out;
    double rk_a, rk_b;
    double dt_pimax;
    int flags;
    const void* ahat;       // driving (F_FORCE)
    int abar_in, abar_out;  // ctl->abar2 slots
    double beta;            // stage weight of the injected energy
    double cs_reset;        // reset mode
    double kap;             // energy offset of the stored states: e_s = e - kap rho
    int bc[3];              // boundaries per axis (DG_BC_*)
    double inflow[5];       // DG_BC_INFLOW: rho, v, p at the face at coordinate 0
};
template <typename T>
cudaError_t launch_adi(const Launch& L, double gamma, const AdiLaunch& t);
// per-block FP64 totals [nblocks][8]: mass, momentum (3), energy, kinetic
// energy, min rho and min p at the volume points
template <typename T>
cudaError_t launch_adi_totals(const Launch& L, double gamma, double kap, const void* u, double* partials, int* nblocks);
// e_s += d rho on a state (a change of the energy offset)
template <typename T>
cudaError_t launch_adi_shift(const Launch& L, void* u, double d);

// turbulence statistics (dg_analysis.cu)
template <typename T>
cudaError_t launch_density_pdf(const Launch& L, const T* u, double lo, double hi, int nbins, double* mean, double* acc);
template <typename T>
cudaError_t launch_structure(const Launch& L, const T* u, int nbins, long npairs, unsigned long long seed, double* acc);
template <typename T>
cudaError_t launch_sample(const Launch& L, const T* u, int d, double* out);
cudaError_t launch_shell(const Launch& L, const void* F, int Ng, int nbins, double scale2, int first, double* power,
                         double* ksum, unsigned long long* count);

// learned viscosity sensor
constexpr int kMlpHidden = 64;
constexpr int kMlpBatchMax = 4096;
inline int mlp_params(int D) { return kMlpHidden * D + kMlpHidden + kMlpHidden * kMlpHidden + 2 * kMlpHidden + 1; }
// partial gradient sums: pairs of floats per block of 32 samples (the largest network: D = 40)
inline size_t mlp_work_floats_host() { return (size_t)(kMlpBatchMax / 32) * 2 * (mlp_params(40) + 1); }
cudaError_t mlp_train_pass(cudaStream_t st, int D, const float* W, const float* X, const float* Y, int n, float* work,
                           float* G, double* loss);
cudaError_t mlp_adam(cudaStream_t st, int P, float* W, const float* G, float* m, float* v, float lr, float b1, float b2,
                     float eps, float c1, float c2);
template <typename T>
cudaError_t mlp_infer(const Launch& L, const T* u, const T* vabs, const float* X, long n, const uint32_t* packed,
                      float* nu, float* y);
template <typename T>
cudaError_t launch_features(const Launch& L, const T* u, const T* vabs, const T* phiv, double dt, float* X, float* Y);

}  // namespace dg
