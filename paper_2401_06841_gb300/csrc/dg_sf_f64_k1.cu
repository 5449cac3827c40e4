// sum-factorised kernels, f64, degree 1
#include "dg_sf_impl.cuh"
namespace dg {
DG_SF_INSTANTIATE(double, 1)
}
