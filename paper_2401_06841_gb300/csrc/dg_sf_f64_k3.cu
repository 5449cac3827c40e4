// sum-factorised kernels, f64, degree 3
#include "dg_sf_impl.cuh"
namespace dg {
DG_SF_INSTANTIATE(double, 3)
}
