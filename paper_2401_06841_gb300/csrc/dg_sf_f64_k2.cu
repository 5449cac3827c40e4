// sum-factorised kernels, f64, degree 2
#include "dg_sf_impl.cuh"
namespace dg {
DG_SF_INSTANTIATE(double, 2)
}
