// sum-factorised kernels, f32, degree 1
#include "dg_sf_impl.cuh"
namespace dg {
DG_SF_INSTANTIATE(float, 1)
}
