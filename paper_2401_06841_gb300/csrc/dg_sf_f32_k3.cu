// sum-factorised kernels, f32, degree 3
#include "dg_sf_impl.cuh"
namespace dg {
DG_SF_INSTANTIATE(float, 3)
}
