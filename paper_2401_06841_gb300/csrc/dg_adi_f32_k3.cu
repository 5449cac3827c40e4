// dg_adi_f32_k3.cu -- F32 degree-3 launcher of the adiabatic system.
#include "dg_adi_impl.cuh"

namespace dg {
DG_ADI_K3_INSTANTIATE(float)
}
