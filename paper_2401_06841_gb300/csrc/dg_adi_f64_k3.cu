// dg_adi_f64_k3.cu -- F64 degree-3 launcher of the adiabatic system.
#include "dg_adi_impl.cuh"

namespace dg {
DG_ADI_K3_INSTANTIATE(double)
}
