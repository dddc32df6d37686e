// gsm_fx3_c.cu -- the fixed-length passes (gsm_fx3.cuh) of R = 3, 2, 1.
#include "gsm_fx3.cuh"

namespace gsm {

template cudaError_t f3_raise_smem<3>(const Plan *p);
template void f3_launch<3>(const FxCall &c, int pass);
template cudaError_t f3_raise_smem<2>(const Plan *p);
template void f3_launch<2>(const FxCall &c, int pass);
template cudaError_t f3_raise_smem<1>(const Plan *p);
template void f3_launch<1>(const FxCall &c, int pass);

}  // namespace gsm
