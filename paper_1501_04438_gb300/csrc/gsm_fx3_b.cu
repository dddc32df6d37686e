// gsm_fx3_b.cu -- the fixed-length passes (gsm_fx3.cuh) of R = 6, 4.
#include "gsm_fx3.cuh"

namespace gsm {

template cudaError_t f3_raise_smem<6>(const Plan *p);
template void f3_launch<6>(const FxCall &c, int pass);
template cudaError_t f3_raise_smem<4>(const Plan *p);
template void f3_launch<4>(const FxCall &c, int pass);

}  // namespace gsm
