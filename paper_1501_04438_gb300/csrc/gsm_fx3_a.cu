// gsm_fx3_a.cu -- the fixed-length passes (gsm_fx3.cuh) of R = 8, 5.
#include "gsm_fx3.cuh"

namespace gsm {

template cudaError_t f3_raise_smem<8>(const Plan *p);
template void f3_launch<8>(const FxCall &c, int pass);
template cudaError_t f3_raise_smem<5>(const Plan *p);
template void f3_launch<5>(const FxCall &c, int pass);

}  // namespace gsm
