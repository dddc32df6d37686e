// gsm_fx3_a.cu -- the fixed-length passes (gsm_fx3.cuh) of R = 8, 5.
#include "gsm_fx3.cuh"

namespace gsm {

template void f3_launch<8>(const F3Call &c, int pass);
template void f3_launch<5>(const F3Call &c, int pass);

}  // namespace gsm
