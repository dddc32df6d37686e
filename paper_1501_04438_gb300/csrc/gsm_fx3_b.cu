// gsm_fx3_b.cu -- the fixed-length passes (gsm_fx3.cuh) of R = 6, 4.
#include "gsm_fx3.cuh"

namespace gsm {

template void f3_launch<6>(const F3Call &c, int pass);
template void f3_launch<4>(const F3Call &c, int pass);

}  // namespace gsm
