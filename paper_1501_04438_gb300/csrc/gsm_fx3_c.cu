// gsm_fx3_c.cu -- the fixed-length passes (gsm_fx3.cuh) of R = 3, 2, 1.
#include "gsm_fx3.cuh"

namespace gsm {

template void f3_launch<3>(const F3Call &c, int pass);
template void f3_launch<2>(const F3Call &c, int pass);
template void f3_launch<1>(const F3Call &c, int pass);

}  // namespace gsm
