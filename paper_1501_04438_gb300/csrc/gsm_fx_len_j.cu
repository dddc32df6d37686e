// gsm_fx_len_j.cu -- fixed-point passes of padded lengths known at compile time (gsm_fx_kernels.cuh).
#define GSM_FX_LENGTH_UNIT
#include "gsm_fx_kernels.cuh"

namespace gsm {
GSM_FX_LENGTHS_J(GSM_FX_DEFINE)
}  // namespace gsm
