// gsm_fx_len_k.cu -- fixed-point passes of padded lengths known at compile time (gsm_fx_kernels.cuh).
#define GSM_FX_LENGTH_UNIT
#include "gsm_fx_kernels.cuh"

namespace gsm {
GSM_FX_LENGTHS_K(GSM_FX_DEFINE)
}  // namespace gsm
