// gsm_fx_split_e.cu -- split passes of half lengths known at compile time (gsm_fx_split.cuh).
#define GSM_FX_LENGTH_UNIT
#include "gsm_fx_split.cuh"

namespace gsm {
GSM_FX_HALVES_E(GSM_FX_DEFINE_HALF)
}  // namespace gsm
