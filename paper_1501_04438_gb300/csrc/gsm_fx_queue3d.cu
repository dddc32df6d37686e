// gsm_fx_queue3d.cu -- fixed point: the batch queue kernel of 3D plans.
#include "gsm_fx_queue.cuh"

namespace gsm {

cudaError_t launch_queue_fx3(const QueueArgs &a, size_t smem, cudaStream_t st, bool dry)
{
    return launch_queue_d<FX, 3>(a, smem, st, dry);
}

}  // namespace gsm
