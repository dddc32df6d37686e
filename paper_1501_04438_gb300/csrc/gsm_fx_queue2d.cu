// gsm_fx_queue2d.cu -- fixed point: the batch queue kernel of 2D plans.
#include "gsm_fx_queue.cuh"

namespace gsm {

cudaError_t launch_queue_fx2(const QueueArgs &a, size_t smem, cudaStream_t st, bool dry)
{
    return launch_queue_d<FX, 2>(a, smem, st, dry);
}

}  // namespace gsm
