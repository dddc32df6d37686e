// gsm_f3_f32.cu -- the FP32 fixed-length passes (gsm_f3_f32.cuh) and their tables.
#include "gsm_f3_f32.cuh"

namespace gsm {
namespace {

// exp(-2 pi i j t / (R Ns)) at Ns - r0 + (t - 1) Ns + j (see fx_stage_table)
__global__ void k_f32_stage_twiddles(Sched sc, float2 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int j = i, Ns = sc.r[0];
    if (i >= sc.M - Ns) return;
    for (int st = 1; st < sc.nst; ++st) {
        const int R = sc.r[st], cnt = (R - 1) * Ns;
        if (j < cnt) {
            double sn, cs;
            sincospi(2.0 * (double)((long)(j % Ns) * (j / Ns + 1)) / (double)((long)R * Ns), &sn, &cs);
            out[i] = make_float2((float)cs, (float)-sn);
            return;
        }
        j -= cnt;
        Ns *= R;
    }
}

}  // namespace

void launch_f32_stage_twiddles(const Sched &sc, float2 *out, cudaStream_t st)
{
    k_f32_stage_twiddles<<<(sc.M + 127) / 128, 128, 0, st>>>(sc, out);
}

template void f3f_launch<1>(const F3Call &c, int pass);
template void f3f_launch<2>(const F3Call &c, int pass);
template void f3f_launch<3>(const F3Call &c, int pass);
template void f3f_launch<4>(const F3Call &c, int pass);
template void f3f_launch<5>(const F3Call &c, int pass);
template void f3f_launch<6>(const F3Call &c, int pass);

}  // namespace gsm
