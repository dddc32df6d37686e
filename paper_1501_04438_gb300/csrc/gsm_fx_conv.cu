// gsm_fx_conv.cu -- fixed point: the conv pass and the split passes of long 2D lines.
#include "gsm_fx_kernels.cuh"
#include "gsm_fx_split.cuh"

namespace gsm {

cudaError_t fx_raise_conv_smem(const Plan *p, const PassCfg &c)
{
    cudaError_t e = fixed_raise(p, p->d == 3 ? 2 : 1, c);
    with_emax(c, [&](auto E) { if (e == cudaSuccess) e = raise_smem(k_fx_conv<E(), Sched, Sched>, c.smem); });
    return e;
}

// half: the half length (its schedules are the default ones, make_split_tables and
// make_xsplit_tables)
cudaError_t fx_raise_split_smem(bool conv, int half, size_t smem)
{
    const cudaError_t e = split_raise<16, Sched, Sched>(conv, smem);
    if (e != cudaSuccess) return e;
#define GSM_FX_CASE(M) case M: return FixedSplit<M>::raise(conv, smem);
    switch (half) { GSM_FX_HALVES(GSM_FX_CASE) }
#undef GSM_FX_CASE
    return cudaSuccess;
}

void fx_launch_conv(const FxCall &a, const PassCfg &c)
{
    const Plan *p = a.p;
    if (fixed_launch(a, p->d == 3 ? 2 : 1, c)) return;
    const int z = p->d - 1, ny = p->n[1], hx = p->n[0] + 1, My = p->d == 3 ? p->M[1] : 1;
    const int2 *mult = static_cast<const int2 *>(p->d_mult);
    const int4 *tw = static_cast<const int4 *>(p->d_tw[z]), *twi = static_cast<const int4 *>(p->d_twi[z]);
    fxc *W = static_cast<fxc *>(p->d == 3 ? a.W2 : a.W1);
    const dim3 g = p->d == 3 ? dim3((My + c.nl - 1) / c.nl, hx) : dim3((hx + c.nl - 1) / c.nl), b(c.gthr, c.nl);
    with_emax(c, [&](auto E) {
        k_fx_conv<E(), Sched, Sched><<<g, b, c.smem, a.st>>>(
            W, mult, p->d_mrow, a.ex, p->d == 3 ? hx * My : hx, p->n[z], p->d == 3, My, ny + 1, p->sched_f[z],
            p->sched_i[z], c.nl, tw, twi, p->mult_full ? 1 : 0);
    });
}

// A split pass (0 xf, 1 conv, 2 xi) of a 2D plan.
void fx_launch_split(const FxCall &a, int pass)
{
    const Plan *p = a.p;
    const Sched &f = pass == 1 ? p->sched_hf : p->sched_xh;
    if ((p->opt.debug & 4) == 0) {
#define GSM_FX_CASE(M) case M: return FixedSplit<M>::launch(a, pass);
        switch (f.M) { GSM_FX_HALVES(GSM_FX_CASE) }
#undef GSM_FX_CASE
    }
    split_launch<16>(a, pass, f, pass == 1 ? p->sched_hi : f);
}

}  // namespace gsm
