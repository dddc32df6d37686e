"""Every way a batch applies a plan (queue, one launch per pass for plans of one size, alone), mixed in
one call, against gsm_apply: equal bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SPECS = {
    "3d": [(32, 32, 32), (64, 64, 64), (24, 20, 16), (60, 32, 90), (192, 32, 32), (64, 64, 64), (100, 60, 48),
           (32, 32, 32), (32, 64, 24), (192, 32, 32), (8, 8, 256)],
    "2d": [(32, 32), (192, 64), (54, 64), (256, 128), (192, 64), (32, 32), (54, 40), (256, 256), (24, 192)],
}


@pytest.mark.parametrize("precision", ["fp64", "fp32x2", "fp32"])
@pytest.mark.parametrize("dim", ["3d", "2d"])
def test_batch_gives_the_bits_of_single_applies(dim, precision):
    import torch
    import paper_1501_04438_gb300 as gsm
    rng = np.random.default_rng(9)
    dt = torch.float32 if precision == "fp32" else torch.float64
    kernels = {"3d": ("coulomb3d", "power3d"), "2d": ("coulomb2d", "poisson2d")}[dim]
    plans = [gsm.Plan(kernels[i % 2], 4.0, n, precision=precision) for i, n in enumerate(SPECS[dim])]
    rhos = [torch.tensor(rng.standard_normal(n[::-1]), dtype=dt, device="cuda") for n in SPECS[dim]]
    single = [p.apply(r) for p, r in zip(plans, rhos)]
    batch = gsm.Batch(plans, rhos)
    for outs in (gsm.apply_batched(plans, rhos), batch.launch()):
        torch.cuda.synchronize()
        assert [n for n, a, b in zip(SPECS[dim], outs, single) if not torch.equal(a, b)] == []
    batch.destroy()


def test_more_plans_of_one_size_than_one_launch_takes():
    """50 plans of one size: a launch of 48 and one of 2."""
    import torch
    import paper_1501_04438_gb300 as gsm
    rng = np.random.default_rng(10)
    plans = [gsm.Plan("coulomb2d", 4.0, (192, 32)) for _ in range(50)]
    rhos = [torch.tensor(rng.standard_normal((32, 192)), device="cuda") for _ in plans]
    for a, p, r in zip(gsm.apply_batched(plans, rhos), plans, rhos):
        assert torch.equal(a, p.apply(r))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_groups_before_the_queue_and_streams_beside_the_callers(precision):
    """Four small plans of one size (grouped), two of another (queue), more plans applied alone than
    there are streams, several times in a row on a stream of the caller's, inputs rewritten on it between
    calls: equal bits, and the graph's too."""
    import torch
    import paper_1501_04438_gb300 as gsm
    rng = np.random.default_rng(11)
    dt = torch.float32 if precision == "fp32" else torch.float64
    sizes = [(32, 32, 32)] * 5 + [(64, 32, 32)] * 2 + [(64, 36, 48), (32, 60, 40), (48, 64, 50), (40, 32, 72)] * 3
    plans = [gsm.Plan("coulomb3d", 4.0, n, precision=precision) for n in sizes]
    data = [[torch.tensor(rng.standard_normal(n[::-1]), dtype=dt, device="cuda") for n in sizes] for _ in range(3)]
    want = [[p.apply(r) for p, r in zip(plans, d)] for d in data]
    rhos = [torch.empty_like(r) for r in data[0]]
    outs = [torch.empty_like(r) for r in rhos]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        batch = gsm.Batch(plans, rhos, outs, stream=stream)
        for launch in (lambda: gsm.apply_batched(plans, rhos, outs, stream=stream), lambda: batch.launch(stream=stream)):
            for d, w in zip(data, want):
                for r, x in zip(rhos, d):
                    r.copy_(x)
                launch()
                got = [o.clone() for o in outs]
                stream.synchronize()
                assert [n for n, a, b in zip(sizes, got, w) if not torch.equal(a, b)] == []
        batch.destroy()
