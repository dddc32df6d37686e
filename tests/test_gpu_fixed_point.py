"""GPU tests of the block fixed-point transforms of the FP64 and FP32X2 passes:
the accuracy of single lines against long double, and what one exponent per
line has to carry (magnitudes far apart, scaling, zeros, subnormals,
infinities and NaN)."""
import struct

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gsm():
    import paper_1501_04438_gb300 as m
    return m


def _dft_long(x, sign):
    """Rows of x transformed in long double (matrix product with a table of w_M^m)."""
    M = x.shape[-1]
    m = np.arange(M)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    ang = sign * 2 * pi * m.astype(np.longdouble) / M
    c, s = np.cos(ang), np.sin(ang)
    idx = np.outer(m, m) % M
    re, im = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
    return re @ c[idx] - im @ s[idx], re @ s[idx] + im @ c[idx]


# lengths around the kernels' edges: two stages, odd radices, the last length with one scale per
# line (512) and the first rescaled after every stage (540), several threads groups
@pytest.mark.parametrize("M", [16, 40, 100, 128, 320, 384, 512, 540, 1024, 2000])
@pytest.mark.parametrize("sign", [-1, 1])
def test_line_errors_are_those_of_fp64_or_less(gsm, M, sign):
    """Relative rms error of a transform below 2^-53 sqrt(log2 M): the usual estimate of an FP64
    FFT, u times the root of its number of radix-2 levels."""
    import torch
    rng = np.random.default_rng(M)
    g = np.exp(-((np.arange(M) - 0.45 * M) / (0.06 * M)) ** 2)
    x = np.stack([rng.standard_normal(M) + 1j * rng.standard_normal(M), g * (1 + 0.3j),
                  (np.arange(M) == 3) * (1.0 + 0j), g * (1e-3 * rng.standard_normal(M) + 1j * rng.standard_normal(M)),
                  np.where(np.arange(M) % 2 == 0, 1.0, 1e-14) * rng.standard_normal(M) + 0j])
    re, im = _dft_long(x, sign)
    got = gsm.fft_lines(torch.tensor(x, device="cuda"), sign, "fp64").cpu().numpy()
    err = np.sqrt(np.sum((got.real - re) ** 2 + (got.imag - im) ** 2, axis=1) / np.sum(re ** 2 + im ** 2, axis=1))
    assert np.all(err.astype(float) < 2.0 ** -53 * np.sqrt(np.log2(M))), err


GRIDS = [("coulomb3d", (24, 20, 16)), ("poisson2d", (40, 54)), ("coulomb2d", (16, 2048)), ("coulomb2d", (2048, 16))]


@pytest.mark.parametrize("precision", ["fp64", "fp32x2"])
@pytest.mark.parametrize("kernel,n", GRIDS, ids=[f"{k}-{'x'.join(map(str, n))}" for k, n in GRIDS])
def test_scaling_zeros_and_non_finite_values(gsm, kernel, n, precision):
    """Powers of two scale the result exactly (exponents only), a density of zeros gives zeros,
    subnormal results are rounded once more, an infinity or a NaN makes every output NaN."""
    import torch
    plan = gsm.Plan(kernel, 4.0, n, precision=precision)
    rho = torch.tensor(np.random.default_rng(5).standard_normal(n[::-1]), device="cuda")
    u = plan.apply(rho)
    for k in (-600, 1, 600):
        assert torch.equal(plan.apply(rho * 2.0 ** k), u * 2.0 ** k)
    if kernel.startswith("coulomb"):
        # the input's rounding to multiples of 2^-1074, half a unit each, through the (positive)
        # kernel's row sums, and the output's own rounding
        tiny = plan.apply(rho * 2.0 ** -500 * 2.0 ** -540)
        rows = float(plan.apply(torch.ones_like(rho)).max())
        err = (tiny - u * 2.0 ** -500 * 2.0 ** -540).abs().max() * 2.0 ** 500 * 2.0 ** 574
        assert float(err) <= rows + 2.0
    assert torch.equal(plan.apply(torch.zeros_like(rho)), torch.zeros_like(rho))
    for bad in (float("nan"), float("inf"), -float("inf")):
        r = rho.clone()
        r.view(-1)[r.numel() // 3] = bad
        assert bool(torch.isnan(plan.apply(r)).all())


@pytest.mark.parametrize("kernel,n", GRIDS[:2], ids=["3d", "2d"])
def test_lines_of_magnitudes_far_apart(gsm, kernel, n):
    """Rows, columns and planes whose magnitudes differ by up to 1e30, against the oracle in the
    relative max norm (FP64's own tolerance)."""
    import torch
    rng = np.random.default_rng(8)
    rho = rng.standard_normal(n[::-1])
    for axis, m in enumerate(rho.shape):
        shape = [1] * rho.ndim
        shape[axis] = m
        rho = rho * (10.0 ** rng.uniform(-15, 0, size=m)).reshape(shape)
    plan = gsm.Plan(kernel, 4.0, n)
    u = plan.apply(torch.tensor(rho, device="cuda")).cpu().numpy()
    uo, _ = oracle.apply(kernel, rho, 4.0, taylor_mode=1)
    assert np.max(np.abs(u - uo)) / np.max(np.abs(uo)) < 1e-12


# padded lengths 64 R with kernels of their own, as the x, y and z lines of grids whose other
# axes leave the last CTA ragged, and 2D; general dipole axes take the half-spectrum multiplier
FIXED = (32, 64, 96, 128, 160, 192, 256)
ROLES = [("coulomb3d", lambda N: (N, 10, 8)), ("coulomb3d", lambda N: (10, N, 18)), ("dipolar3d", lambda N: (8, 10, N)),
         ("coulomb2d", lambda N: (N, 54)), ("ds2d", lambda N: (18, N))]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("role", range(len(ROLES)), ids=["x", "y", "z_full", "x2d", "y2d"])
@pytest.mark.parametrize("N", FIXED)
def test_fixed_length_kernels(gsm, N, role, precision):
    """The fixed-length kernels against the oracle and against the kernels of any length
    (options.debug bit 2): relative differences of a few roundings of the result, u log2 of the
    padded volume with u = 2^-53 or, in FP32 (whose steps may be ordered differently), 2^-24 with
    the factor 4 of the FP32 tolerance."""
    import torch
    kernel, shape = ROLES[role]
    n = shape(N)
    kw = dict(dip_n=(0.6, 0.0, 0.8), dip_m=(0.0, 0.8, 0.6)) if kernel == "dipolar3d" else {}
    rho = np.random.default_rng(N).standard_normal(n[::-1])
    r = torch.tensor(rho, dtype=torch.float32 if precision == "fp32" else torch.float64, device="cuda")
    u = gsm.Plan(kernel, 4.0, n, precision=precision, **kw).apply(r).double().cpu().numpy()
    v = gsm.Plan(kernel, 4.0, n, precision=precision, debug=4, **kw).apply(r).double().cpu().numpy()
    unit = 4 * 2.0 ** -24 if precision == "fp32" else 2.0 ** -53
    assert np.max(np.abs(u - v)) / np.max(np.abs(u)) < unit * np.log2(np.prod([2.0 * m for m in n]))
    # ds2d: ln r, see the split-conv test on white noise; dipolar3d: the two Gaussian sums, each
    # within 2e-15, differ by up to 3e-12 of max|u| after the derivatives on these spacings (the
    # FP64 arithmetic gave the same difference)
    if kernel.startswith("coulomb"):
        uo, _ = oracle.apply(kernel, r.double().cpu().numpy(), 4.0, taylor_mode=1, **kw)
        bound = unit * np.log2(2 * max(n)) if precision == "fp32" else 1e-12
        assert np.max(np.abs(u - uo)) / np.max(np.abs(uo)) < bound


# every length whose default schedule is compiled in, as x, y and z lines of grids whose other axes
# have none, with the octant and (general dipole axes) the half-spectrum multiplier; n = 216 has none
COMPILED = [24, 30, 36, 40, 48, 50, 54, 60, 72, 80, 90, 100, 108, 120, 144, 150, 162, 180, 200, 216, 240, 250]
LONG = [(512, 18), (18, 512), (1024, 10), (10, 1024), (2048, 18), (18, 2048), (4096, 10), (12, 4096)]
CASES = ([("coulomb3d", s) for N in COMPILED for s in ((N, 10, 18), (10, N, 18), (10, 18, N))] +
         [("dipolar3d", (10, 18, N)) for N in COMPILED] + [("ds2d", s) for s in LONG])


@pytest.mark.parametrize("kernel,n", CASES, ids=[k[0] + "x".join(map(str, s)) for k, s in CASES])
def test_schedules_known_at_compile_time(gsm, kernel, n):
    """The kernels of a compiled-in schedule run the integer operations of the kernels of any
    schedule (options.debug bit 2) in the same order: equal bits."""
    import torch
    kw = dict(dip_n=(0.6, 0.0, 0.8), dip_m=(0.0, 0.8, 0.6)) if kernel == "dipolar3d" else {}
    r = torch.tensor(np.random.default_rng(sum(n)).standard_normal(n[::-1]), device="cuda")
    assert torch.equal(gsm.Plan(kernel, 4.0, n, **kw).apply(r), gsm.Plan(kernel, 4.0, n, debug=4, **kw).apply(r))


@pytest.mark.parametrize("n", [(2048, 18), (2160, 10), (4096, 10)], ids=lambda n: "x".join(map(str, n)))
def test_split_inverse_x(gsm, n):
    """Long x lines as two halves on a CTA pair against whole lines (debug bit 1): a few roundings of
    the result, u log2 of the padded size."""
    import torch
    r = torch.tensor(np.random.default_rng(n[0]).standard_normal(n[::-1]), device="cuda")
    u = gsm.Plan("coulomb2d", 4.0, n).apply(r)
    for debug in (2, 6):
        v = gsm.Plan("coulomb2d", 4.0, n, debug=debug).apply(r)
        assert float((u - v).abs().max() / v.abs().max()) < 2.0 ** -53 * np.log2(4.0 * n[0] * n[1])


@pytest.mark.parametrize("N", [96, 160, 192])
def test_conv_of_several_sync_groups_repeats_its_bits(gsm, N):
    """The conv lines of a CTA whose sync groups are not ordered against one another (three to six
    warps each): 200 applies with equal bits."""
    import torch
    r = torch.tensor(np.random.default_rng(N).standard_normal((N, 60, 64)), device="cuda")
    plan = gsm.Plan("coulomb3d", 4.0, (64, 60, N))
    u = plan.apply(r)
    for _ in range(200):
        assert torch.equal(plan.apply(r), u)


def _fnv1a(data):
    h = 14695981039346656037
    for b in data:
        h = ((h ^ b) * 1099511628211) & 0xFFFFFFFFFFFFFFFF
    return h


def _resaved(data, **fields):
    """A saved plan's bytes with header fields replaced: version, nl and emax (one value for every
    pass)."""
    b = bytearray(data)
    if "version" in fields:
        b[8:12] = struct.pack("<I", fields["version"])
    for at, key in ((52, "nl"), (72, "emax")):
        if key in fields:
            b[at:at + 20] = struct.pack("<5i", *[fields[key]] * 5)
    b[-8:] = struct.pack("<Q", _fnv1a(b[:-8]))
    return bytes(b)


@pytest.mark.parametrize("nl", [1, 2, 3, 4, 8])
@pytest.mark.parametrize("n", [(216, 20, 18), (18, 216, 20), (20, 18, 216), (100, 60, 48), (40, 250, 54), (512, 30)],
                         ids=lambda n: "x".join(map(str, n)))
def test_lines_per_cta_do_not_change_the_bits(gsm, n, nl):
    """Compiled-in schedules with every number of lines per CTA (a number that does not fit keeps the
    default) against the kernels of any schedule, and 16 values per thread, which are those."""
    import torch
    kernel = "coulomb3d" if len(n) == 3 else "coulomb2d"
    r = torch.tensor(np.random.default_rng(nl).standard_normal(n[::-1]), device="cuda")
    data = gsm.Plan(kernel, 4.0, n).save()
    u = gsm.Plan(kernel, 4.0, n, debug=4).apply(r)
    for emax in (8, 16):
        assert torch.equal(gsm.Plan.load(_resaved(data, nl=nl, emax=emax)).apply(r), u)


@pytest.mark.parametrize("n", [(216, 60, 96), (64, 216, 36), (60, 36, 216), (150, 90, 120), (96, 128, 160), (32, 64, 128),
                               (256, 60, 32), (60, 256, 48), (48, 60, 256), (32, 256), (128, 160), (64, 96), (256, 32),
                               (60, 90), (250, 120)], ids=lambda n: "x".join(map(str, n)))
def test_larger_grids_have_the_general_kernels_bits(gsm, n):
    """Many CTAs per pass: compiled-in schedules, and the lengths 64 R whose stages are those of the
    default schedule (all but n = 192), against the kernels of any schedule."""
    import torch
    r = torch.tensor(np.random.default_rng(sum(n)).standard_normal(n[::-1]), device="cuda")
    kernel = "coulomb3d" if len(n) == 3 else "coulomb2d"
    assert torch.equal(gsm.Plan(kernel, 4.0, n).apply(r), gsm.Plan(kernel, 4.0, n, debug=4).apply(r))


@pytest.mark.parametrize("precision", ["fp64", "fp32x2", "fp32"])
def test_plans_saved_before_fixed_point(gsm, precision):
    """A plan saved in format version 3 with the schedules of that time (on the conv axis forward and
    inverse alike) is read; in fixed point it takes the default schedules, FP32 keeps the stored ones."""
    n = (100, 24, 18)
    plan = gsm.Plan("coulomb3d", 4.0, n, precision=precision)
    fresh = plan.info()
    plan.set_schedule(0, [4, 2, 5, 5])
    loaded = gsm.Plan.load(_resaved(plan.save(), version=3)).info()
    assert loaded["radix_fwd"][0] == (plan.info() if precision == "fp32" else fresh)["radix_fwd"][0]
    assert gsm.Plan.load(plan.save()).info()["radix_fwd"][0] == plan.info()["radix_fwd"][0]


def test_tuned_choices_of_another_version_are_not_used(gsm, tmp_path, monkeypatch):
    """Entries of the tuner's cache are used again by the version that wrote them and by no other."""
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("GSM_AUTOTUNE_CACHE", str(cache))
    n = (54, 40, 36)
    assert "cached" not in gsm.Plan("coulomb3d", 4.0, n).autotune()
    entries = cache.read_text()
    assert entries.startswith("v6 ") and gsm.Plan("coulomb3d", 4.0, n).autotune().count(" cached ") == 5
    cache.write_text(entries.replace("v6 ", "v5 "))
    assert "cached" not in gsm.Plan("coulomb3d", 4.0, n).autotune()


LONG = sorted(n for n in (2 ** a * 3 ** b * 5 ** c for a in range(1, 13) for b in range(8) for c in range(6))
              if 256 < n <= 4096)


@pytest.mark.parametrize("n", LONG)
def test_long_lengths_have_the_general_kernels_bits(gsm, n):
    """Compiled-in schedules of the lengths over 256, whole lines and (from 2048 on) half lines, as x and
    y of 2D grids and, up to 512, as x and z of 3D grids, against the kernels of any schedule."""
    import torch
    rng = np.random.default_rng(n)
    grids = [(n, 18), (20, n)] + ([(n, 8, 10), (8, 10, n)] if n <= 512 else [])
    for g in grids:
        kernel = "coulomb3d" if len(g) == 3 else "poisson2d"
        r = torch.tensor(rng.standard_normal(g[::-1]), device="cuda")
        assert torch.equal(gsm.Plan(kernel, 4.0, g).apply(r), gsm.Plan(kernel, 4.0, g, debug=4).apply(r)), g


@pytest.mark.parametrize("nl", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [(320, 54), (54, 750), (1080, 40), (40, 2000)], ids=lambda n: "x".join(map(str, n)))
def test_lines_per_cta_of_long_lengths(gsm, n, nl):
    """The same with every number of lines per CTA, with 8 and (padded lengths over 2048) 16 values
    per thread."""
    import torch
    r = torch.tensor(np.random.default_rng(nl).standard_normal(n[::-1]), device="cuda")
    data = gsm.Plan("coulomb2d", 4.0, n).save()
    u = gsm.Plan("coulomb2d", 4.0, n, debug=4).apply(r)
    for emax in (8, 16):
        assert torch.equal(gsm.Plan.load(_resaved(data, nl=nl, emax=emax)).apply(r), u)
