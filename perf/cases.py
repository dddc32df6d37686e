"""Cases for timing the library: what its users call, over the range of sizes they call it with.

Every case is one public call (Plan.apply, Plan.apply_host, Plan.hartree, GSMApply forward and
backward, apply_batched) on densities shaped like the ones the method is used for: mixtures of a
few Gaussians, resolved by the grid and small at the edge of the box.  The grid of axis a has
n_a points of spacing h = 24 / max(n), so that the longest half-width is 12 (Sec. 4 of the paper),
x_j = -L_a + j h, j = 1..n_a, and arrays are C-ordered with x fastest.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  plan and inputs
    run(state)           one call
    work(case)           bytes and operations of one call
    exact(case, seed)    what the call returns, from the potentials of Gaussians in 64 bits
"""
import math

import numpy as np
import torch

import paper_1501_04438_gb300 as gsm

DIM = {"coulomb3d": 3, "dipolar3d": 3, "power3d": 3, "coulomb2d": 2, "poisson2d": 2, "ds2d": 2}
PRECISIONS = ("fp64", "fp32x2", "fp32")
DIP_N, DIP_M = (0.6, 0.0, 0.8), (0.0, 1.0, 0.0)
BETA = 1.7
HALF_WIDTH = 12.0
BATCH_SIZES = (48, 64, 96, 128, 160)
# the even products of 2, 3 and 5, those with a single factor 2 (54, 90, 150, 250, ...) among them
LENGTHS = sorted(2 ** a * 3 ** b * 5 ** c for a in range(1, 13) for b in range(8) for c in range(6)
                 if 24 <= 2 ** a * 3 ** b * 5 ** c <= 4096)
LARGEST_3D = 256 ** 3


def _case(name, op, kernel, n, precision, tune=False, count=0):
    n = tuple(n) + (1,) * (3 - len(n))
    c = {"op": op, "kernel": kernel, "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision, "tune": tune,
         "count": count}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest solve: one potential of a coarse 3D grid inside a time step, bound by launches
        _case("coulomb3d_32_fp64", "apply", "coulomb3d", (32, 32, 32), "fp64"),
        # the headline: one 3D solve in double, the plan tuned once by its owner
        _case("coulomb3d_256_fp64_tuned", "apply", "coulomb3d", (256, 256, 256), "fp64", tune=True),
        # the same solve for a user who needs single precision only
        _case("coulomb3d_256_fp32", "apply", "coulomb3d", (256, 256, 256), "fp32"),
        # an ordinary 3D solve in the double-float precision
        _case("coulomb3d_128_fp32x2", "apply", "coulomb3d", (128, 128, 128), "fp32x2"),
        # 3D dipolar condensate in an elongated box, general dipole axes, ragged sizes
        _case("dipolar3d_120x90x50_fp64", "apply", "dipolar3d", (120, 90, 50), "fp64"),
        # an ordinary 2D solve
        _case("poisson2d_1024_fp32x2", "apply", "poisson2d", (1024, 1024), "fp32x2"),
        # the largest 2D solve of the paper's tables' kind
        _case("poisson2d_4096_fp64", "apply", "poisson2d", (4096, 4096), "fp64"),
        # Davey-Stewartson source on a ragged 2D grid, single precision
        _case("ds2d_1500x648_fp32", "apply", "ds2d", (1500, 648), "fp32"),
        # energy and gradient of one step of a ground-state search
        _case("hartree3d_192_fp64", "hartree", "coulomb3d", (192, 192, 192), "fp64"),
        # the potential inside a model that is trained: forward and backward, ragged sizes
        _case("backward_power3d_150x90x64_fp32", "backward", "power3d", (150, 90, 64), "fp32"),
        # host arrays in and out (page-locked), a user without device arrays
        _case("host_coulomb3d_160_fp64", "host", "coulomb3d", (160, 160, 160), "fp64"),
        # many independent systems of uneven sizes in one call
        _case("batch48_coulomb3d_fp64", "batch", "coulomb3d", (160, 160, 160), "fp64", count=48),
    ]


def _length(rng, lo, hi):
    """A length of LENGTHS near one whose logarithm is uniform."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(LENGTHS, key=lambda v: abs(math.log(v / want)))


def draw(rng):
    precision = rng.choice(PRECISIONS)
    op = rng.choice(("apply", "apply", "apply", "apply", "hartree", "backward", "host", "batch"))
    if op == "batch":
        return _case(None, op, "coulomb3d", (rng.choice(BATCH_SIZES),) * 3, precision, count=rng.randint(2, 32))
    kernel = rng.choice(tuple(DIM)) if op == "apply" else rng.choice(("coulomb3d", "power3d", "coulomb2d"))
    if DIM[kernel] == 2:
        return _case(None, op, kernel, (_length(rng, 32, 4096), _length(rng, 32, 4096)), precision)
    base = _length(rng, 24, 256)   # axes within a factor of two and a half of each other
    n = [min(400, _length(rng, max(24, base / 2.5), base)) for _ in range(2)] + [base]
    rng.shuffle(n)
    return _case(None, op, kernel, n, precision)


# ------------------------------------------------------------------ inputs

def _sizes(case):
    return tuple(case["n" + a] for a in "xyz"[:DIM[case["kernel"]]])


def _instances(case):
    """Grid sizes of the call's instances: one, or `count` of a batch (sizes up to the case's)."""
    n = _sizes(case)
    if case["op"] != "batch":
        return [n]
    sizes = [s for s in BATCH_SIZES if s <= n[0]]
    rng = np.random.default_rng(20150106 + case["count"])
    return [(int(sizes[rng.integers(len(sizes))]),) * 3 for _ in range(case["count"])]


def _box(n):
    h = 2.0 * HALF_WIDTH / max(n)
    return h, tuple(0.5 * h * m for m in n)


def _axes(n, device):
    h, box = _box(n)
    return [(torch.arange(m, dtype=torch.float64, device=device) + 1.0) * h - L for m, L in zip(n, box)]


def _mixture(rng, n, count, isotropic, same_width=False):
    """`count` Gaussians a exp(-sum ((x - c) / s)^2): centres in the inner eighth of the box, widths
    1/24 to 1/8 of its shortest half-width and at least 3.2 grid spacings."""
    h, box = _box(n)
    d, L = len(n), min(box)
    out, s = [], None
    for _ in range(count):
        c = [rng.uniform(-0.125, 0.125) * b for b in box]
        if s is None or not same_width:
            s = [max(3.2 * h, rng.uniform(0.5, 1.5) * L / HALF_WIDTH) for _ in range(1 if isotropic else d)]
            s = s * d if isotropic else s
        out.append((c, s, rng.uniform(0.5, 2.0)))
    return out


def _outer(fx, *rest):
    """sum_q prod_a f_a[q, x_a] as an array with x fastest."""
    if len(rest) == 1:
        return rest[0].T @ fx
    fy, fz = rest
    q, ny, nz = fy.shape[0], fy.shape[1], fz.shape[1]
    out = torch.empty(nz, ny, fx.shape[1], dtype=fx.dtype, device=fx.device)
    for z in range(nz):
        out[z] = (fy * fz[:, z:z + 1]).T @ fx
    return out


def _sample(n, params, device="cuda"):
    axes = _axes(n, device)
    f = [torch.stack([(a if k == 0 else 1.0) * torch.exp(-((x - c[k]) / s[k]) ** 2) for c, s, a in params])
         for k, x in enumerate(axes)]
    return _outer(*f)


def _params(case, seed):
    rng = np.random.default_rng(seed)
    isotropic = DIM[case["kernel"]] == 2 or case["op"] == "hartree"
    count = {"apply": 8, "host": 8, "backward": 4, "batch": 4, "hartree": 2}[case["op"]]
    count = 1 if max(_sizes(case)) <= 32 else count
    params = [_mixture(rng, n, count, isotropic, case["op"] == "hartree") for n in _instances(case)]
    if case["op"] == "backward":   # the gradient that comes back from the rest of the model
        params.append(_mixture(rng, _sizes(case), count, isotropic))
    if case["op"] == "hartree":    # the plane wave of the wave function
        params.append([rng.uniform(-1.0, 1.0) for _ in range(DIM[case["kernel"]])])
    return params


def _psi(case, params):
    """sum_g a_g exp(-|x - c_g|^2 / (2 s^2)) exp(i k.x), one width for all g."""
    n = _sizes(case)
    mix = [(c, [math.sqrt(2.0) * v for v in s], a) for c, s, a in params[0]]
    amp = _sample(n, mix)
    phase = 0.0
    for k, x in enumerate(_axes(n, "cuda")):
        shape = [1] * len(n)
        shape[len(n) - 1 - k] = -1
        phase = phase + params[1][k] * x.reshape(shape)
    return torch.complex(amp * torch.cos(phase), amp * torch.sin(phase))


def _plan(case, n):
    p = gsm.Plan(case["kernel"], HALF_WIDTH, n, precision=case["precision"], box=_box(n)[1], dip_n=DIP_N, dip_m=DIP_M,
                 beta=BETA)
    if case["tune"]:
        p.autotune()
    return p


def prepare(case, seed):
    real = torch.float32 if case["precision"] == "fp32" else torch.float64
    params = _params(case, seed)
    sizes = _instances(case)
    plans = [_plan(case, n) for n in sizes]
    st = {"op": case["op"], "plan": plans[0]}
    if case["op"] == "batch":
        st["plans"] = plans
        st["rhos"] = [_sample(n, p).to(real) for n, p in zip(sizes, params)]
        st["outs"] = [torch.empty_like(r) for r in st["rhos"]]
    elif case["op"] == "hartree":
        st["psi"] = _psi(case, params).to(torch.complex64 if real == torch.float32 else torch.complex128)
    else:
        rho = _sample(sizes[0], params[0]).to(real)
        if case["op"] == "host":
            host = torch.empty(rho.shape, dtype=real, pin_memory=True)
            host.copy_(rho)
            st["rho"], st["out"] = host.numpy(), torch.empty(rho.shape, dtype=real, pin_memory=True).numpy()
        elif case["op"] == "backward":
            st["rho"] = rho.requires_grad_(True)
            st["weight"] = _sample(sizes[0], params[1]).to(real)
        else:
            st["rho"], st["out"] = rho, torch.empty_like(rho)
    return st


def run(state):
    op, plan = state["op"], state["plan"]
    if op == "apply":
        return plan.apply(state["rho"], out=state["out"])
    if op == "host":
        return plan.apply_host(state["rho"], out=state["out"])
    if op == "batch":
        return gsm.apply_batched(state["plans"], state["rhos"], state["outs"])
    if op == "hartree":
        energy, u, grad = plan.hartree(state["psi"])
        return {"energy": energy, "u": u, "grad": grad}
    u = gsm.GSMApply.apply(state["rho"], plan)
    (grad,) = torch.autograd.grad(u, state["rho"], state["weight"])
    return {"u": u.detach(), "grad": grad}


def work(case):
    """Inputs and outputs once, the plan's multiplier table once per pass; radix-2 operation counts
    (5 M log2 M a complex transform) of the zero-padded real transforms that the method asks for."""
    total = {"bytes": 0.0, "flops": 0.0}
    item = 4 if case["precision"] == "fp32" else 8
    fields = {"apply": 2, "host": 2, "batch": 2, "backward": 4, "hartree": 5}[case["op"]]
    passes = 2 if case["op"] == "backward" else 1
    for n in _instances(case):
        pts, table = math.prod(n), math.prod(m + 1 for m in n)
        if case["kernel"] == "dipolar3d":   # general axes: the half spectrum
            table = (n[0] + 1) * math.prod(2 * m for m in n[1:])
        fft = [5.0 * 2 * m * math.log2(2 * m) for m in n]
        flops = pts / n[0] * fft[0] + 2.0 * (n[0] + 1) * 2 * n[-1]   # x transforms, both ways, two rows at a time
        if len(n) == 2:
            flops += 2.0 * (n[0] + 1) * fft[1]
        else:
            flops += 2.0 * (n[0] + 1) * n[2] * fft[1] + 2.0 * (n[0] + 1) * 2 * n[1] * fft[2]
        total["bytes"] += item * (fields * pts + passes * table)
        total["flops"] += passes * flops
    return total


# ------------------------------------------------------------------ exact potentials

def _quadrature(beta, d, widths, device):
    """Nodes t and weights of r^-beta = (2 / Gamma(beta/2)) int t^(beta-1) exp(-r^2 t^2) dt,
    t = e^s, by the trapezoidal rule, for Gaussians of the given widths in d dimensions."""
    lo = -42.0 / beta - math.log(max(widths))
    hi = 42.0 / (d - beta) - math.log(min(widths))
    step = 0.1
    t = torch.exp(torch.arange(lo, hi, step, dtype=torch.float64, device=device))
    return t, (2.0 / math.gamma(beta / 2.0)) * step * t ** beta


def _power_potential(n, params, beta, device, hessian=None):
    """|x|^-beta convolved with the mixture, on the grid; with hessian = (a, b), the second
    derivative along the axes a and b of it."""
    axes, d = _axes(n, device), len(n)
    fs = [[] for _ in range(d)]
    for c, s, a in params:
        t, w = _quadrature(beta, d, s, device)
        for k, x in enumerate(axes):
            b = (t * t / (1.0 + (t * s[k]) ** 2))[:, None]
            y = x[None, :] - c[k]
            f = (math.sqrt(math.pi) * s[k]) / torch.sqrt(1.0 + (t * s[k]) ** 2)[:, None] * torch.exp(-b * y * y)
            if hessian is not None and k in hessian:
                f = f * ((4.0 * b * b * y * y - 2.0 * b) if hessian[0] == hessian[1] else -2.0 * b * y)
            fs[k].append(f * (a * w[:, None] if k == 0 else 1.0))
    return _outer(*[torch.cat(f) for f in fs])


def _exp1(x):
    """E_1(x), x > 0: its power series below 2, its continued fraction above."""
    small = torch.clamp(x, max=2.0)
    term, total = torch.ones_like(x), torch.zeros_like(x)
    for k in range(1, 40):
        term = term * (-small / k)
        total = total - term / k
    series = total - torch.log(small) - 0.57721566490153286061
    big = torch.clamp(x, min=2.0)
    frac = torch.zeros_like(x)
    for k in range(90, 0, -1):
        frac = k / (1.0 + k / (big + frac))
    return torch.where(x < 2.0, series, torch.exp(-big) / (big + frac))


def _potential(case, n, params, device="cuda"):
    kernel = case["kernel"]
    if kernel == "coulomb3d":
        return _power_potential(n, params, 1.0, device) / (4.0 * math.pi)
    if kernel == "power3d":
        return _power_potential(n, params, BETA, device)
    if kernel == "dipolar3d":
        u = -sum(p * q for p, q in zip(DIP_N, DIP_M)) * _sample(n, params, device)
        for i in range(3):
            for j in range(3):
                if DIP_N[i] * DIP_M[j] != 0.0:
                    u = u - 3.0 * DIP_N[i] * DIP_M[j] * _power_potential(n, params, 1.0, device, (i, j)) / (4.0 * math.pi)
        return u
    x, y = _axes(n, device)
    u = torch.zeros(n[1], n[0], dtype=torch.float64, device=device)
    for c, s, a in params:   # isotropic
        s2, dx = s[0] ** 2, (x - c[0])[None, :]
        q = torch.clamp(dx ** 2 + ((y - c[1]) ** 2)[:, None], min=1e-30)
        if kernel == "coulomb2d":
            u += a * math.sqrt(math.pi) * s[0] / 2.0 * torch.special.i0e(q / (2.0 * s2))
        elif kernel == "poisson2d":
            u -= a * s2 / 4.0 * (_exp1(q / s2) + torch.log(q))
        else:                # second x derivative of the 2D Poisson potential
            g = -torch.expm1(-q / s2) / q
            u -= a * s2 / 2.0 * (g + 2.0 * dx * dx * (torch.exp(-q / s2) / s2 - g) / q)
    return u


def exact(case, seed):
    params, sizes = _params(case, seed), _instances(case)
    if case["op"] == "batch":
        return [_potential(case, n, p) for n, p in zip(sizes, params)]
    if case["op"] == "backward":
        return {"u": _potential(case, sizes[0], params[0]), "grad": _potential(case, sizes[0], params[1])}
    if case["op"] == "hartree":
        # |psi|^2: Gaussians of width s at the midpoints of each pair of centres
        mix = [([(p + q) / 2 for p, q in zip(c1, c2)], s,
                a1 * a2 * math.exp(-sum((p - q) ** 2 for p, q in zip(c1, c2)) / (4.0 * s[0] ** 2)))
               for c1, s, a1 in params[0] for c2, _, a2 in params[0]]
        psi, u = _psi(case, params), _potential(case, sizes[0], mix)
        cell = _box(sizes[0])[0] ** len(sizes[0])
        return {"energy": 0.5 * cell * (torch.abs(psi) ** 2 * u).sum(), "u": u, "grad": 2.0 * cell * u * psi}
    return _potential(case, sizes[0], params[0])
