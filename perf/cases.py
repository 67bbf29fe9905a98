"""The work a program built on this library has it do, as cases to be timed.

A case is one call of a public entry point (or a forward and backward pair)
on seeded synthetic fields of the library's workloads: elongated two-cloud
interferometers, quasicondensates with thermal axial phases and solitons, and
the noise that every realization of an ensemble carries.  Lattices are written
"64x64x64" (row-major, the last axis contiguous), magnifications "30x30x3".

``kind`` says which call a case makes:

* ``density``   ``ffx_expand``: one density per realization, or with ``sum``
                the ensemble sum of an accumulating plan;
* ``field``     ``ffx_expand_field``: the complex field;
* ``column``    ``ffx_expand_column``: the detector image along ``axis``;
* ``gradient``  ``expand_density`` and its backward: the densities and the
                gradient of a loss with respect to the initial field;
* ``mixed``     ``ffx_expand`` on a plan over many instances of different
                lattices, magnifications and flight times.
"""

from __future__ import annotations

import math
import random

import torch

from paper_1602_03395_gb300 import ffx

MIXED_SHAPES = ((48, 48, 48), (64, 64, 64), (96, 96, 96), (128, 32, 32))


def _case(name, kind, dims, dx, lam, t, batch, **more):
    return {"name": name, "kind": kind, "dims": dims, "dx": dx, "lam": lam, "t": t, "batch": batch,
            "cloud": "two", "sum": False, "axis": 0, "form": "auto", **more}


def listed():
    return [
        # one shot of a 1-D trapped gas with solitons, expanded interactively
        # or inside a fitting loop: a few microseconds of work, so the call's
        # own latency is what the user waits for
        _case("line-512", "density", "512", 0.1, "20", 40.0, 1, cloud="quasi"),
        # an ensemble of long 1-D gases, mean density: the longest line length
        # (only the FFT forms take it)
        _case("lines-2048-mean", "density", "2048", 0.1, "20", 40.0, 512, cloud="quasi", sum=True),
        # one interferometer shot, 3-D: latency of a whole expansion
        _case("two-cloud-64-single", "density", "64x64x64", 0.25, "30x30x3", 40.0, 1),
        # the same interferometer, a batch of shots
        _case("two-cloud-64-batch", "density", "64x64x64", 0.25, "30x30x3", 40.0, 64),
        # fitting an initial state to measured densities on a lattice whose
        # axes all differ, an odd number of shots: forward and gradient
        _case("ragged-gradient", "gradient", "48x96x192", 0.25, "7x11x4", 12.0, 5),
        # a stochastic ensemble of elongated quasicondensates: mean density
        _case("quasicondensate-mean", "density", "32x32x512", 0.25, "50x50x5", 40.0, 256, cloud="quasi", sum=True),
        # a long flight of a large lattice at large magnification
        _case("large-256", "density", "256x256x256", 0.25, "100x100x100", 400.0, 1),
        # the same, fitted: forward and gradient
        _case("large-256-gradient", "gradient", "256x256x256", 0.25, "100x100x100", 400.0, 1),
        # a large elongated quasicondensate: the longest 3-D axis
        _case("large-elongated", "density", "128x128x1024", 0.25, "100x100x100", 400.0, 1, cloud="quasi"),
        # detector images of a few shots, integrated along the imaging axis
        _case("detector-image", "column", "128x128x128", 0.25, "40x40x40", 160.0, 4, axis=2),
        # short flights: the field after a barely magnifying expansion
        _case("short-flight-field", "field", "256x64x256", 0.25, "1x2x1", 2.0, 3),
        # a campaign of different traps, magnifications and flight times in one
        # plan (shapes and magnifications drawn from the case's own seed)
        _case("mixed-campaign", "mixed", "", 0.25, "", 0.0, 200, instances=4),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng: random.Random):
    """One more case: the listed families with other lattices (every supported
    length, axes that differ), magnifications, flight times and odd batches."""
    kind = rng.choice(["density", "density", "density", "gradient", "gradient", "field", "column", "mixed"])
    if kind == "mixed":
        c = _case("", "mixed", "", 0.25, "", 0.0, int(_log_uniform(rng, 3, 250)), instances=rng.randrange(10 ** 6))
        del c["name"]
        return c
    ndim = rng.choice([1, 2, 3, 3, 3, 3])
    lengths = {1: (64, 128, 256, 384, 512, 768, 1024, 2048),
               2: (16, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024),
               3: (16, 32, 48, 64, 96, 128, 192, 256)}[ndim]
    dims = [rng.choice(lengths) for _ in range(ndim)]
    if ndim == 3 and rng.random() < 0.3:  # elongated along the last axis
        dims = [rng.choice((32, 64, 128)), rng.choice((32, 64, 128)), rng.choice((384, 512, 768, 1024))]
    if ndim == 3 and rng.random() < 0.2:  # cubes
        dims = [rng.choice((48, 64, 96, 128, 256))] * 3
    m = math.prod(dims)
    if rng.random() < 0.15:
        lam = [rng.choice((1, 2)) for _ in dims]
        t = rng.uniform(0.5, 4.0)
    else:
        lam = [int(_log_uniform(rng, 3, 100)) for _ in dims]
        if ndim == 1 and dims[0] == 2048:
            lam = [min(lam[0], 24)]
        t = 4.0 * max(lam) * rng.uniform(0.3, 1.0)
    c = _case("", kind, "x".join(map(str, dims)), rng.choice([0.1, 0.25, 0.5]), "x".join(map(str, lam)),
              round(t, 3), 1, cloud=rng.choice(["two", "quasi"]), axis=rng.randrange(ndim))
    # no drawn case costs more than the largest listed ones: at most 2^25
    # points and 2e11 operations a call
    one = work(c)
    if kind == "gradient" and one["flops"] > 2e11:
        c["kind"], one = "density", work({**c, "kind": "density"})
    cap = min(4096, 2 ** 25 // math.prod(dims), int(2e11 // one["flops"]))
    c["batch"] = max(1, int(_log_uniform(rng, 1, max(1, cap) + 0.99)))
    c["sum"] = c["kind"] in ("density", "column") and ndim > 1 and c["batch"] > 1 and rng.random() < 0.4
    del c["name"]
    return c


def _ints(text):
    return tuple(int(v) for v in text.split("x"))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)


def _fields(dims, dx, batch, cloud, gen):
    """`batch` realizations as complex64 [batch, *dims]: an envelope common to
    all, each one's random phases, and 2% complex noise."""
    d = len(dims)
    axes = [(torch.arange(n, device="cuda", dtype=torch.float32) - 0.5 * n) * dx for n in dims]
    half = [0.5 * n * dx for n in dims]

    def shaped(v, j):
        return v.view([1] * j + [-1] + [1] * (d - 1 - j))

    def unif(*shape):
        return torch.rand(shape, generator=gen, device="cuda")

    if cloud == "two":
        # two clouds along the first axis, random relative phase per realization
        env = torch.ones((1,) * d, device="cuda")
        for j in range(1, d):
            env = env * torch.exp(-0.5 * shaped((axes[j] / (0.5 * half[j])) ** 2, j))
        c, s = 0.375 * 2 * half[0], 0.25 * half[0]
        g1 = env * torch.exp(-0.5 * shaped(((axes[0] - c) / s) ** 2, 0))
        g2 = env * torch.exp(-0.5 * shaped(((axes[0] + c) / s) ** 2, 0))
        phi = 2 * math.pi * unif(batch, *([1] * d))
        psi = g1 + torch.polar(torch.ones_like(phi), phi) * g2
    else:
        # Thomas-Fermi envelope, thermal phase and up to three solitons along
        # the last axis
        r = sum(shaped((axes[j] / (0.75 * half[j])) ** 2, j) for j in range(d))
        env = torch.sqrt(torch.clamp(1.0 - r, min=0.0))
        z = axes[-1] / half[-1]  # -1 .. 1
        k = math.pi * torch.arange(1, 65, device="cuda", dtype=torch.float32)
        ab = torch.randn((2, batch, 64), generator=gen, device="cuda") * (2.0 / k)
        theta = ab[0] @ torch.cos(k[:, None] * z) + ab[1] @ torch.sin(k[:, None] * z)
        axial = torch.ones_like(theta)
        for zk in (unif(batch, 3) - 0.5).unbind(1):
            axial = axial * torch.tanh((z[None, :] - zk[:, None]) * (half[-1] / (5 * dx)))
        psi = torch.polar(axial.abs(), theta + math.pi * (axial < 0))
        psi = env * psi.view(batch, *([1] * (d - 1)), -1)
    psi = psi.to(torch.complex64).contiguous()
    noise = torch.view_as_real(psi)
    noise += 0.02 * torch.randn(noise.shape, generator=gen, device="cuda")
    return psi


def _instances(case):
    """(dims, spacing, t, lam) of each instance of a mixed case."""
    rng = random.Random(case["instances"])
    out = []
    for _ in range(case["batch"]):
        lam = rng.randint(10, 100)
        out.append((rng.choice(MIXED_SHAPES), (case["dx"],) * 3, 4.0 * lam, (lam,) * 3))
    return out


def _inputs(case, seed):
    gen = _gen(seed)
    if case["kind"] == "mixed":
        return torch.cat([_fields(dims, spacing[0], 1, "two", gen).reshape(-1)
                          for dims, spacing, _, _ in _instances(case)]), None
    psi = _fields(_ints(case["dims"]), case["dx"], case["batch"], case["cloud"], gen)
    grad = None
    if case["kind"] == "gradient":
        grad = torch.randn(psi.shape, generator=gen, device="cuda")
    return psi, grad


def prepare(case, seed):
    psi, grad = _inputs(case, seed)
    if case["kind"] == "mixed":
        plan = ffx.PlanMany(_instances(case))
    else:
        dims, lam = _ints(case["dims"]), _ints(case["lam"])
        plan = ffx.Plan(dims, (case["dx"],) * len(dims), case["t"], lam, form=case["form"], accumulate=case["sum"])
    if case["kind"] == "gradient":
        psi.requires_grad_(True)
    return {"case": case, "plan": plan, "psi": psi, "grad": grad}


def run(state):
    case, plan, psi = state["case"], state["plan"], state["psi"]
    if case["kind"] == "gradient":
        rho = ffx.expand_density(psi, plan)
        (g,) = torch.autograd.grad(rho, psi, state["grad"])
        return rho.detach(), g
    if case["kind"] == "field":
        return ffx.ffx_expand_field(plan, psi)
    if case["kind"] == "column":
        return ffx.ffx_expand_column(plan, psi, case["axis"])
    return ffx.ffx_expand(plan, psi)


def _points(case):
    if case["kind"] == "mixed":
        return [(dims, lam, 1) for dims, _, _, lam in _instances(case)]
    return [(_ints(case["dims"]), _ints(case["lam"]), case["batch"])]


def _flops_per_point(n, lam):
    # the per-axis map as one n x n complex product, or as lam + 1 line FFTs
    # with their phase products, whichever is less
    lg = math.log2(n)
    return min(8.0 * n, lam * (5.0 * lg + 14.0) + 5.0 * lg)


def work(case):
    """Input read once, output written once (gradients: the density gradient
    read and the field gradient written too); the map's arithmetic."""
    nbytes = flops = 0
    for dims, lam, batch in _points(case):
        m = math.prod(dims)
        outs = m if case["sum"] else m * batch
        if case["kind"] == "column":
            outs //= dims[case["axis"]]
        nbytes += 8 * m * batch + (8 if case["kind"] == "field" else 4) * outs
        if case["kind"] == "gradient":
            nbytes += 12 * m * batch
        passes = 2 if case["kind"] == "gradient" else 1
        flops += passes * m * batch * sum(_flops_per_point(n, l) for n, l in zip(dims, lam))
    return {"bytes": nbytes, "flops": int(flops)}


def _axis_map(n, lam, dx, t):
    """T[nbar, n] of one axis in complex128: free flight of the vacuum-padded
    line on the periodic lattice of lam n points, sampled every lam points."""
    m = lam * n
    u = torch.arange(m, device="cuda", dtype=torch.float64)
    u = torch.where(2 * u < m, u, u - m)
    k = 2.0 * math.pi * u / (m * dx)
    kernel = torch.fft.ifft(torch.polar(torch.ones_like(k), -0.5 * t * k * k))
    s0 = -(((lam - 1) * n) // 2)
    i = torch.arange(n, device="cuda")
    return kernel[(s0 + lam * i[:, None] - i[None, :]) % m]


def _apply(maps, x):
    for j, mat in enumerate(maps):
        x = torch.movedim(torch.tensordot(mat, x, dims=([1], [j])), 0, j)
    return x


def exact(case, seed):
    psi, grad = _inputs(case, seed)
    if case["kind"] == "mixed":
        out, off = torch.empty(psi.numel(), dtype=torch.float64, device="cuda"), 0
        for dims, spacing, t, lam in _instances(case):
            m = math.prod(dims)
            maps = [_axis_map(n, l, h, t) for n, l, h in zip(dims, lam, spacing)]
            f = _apply(maps, psi[off:off + m].view(dims).to(torch.complex128))
            out[off:off + m] = (f.real ** 2 + f.imag ** 2).reshape(-1)
            off += m
        return out
    dims, lam = _ints(case["dims"]), _ints(case["lam"])
    maps = [_axis_map(n, l, case["dx"], case["t"]) for n, l in zip(dims, lam)]
    rhos, fields, grads, total = [], [], [], 0.0
    for b in range(psi.shape[0]):
        f = _apply(maps, psi[b].to(torch.complex128))
        if case["kind"] == "field":
            fields.append(f)
            continue
        rho = f.real ** 2 + f.imag ** 2
        if case["kind"] == "gradient":
            grads.append(_apply([mat.conj().T for mat in maps], 2.0 * grad[b].to(torch.float64) * f))
        if case["kind"] == "column":
            rho = rho.sum(dim=case["axis"]) * (lam[case["axis"]] * case["dx"])
        if case["sum"]:
            total = total + rho
        else:
            rhos.append(rho)
    if case["kind"] == "field":
        return torch.stack(fields)
    if case["sum"]:
        return total
    if case["kind"] == "gradient":
        return torch.stack(rhos), torch.stack(grads)
    return torch.stack(rhos)
