"""FFT-form passes on contiguous lines of 512, 1024 and 2048 points
(csrc/ffx_line3.cu) against the FP64 oracle: paper and fold forms and the
adjoint, magnifications whose gcd with the length is 1, 2, 4, 8, 16 (the fold
sums that many registers) and 32 (the general engine), odd and even, line counts
that leave part of a block idle, contiguous last axes beside strided ones, and
the densities, field, ensemble sum and gradient each writes.

FP32 transforms: a few 1e-7 of relative error; the tests hold the FP32 path's
own bars."""

import numpy as np
import pytest

import oracle as O
from gpu_common import DENSITY_TOL, FIELD_TOL, random_field, rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu

CASES = [
    ((512,), (3,), 9), ((512,), (2,), 17), ((512,), (48,), 1),
    ((1024,), (5,), 3), ((1024,), (20,), 6), ((1024,), (8,), 1),
    ((2048,), (7,), 5), ((2048,), (20,), 2), ((2048,), (1,), 3), ((2048,), (16,), 2), ((2048,), (32,), 2),
    ((16, 512), (3, 6), 2), ((3 * 16, 1024), (2, 3), 1),
]


@pytest.mark.parametrize("form", ["fold", "paper"])
@pytest.mark.parametrize("dims,lam,batch", CASES)
def test_line3(dims, lam, batch, form):
    ffx = require_gpu()
    rng = np.random.default_rng(batch + sum(dims) + lam[-1])
    dx, t = (0.2,) * len(dims), 4.0
    psi = random_field(rng, (batch,) + dims)
    grad = rng.normal(size=(batch,) + dims).astype(np.float32)
    ref = O.expand_field(psi, dx, t, lam)
    dens = np.abs(ref) ** 2
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form=form) as plan:
        rho = ffx.ffx_expand(plan, x).cpu().numpy()
        fld = ffx.ffx_expand_field(plan, x).cpu().numpy()
        g = ffx.ffx_expand_backward(plan, x, to_dev(grad)).cpu().numpy()
    with ffx.Plan(dims, dx, t, lam, form=form, accumulate=True) as plan:
        acc = ffx.ffx_expand(plan, x).cpu().numpy()
    assert rel_l2(rho, dens) < DENSITY_TOL
    assert rel_l2(fld, ref) < FIELD_TOL
    assert rel_l2(acc, dens.sum(0)) < DENSITY_TOL
    assert rel_l2(g, O.density_loss_gradient(psi, grad, dx, t, lam)) < FIELD_TOL
    print(f"{dims} lam={lam} {form}: field {rel_l2(fld, ref):.2e}")
