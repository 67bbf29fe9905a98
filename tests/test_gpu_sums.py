"""Ensemble sums (accumulating plans) over batches that run in several groups of
realizations, whose partial densities are added at the end: every kernel that
sums (FFT forms, FP32 dense, tensor cores, BF16 planes), group counts that do
and do not divide the batch, against the FP64 oracle added to what the output
held.  The sum adds at most a few hundred terms in FP32, far below the density
bar (DENSITY_TOL) of the terms themselves; its order is fixed, so a repeated
call gives the same bits."""

import numpy as np
import pytest
import torch

import oracle as O
from gpu_common import DENSITY_TOL, random_field, rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu

CASES = [
    # (dims, lam, batch, form)
    ((2048,), (3,), 37, "auto"),           # FFT forms, one line a realization
    ((256,), (1,), 33, "fold"),
    ((64, 16), (2, 3), 9, "paper"),
    ((512,), (20,), 100, "auto"),          # FP32 dense
    ((48, 16), (7, 5), 50, "dense"),
    ((32, 32, 64), (5, 6, 7), 2, "tc"),    # 32-point tensor-core sums: groups of one
    ((32, 32, 64), (5, 6, 7), 45, "tc"),   # ... and uneven groups
    ((32, 48), (5, 6), 300, "tc"),         # 48 lines: a partly empty tile
    ((48, 96), (5, 6), 29, "tc"),          # streaming tensor-core kernel
    ((256, 96), (5, 9), 31, "tc"),         # BF16 chain, planes on CTA pairs
    ((64, 64, 128), (5, 9, 4), 6, "tc"),
    ((256,), (9,), 1000, "tc"),            # planes, contiguous lines
]


@pytest.mark.parametrize("dims,lam,batch,form", CASES)
def test_ensemble_sum_groups(dims, lam, batch, form):
    ffx = require_gpu()
    rng = np.random.default_rng(batch + sum(dims))
    dx, t = (0.25,) * len(dims), 5.0
    psi = random_field(rng, (batch,) + dims)
    start = rng.random(dims).astype(np.float32)
    ref = start + (np.abs(O.expand_field(psi, dx, t, lam)) ** 2).sum(0)
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form=form, accumulate=True) as plan:
        got = ffx.ffx_expand(plan, x, to_dev(start.copy()))
        again = ffx.ffx_expand(plan, x, to_dev(start.copy()))
        assert plan.device_errors() == 0
    assert torch.equal(got, again)
    assert rel_l2(got.cpu().numpy(), ref) < DENSITY_TOL
