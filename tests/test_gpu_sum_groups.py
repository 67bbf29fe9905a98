"""Ensemble sums whose last pass runs over planes or strided FP32 lines on the
BF16 kernels, in several groups of realizations: the groups are counted in that
kernel's own waves (152 SMs), so that these batches divide into groups without a
remainder launch, and the sums hold the FP64 oracle's bar."""

import numpy as np
import pytest
import torch

import oracle as O
from gpu_common import DENSITY_TOL, random_field, rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,lam,batch,chain", [
    ((96, 64), (5, 9), 331, False),    # 331 groups; by the streaming kernel's waves 114 and a remainder
    ((192, 64), (4, 7), 203, False),
    ((384, 64), (9, 5), 61, False),    # CTA pairs
    ((128, 64), (5, 4), 512, False),   # two realizations a group
    ((96, 64), (5, 9), 1000, True),    # the same from planes
])
def test_groups_of_plane_sums(dims, lam, batch, chain):
    ffx = require_gpu()
    rng = np.random.default_rng(batch)
    dx, t = (0.25,) * len(dims), 5.0
    psi = random_field(rng, (batch,) + dims)
    start = rng.random(dims).astype(np.float32)
    ref = start + (np.abs(O.expand_field(psi, dx, t, lam)) ** 2).sum(0)
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, accumulate=True) as plan:
        assert plan.bf16_chain(batch) == chain
        n0 = plan.launch_count()
        got = ffx.ffx_expand(plan, x, to_dev(start.copy()))
        launches = plan.launch_count() - n0
        again = ffx.ffx_expand(plan, x, to_dev(start.copy()))
        assert plan.device_errors() == 0
    assert launches == len(dims) + 1  # the passes and the sum of the groups
    assert torch.equal(got, again)
    assert rel_l2(got.cpu().numpy(), ref) < DENSITY_TOL
