"""The passes over BF16 planes (csrc/ffx_planes.cu) against the FP64 oracle, at
the sizes where their tiling can go wrong: every row-block variant (64, 96, 128
outputs with T resident, 192 and 256 ... 1024 streamed, the latter on CTA
pairs), line counts that are not whole tiles or leave half a pair without
lines, chains (transposed planes between the passes) and single passes over
contiguous lines, and every kind of output: planes, fields, densities, the
ensemble sum, and the adjoint.

Split operands: each operand is hi + lo to 2^-17 relative and the lo*lo term is
dropped, a few 2^-18 per pass of random sign, within the FP32 path's 2e-5 bar
(DENSITY_TOL, FIELD_TOL; the gradient runs twice the passes, within the same
bar).  Unsplit: 2^-9 per operand, the 1e-2 class."""

import numpy as np
import pytest

import oracle as O
from gpu_common import DENSITY_TOL, FIELD_TOL, random_field, rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu

UNSPLIT_TOL = 1e-2

CASES = [
    # chains: lines per pass (axis 1, axis 0)
    ((256, 96), (5, 9), 1),       # 256 lines of 96; 96 lines of 256 (one tile, half a pair empty)
    ((256, 96), (5, 9), 3),       # 288 lines of 256: three tiles, the last pair's second past the end
    ((384, 128), (3, 30), 2),     # three row blocks; T resident at 128
    ((512, 192), (4, 7), 1),      # four row blocks; 192 in two blocks of 96
    ((1024, 32 * 3), (6, 5), 1),  # eight row blocks
    ((64, 64, 256), (4, 5, 6), 3),
    ((512, 64), (4, 5), 40),      # 64-output items on single CTAs (too few for pairs) and on pairs
    # single passes over contiguous lines (a 1-D field has no chain)
    ((256,), (100,), 5), ((256,), (3,), 129), ((768,), (7,), 257), ((128,), (9,), 131), ((192,), (4,), 3),
    ((96,), (11,), 400),
]


@pytest.fixture(scope="module")
def ffx():
    return require_gpu()


@pytest.mark.parametrize("dims,lam,batch", CASES)
def test_plane_passes(ffx, dims, lam, batch):
    rng = np.random.default_rng(7 * batch + sum(dims))
    dx, t = (0.25,) * len(dims), 6.0
    psi = random_field(rng, (batch,) + dims)
    grad = rng.normal(size=(batch,) + dims).astype(np.float32)
    ref = O.expand_field(psi, dx, t, lam)
    dens = np.abs(ref) ** 2
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True) as plan:
        rho = ffx.ffx_expand(plan, x).cpu().numpy()
        fld = ffx.ffx_expand_field(plan, x).cpu().numpy()
        g = ffx.ffx_expand_backward(plan, x, to_dev(grad)).cpu().numpy()
        assert plan.device_errors() == 0
    start = rng.random(dims).astype(np.float32)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, accumulate=True) as plan:
        acc = ffx.ffx_expand(plan, x, to_dev(start.copy())).cpu().numpy()
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, unsplit=True) as plan:
        rough = ffx.ffx_expand(plan, x).cpu().numpy()
        assert plan.device_errors() == 0
    assert rel_l2(rho, dens) < DENSITY_TOL
    assert rel_l2(fld, ref) < FIELD_TOL
    assert rel_l2(acc, start + dens.sum(0)) < DENSITY_TOL
    assert rel_l2(g, O.density_loss_gradient(psi, grad, dx, t, lam)) < FIELD_TOL
    assert rel_l2(rough, dens) < UNSPLIT_TOL


# passes that fill the chip read their FP32 lines themselves (chains of 192-point
# lines excepted): whole and ragged last tiles, chains and single passes, several
# row blocks
FP32_CASES = [
    ((96, 64, 256), (4, 5, 6), 4),     # chain: 24576 lines of 256
    ((64, 1024), (5, 6), 160),         # chain: 10240 lines of 1024, eight row blocks
    ((512,), (7,), 4900),              # single pass: a last tile of 36 lines
    ((384,), (5,), 13001),             # ... and half a pair without lines
    ((32, 32, 256), (3, 4, 5), 10),    # per-axis passes behind it
    ((64, 64, 64), (5, 3, 7), 6),      # T resident: chains and single passes
    ((64, 128), (5, 9), 310),
    ((96,), (5,), 19537),
    ((128,), (7,), 20001),
    ((192,), (7,), 9801),              # T streamed: a last tile of 73 lines
    ((48, 48, 192), (3, 4, 5), 5),
]


# chains whose last two axes (64 points each) are one launch: every first axis
# it serves, no first axis (an odd number of squares), items that do and do not
# divide by the blocks, ensemble sums in groups with a remainder
SQUARE_CASES = [
    ((64, 64, 64), (5, 3, 7), 20),
    ((64, 64, 64), (9, 50, 4), 41),
    ((96, 64, 64), (4, 5, 6), 13),
    ((128, 64, 64), (6, 4, 3), 10),
    ((64, 64), (5, 8), 1217),
]


@pytest.mark.parametrize("dims,lam,batch", SQUARE_CASES)
def test_square_of_64_points(ffx, dims, lam, batch):
    rng = np.random.default_rng(batch + sum(dims))
    dx, t = (0.25, 0.3, 0.2)[:len(dims)], 6.0
    psi = random_field(rng, (batch,) + dims)
    ref = O.expand_field(psi, dx, t, lam)
    dens = np.abs(ref) ** 2
    start = rng.random(size=dims).astype(np.float32)
    grad = rng.normal(size=(batch,) + dims).astype(np.float32)
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True) as plan:
        assert plan.chain_square(batch) and not plan.chain_split(batch)
        n0 = plan.launch_count()
        rho = ffx.ffx_expand(plan, x).cpu().numpy()
        assert plan.launch_count() - n0 == len(dims) - 1 == plan.launches_per_call(batch=batch)
        fld = ffx.ffx_expand_field(plan, x).cpu().numpy()
        y = x.clone()
        ffx.ffx_expand_field(plan, y, y)  # in place
        assert np.array_equal(y.cpu().numpy(), fld)
        n0 = plan.launch_count()
        g = ffx.ffx_expand_backward(plan, x, to_dev(grad)).cpu().numpy()
        if len(dims) == 3:
            assert plan.launch_count() - n0 == plan.launches_per_call(backward=True, batch=batch)
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, accumulate=True) as plan:
        assert plan.chain_square(batch) == (len(dims) == 3)
        acc = ffx.ffx_expand(plan, x, to_dev(start.copy())).cpu().numpy()
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, unsplit=True) as plan:
        rough = ffx.ffx_expand(plan, x).cpu().numpy()
        assert plan.device_errors() == 0
    assert rel_l2(rho, dens) < DENSITY_TOL
    assert rel_l2(fld, ref) < FIELD_TOL
    assert rel_l2(rho, np.abs(fld) ** 2) < 1e-6
    assert rel_l2(acc, start + dens.sum(0)) < DENSITY_TOL
    assert rel_l2(g, O.density_loss_gradient(psi, grad, dx, t, lam)) < FIELD_TOL
    assert rel_l2(rough, dens) < UNSPLIT_TOL


@pytest.mark.parametrize("dims,lam,batch", FP32_CASES)
def test_pass_of_fp32_lines(ffx, dims, lam, batch):
    rng = np.random.default_rng(batch + sum(dims))
    dx, t = (0.25,) * len(dims), 6.0
    psi = random_field(rng, (batch,) + dims)
    ref = O.expand_field(psi, dx, t, lam)
    dens = np.abs(ref) ** 2
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True) as plan:
        n0 = plan.launch_count()
        rho = ffx.ffx_expand(plan, x).cpu().numpy()
        assert plan.launch_count() - n0 == len(dims) - plan.chain_square(batch)  # no split launch
        fld = ffx.ffx_expand_field(plan, x).cpu().numpy()
        y = x.clone()
        ffx.ffx_expand_field(plan, y, y)              # in place
        assert np.array_equal(y.cpu().numpy(), fld)
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, accumulate=True) as plan:
        acc = ffx.ffx_expand(plan, x).cpu().numpy()
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, unsplit=True) as plan:
        rough = ffx.ffx_expand(plan, x).cpu().numpy()
    assert rel_l2(rho, dens) < DENSITY_TOL
    assert rel_l2(fld, ref) < FIELD_TOL
    assert rel_l2(acc, dens.sum(0)) < DENSITY_TOL
    assert rel_l2(rough, dens) < UNSPLIT_TOL


def test_first_cuda_call_of_a_thread(ffx):
    """A call that starts with a tile map, from a thread that made no CUDA call
    yet (as an autograd worker may): the same result as from this thread."""
    import threading

    import torch

    dims, lam, batch = (96, 64, 256), (4, 5, 6), 4
    x = to_dev(random_field(np.random.default_rng(3), (batch,) + dims))
    stream = torch.cuda.current_stream()
    with ffx.Plan(dims, (0.25,) * 3, 6.0, lam) as plan:
        want = ffx.ffx_expand(plan, x)
        out = torch.zeros_like(want)
        torch.cuda.synchronize()
        failures = []

        def work():
            try:
                ffx.ffx_expand(plan, x, out, stream)
            except Exception as e:  # reported by the assert below
                failures.append(e)

        thread = threading.Thread(target=work)
        thread.start()
        thread.join()
        torch.cuda.synchronize()
    assert not failures
    assert torch.equal(out, want)


# backward calls whose last forward pass writes the gradient factors: every
# kernel that does (T resident of 64, 96 and 128 points, CTA pairs, after a square
# pass), whole and ragged last tiles; and calls with a launch of their own for them
GRAD_CASES = [
    ((64, 64, 64), (5, 3, 7), 20, True),
    ((96, 64, 64), (4, 5, 6), 13, True),
    ((128, 128, 96), (4, 5, 6), 3, True),
    ((64, 128, 96), (5, 3, 4), 7, True),
    ((96, 96, 128), (3, 4, 5), 5, True),
    ((256, 96, 128), (3, 4, 5), 3, True),
    ((192, 96, 128), (3, 4, 5), 3, False),
    ((96, 96, 96), (3, 4, 5), 1, False),
]


@pytest.mark.parametrize("dims,lam,batch,fused", GRAD_CASES)
def test_gradient_factors_of_the_last_forward_pass(ffx, dims, lam, batch, fused):
    rng = np.random.default_rng(batch + sum(dims))
    dx, t = (0.25, 0.3, 0.2), 6.0
    psi = random_field(rng, (batch,) + dims)
    grad = rng.normal(size=(batch,) + dims).astype(np.float32)
    gsum = rng.normal(size=dims).astype(np.float32)
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True) as plan:
        assert plan.chain_grad(batch) == fused
        n0 = plan.launch_count()
        g = ffx.ffx_expand_backward(plan, x, to_dev(grad)).cpu().numpy()
        assert plan.launch_count() - n0 == plan.launches_per_call(backward=True, batch=batch)
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, accumulate=True) as plan:
        gs = ffx.ffx_expand_backward(plan, x, to_dev(gsum)).cpu().numpy()
        assert plan.device_errors() == 0
    assert rel_l2(g, O.density_loss_gradient(psi, grad, dx, t, lam)) < FIELD_TOL
    ref = O.density_loss_gradient(psi, np.broadcast_to(gsum, psi.shape), dx, t, lam)
    assert rel_l2(gs, ref) < FIELD_TOL


# strided FP32 lines of 64, 96, 128 points and (on CTA pairs) 256, 384, ...
# outside a chain: a group of 64
# lines too few for the last tile, one group per outer block, several, first and
# middle axes, ensemble sums (one group of realizations and many)
STRIDED_CASES = [
    ((64, 48, 64), (5, 3, 7), 27),
    ((32, 64, 64), (3, 5, 4), 39),
    ((96, 64), (9, 5), 3),
    ((96, 32, 64), (4, 5, 6), 2),
    ((32, 96, 64), (6, 4, 3), 3),
    ((128, 32, 32), (11, 4, 3), 5),
    ((32, 128, 192), (3, 30, 4), 2),
    ((256, 32, 64), (4, 5, 6), 3),
    ((32, 256, 64), (3, 7, 5), 5),
    ((384, 64), (9, 5), 61),
    ((32, 512, 32), (3, 20, 5), 2),
    ((32, 96, 48), (3, 5, 4), 3),      # groups of 16 lines: tiles over several outer blocks
    ((32, 128, 16), (3, 5, 4), 1),
    ((16, 64, 48), (3, 5, 4), 103),
    ((48, 256, 16), (3, 5, 4), 7),
    ((192, 32, 48), (3, 5, 4), 2),     # T streamed: 192, and few lines of long ones
    ((32, 192, 16), (3, 5, 4), 3),
    ((256, 48), (9, 5), 3),
    ((1024, 32), (9, 5), 2),
]


@pytest.mark.parametrize("dims,lam,batch", STRIDED_CASES)
def test_strided_lines(ffx, dims, lam, batch):
    rng = np.random.default_rng(batch + sum(dims))
    dx, t = (0.25, 0.3, 0.2)[:len(dims)], 6.0
    psi = random_field(rng, (batch,) + dims)
    ref = O.expand_field(psi, dx, t, lam)
    dens = np.abs(ref) ** 2
    start = rng.random(size=dims).astype(np.float32)
    grad = rng.normal(size=(batch,) + dims).astype(np.float32)
    x = to_dev(psi)
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True) as plan:
        assert not plan.bf16_chain(batch)
        rho = ffx.ffx_expand(plan, x).cpu().numpy()
        fld = ffx.ffx_expand_field(plan, x).cpu().numpy()
        y = x.clone()
        ffx.ffx_expand_field(plan, y, y)  # in place
        assert np.array_equal(y.cpu().numpy(), fld)
        g = ffx.ffx_expand_backward(plan, x, to_dev(grad)).cpu().numpy()
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, accumulate=True) as plan:
        acc = ffx.ffx_expand(plan, x, to_dev(start.copy())).cpu().numpy()
        assert plan.device_errors() == 0
    with ffx.Plan(dims, dx, t, lam, form="tc", bf16=True, unsplit=True) as plan:
        rough = ffx.ffx_expand(plan, x).cpu().numpy()
        assert plan.device_errors() == 0
    assert rel_l2(rho, dens) < DENSITY_TOL
    assert rel_l2(fld, ref) < FIELD_TOL
    assert rel_l2(acc, start + dens.sum(0)) < DENSITY_TOL
    assert rel_l2(g, O.density_loss_gradient(psi, grad, dx, t, lam)) < FIELD_TOL
    assert rel_l2(rough, dens) < UNSPLIT_TOL
