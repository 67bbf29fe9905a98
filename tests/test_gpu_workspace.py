"""A plan's workspace across calls with other batches and under graph capture:
what one call prepares stays valid for the graphs that use it, and a call that
needs no more than an earlier one can be captured."""

import numpy as np
import pytest
import torch

from gpu_common import random_field, rel_l2, require_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ffx():
    return require_gpu()


def fields(dims, batch, seed=1):
    return to_dev(random_field(np.random.default_rng(seed), (batch,) + dims))


def capture(call):
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


# plans whose sums run in more groups at a smaller batch (the lines of 2048), and
# in partial densities of one group (32 points on the tensor cores)
@pytest.mark.parametrize("dims,lam,form,batch,smaller,larger", [
    ((2048,), (20,), "auto", 1024, 608, 2500),
    ((32,), (5,), "tc", 700, 300, 5000),
])
def test_sum_graph_outlives_other_batches(ffx, dims, lam, form, batch, smaller, larger):
    x = fields(dims, larger)
    with ffx.Plan(dims, (0.2,), 4.0, lam, form=form, accumulate=True) as plan:
        want = ffx.ffx_expand(plan, x[:batch])
        held = plan.workspace_bytes(1)
        ffx.ffx_expand(plan, x[:smaller])
        assert plan.workspace_bytes(1) == held  # (a graph may hold the buffer)
        out = torch.zeros_like(want)
        graph = capture(lambda: ffx.ffx_expand(plan, x[:batch], out))
        ffx.ffx_expand(plan, x[:smaller])
        ffx.ffx_expand(plan, x)  # grows the workspace
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, want)
        assert plan.device_errors() == 0


# a one-dimensional sum needs no workspace: its first call can be captured (the
# groups of lines, and 32-point sums, run without their partial densities then)
@pytest.mark.parametrize("dims,lam,form,batch", [
    ((2048,), (20,), "auto", 64), ((512,), (20,), "auto", 100), ((32,), (5,), "tc", 300),
])
def test_first_sum_of_a_plan_can_be_captured(ffx, dims, lam, form, batch):
    x = fields(dims, batch)
    with ffx.Plan(dims, (0.2,), 4.0, lam, form=form, accumulate=True) as plan:
        out = torch.zeros(dims, device="cuda")
        graph = capture(lambda: ffx.ffx_expand(plan, x, out))
        graph.replay()
        direct = ffx.ffx_expand(plan, x)
        assert plan.device_errors() == 0
    # two orders of one FP32 sum: a few 1e-7
    assert rel_l2(out.cpu().numpy(), direct.cpu().numpy()) < 2e-6


# passes over contiguous FP32 lines: large calls split them in the kernel, small
# ones in a launch of its own into workspace that the large call did not need
@pytest.mark.parametrize("dims,lam,batch,smaller,accumulate", [
    ((96,), (5,), 19537, 40, False),
    ((192,), (7,), 9801, 70, False),
    ((384,), (5,), 13001, 100, False),
    ((384,), (5,), 13001, 1, False),
    ((1024,), (9,), 5000, 300, False),
    ((256,), (9,), 20000, 130, True),
])
def test_smaller_call_can_be_captured(ffx, dims, lam, batch, smaller, accumulate):
    x = fields(dims, batch)
    with ffx.Plan(dims, (0.2,), 4.0, lam, form="tc", bf16=True, accumulate=accumulate) as plan:
        ffx.ffx_expand(plan, x)
        out = torch.zeros(dims if accumulate else (smaller,) + dims, device="cuda")
        graph = capture(lambda: ffx.ffx_expand(plan, x[:smaller], out))
        graph.replay()
        direct = ffx.ffx_expand(plan, x[:smaller])
        assert plan.device_errors() == 0
    # the same split operands and FP32 sums of their products: a few 1e-7
    assert rel_l2(out.cpu().numpy(), direct.cpu().numpy()) < 2e-6


# after a forward call whose last two axes run in one launch: the gradient at the
# same batch and a smaller forward call that takes the axes one by one
@pytest.mark.parametrize("dims,lam,batch,smaller", [((64, 64), (5, 8), 1217, 100), ((64, 64, 64), (5, 3, 7), 20, 3)])
def test_other_calls_after_a_square_call_can_be_captured(ffx, dims, lam, batch, smaller):
    x = fields(dims, batch)
    w = torch.rand((batch,) + dims, device="cuda")
    with ffx.Plan(dims, (0.2,) * len(dims), 4.0, lam, form="tc", bf16=True, fused=False) as plan:
        assert plan.chain_square(batch) and not plan.chain_square(smaller)
        ffx.ffx_expand(plan, x)
        grad, out = torch.zeros_like(x), torch.zeros_like(w[:smaller])
        graph = capture(lambda: ffx.ffx_expand_backward(plan, x, w, grad))
        small = capture(lambda: ffx.ffx_expand(plan, x[:smaller], out))
        graph.replay()
        small.replay()
        want = ffx.ffx_expand_backward(plan, x, w)
        assert torch.equal(grad, want)
        assert torch.equal(out, ffx.ffx_expand(plan, x[:smaller]))
        assert plan.device_errors() == 0


# workspace_bytes against what the plan holds after the call (batch 0 adds nothing):
# fused calls, chains, squares, passes with and without a split launch, FFT forms,
# sums in groups, growing and shrinking batches
@pytest.mark.parametrize("dims,lam,form,accumulate,batches", [
    ((64, 64, 64), (5, 3, 7), "auto", False, (1, 4, 20, 3)),
    ((64, 64), (5, 8), "tc", False, (3, 1217)),
    ((32, 16, 48), (3, 4, 5), "auto", False, (1, 40)),
    ((96, 96, 96), (3, 4, 5), "auto", False, (1, 5)),
    ((48, 96, 192), (7, 11, 4), "auto", False, (2, 1, 5)),
    ((384,), (5,), "tc", False, (100, 13001, 300)),
    ((256, 64, 48), (1, 2, 1), "auto", False, (3,)),
    ((16, 512), (3, 6), "fold", True, (2, 77)),
    ((2048,), (20,), "auto", True, (1, 608, 700, 300, 2500)),
    ((32, 32, 64), (5, 6, 7), "tc", True, (2, 45)),
    ((96, 64), (5, 9), "auto", True, (61, 331, 1000)),
    ((48, 256), (5, 9), "tc", True, (100, 7)),
    ((256,), (9,), "tc", True, (1000, 20000, 30)),
])
def test_workspace_bytes(ffx, dims, lam, form, accumulate, batches):
    x = fields(dims, max(batches))
    with ffx.Plan(dims, (0.2,) * len(dims), 4.0, lam, form=form, accumulate=accumulate) as plan:
        for batch in batches:
            told = plan.workspace_bytes(batch)
            ffx.ffx_expand(plan, x[:batch])
            assert plan.workspace_bytes(0) == told == plan.workspace_bytes(batch)


# a capture at a batch above those called before, whose groups fit what is there
def test_captured_sum_uses_the_groups_that_fit(ffx):
    dims, batch = (2048,), 700
    x = fields(dims, batch)
    with ffx.Plan(dims, (0.2,), 4.0, (20,), accumulate=True) as plan:
        ffx.ffx_expand(plan, x[:512])
        out = torch.zeros(dims, device="cuda")
        graph = capture(lambda: ffx.ffx_expand(plan, x, out))
        graph.replay()
        assert torch.equal(out, ffx.ffx_expand(plan, x))
