"""The tensor-core convolutions of planes small enough that a tile takes those of several grids: the bits
of every grid by itself, at planes of 25 to 60 rows (four to two grids a tile) and just beyond, batches
that leave the last tile part empty, walks of some planes; gradients against the FP32 path; time."""
import numpy as np
import pytest

from test_gpu_net_walk import _setup

pytestmark = pytest.mark.gpu

# rows of a plane: 25, 36, 45, 56, 60, 63 (a grid a tile)
SHAPES = [((4, 4, 4), 6), ((9, 5, 5), 4), ((61, 4, 8), 170), ((5, 6, 7), 3), ((7, 4, 11), 2), ((12, 6, 8), 5)]


@pytest.mark.parametrize("shape,n", SHAPES + [((6, 4, 4), 2), ((5, 5, 5), 7)])
def test_inference_does_not_depend_on_the_batch(shape, n):
    import torch
    import paper_2412_00031_gb300 as tt
    ctx, theta, x, _ = _setup(tt, shape, n)
    tt.tt_net_set_weights(ctx, theta)
    y = torch.full((n,) + shape, float("nan"), device="cuda")
    tt.tt_net_infer(ctx, x, y)
    for b in range(n):
        one = torch.empty((1,) + shape, device="cuda")
        tt.tt_net_infer(ctx, x[b:b + 1].contiguous(), one)
        assert bool(torch.isfinite(one).all()) and torch.equal(one[0], y[b]), b
    ctx.close()


@pytest.mark.parametrize("shape,n", SHAPES)
def test_training_gradient_matches_the_fp32_path(shape, n):
    """As in test_gpu_net_walk: positive values, an entry off by its BF16 roundings alone."""
    import torch
    import paper_2412_00031_gb300 as tt
    ctx, theta, x, gen = _setup(tt, shape, n)
    theta, x = theta.abs(), x.abs()
    target = torch.zeros((n,) + shape, device="cuda")
    mask = (torch.rand((n,) + shape, device="cuda", generator=gen) > 0.2).float()
    g, ref = torch.empty_like(theta), torch.empty_like(theta)
    loss = tt.tt_net_loss_grad_tc(ctx, theta, x, target, mask, g)
    want = tt.tt_net_loss_grad(ctx, theta, x, target, mask, ref)
    ctx.close()
    assert abs(loss / want - 1) <= 16 * 2.0 ** -9
    assert ((g - ref).abs() <= 16 * 2.0 ** -9 * ref).all()


def test_small_planes_do_not_cost_as_much_as_full_tiles():
    """256 grids of 121x4x4 nodes (25 rows a plane) against 121x10x10 (121 rows): as long with a tile
    for each plane."""
    import torch
    import paper_2412_00031_gb300 as tt

    def ms(shape):
        ctx, theta, x, _ = _setup(tt, shape, 256)
        tt.tt_net_set_weights(ctx, theta)
        y = torch.empty((256,) + shape, device="cuda")
        best = np.inf
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            tt.tt_net_infer(ctx, x, y)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ctx.close()
        return best
    assert ms((121, 4, 4)) <= 0.6 * ms((121, 10, 10))
