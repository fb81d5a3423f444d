"""The phi contraction with one to 16 lanes an output (few coarse nodes along phi), against dense FP64
sums, and its time there."""
import numpy as np
import pytest

from test_gpu_descent import _grid, _hats

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cp,H", [(3, 1), (4, 1), (5, 1), (8, 1), (9, 1), (3, 5), (4, 4), (17, 1), (16, 2)])
@pytest.mark.parametrize("shape", [(4, 5, 4), (5, 4, 33), (4, 6, 200)])
def test_projection(shape, cp, H):
    import torch
    import paper_2412_00031_gb300 as tt
    coarse = (3, 4, cp)
    rng = np.random.default_rng(cp + H)
    ctx = tt.tt_ctx_create(_grid(shape))
    K = rng.standard_normal(shape)
    W = [_hats(n, c, H) for n, c in zip(shape, coarse)]
    r = 6371.0 - np.linspace(40.0, 0.0, shape[0])
    th = np.deg2rad(np.linspace(10.0, 11.0, shape[1]))
    vol = 40.0 / (shape[0] - 1) * np.deg2rad(1.0) / (shape[1] - 1) * np.deg2rad(1.0) / (shape[2] - 1)
    KV = K * (r ** 2)[:, None, None] * np.cos(th)[None, :, None] * vol
    dense = lambda v: np.stack([np.einsum("ai,bj,ck,ijk->abc", W[0][h], W[1][h], W[2][h], v) for h in range(H)]) / H
    G = torch.zeros((H,) + coarse, dtype=torch.float64, device="cuda")
    tt.tt_mgrid_project(ctx, tt.mgrid(*coarse, H), torch.as_tensor(K, device="cuda"), G)
    # sums of at most prod(shape) products of a few roundings each, and weights of size 1
    # whose tables round at 1e-16 of a coarse index
    eps = 2.0 ** -53 * (np.sum(shape) + 64) * max(coarse)
    assert (np.abs(G.cpu().numpy() - dense(KV)) <= eps * (dense(np.abs(KV)) + np.abs(KV).max())).all()
    ctx.close()


def test_a_few_coarse_nodes_do_not_take_longer_than_many():
    """One grid of 3 x 11 x 11 coarse nodes along (phi, r, theta) against 11^3: a ninth of a lane's
    nodes each, but 1.9 times the time with one lane an output."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (101, 201, 201)
    ctx = tt.tt_ctx_create(_grid(shape))
    K = torch.randn(shape, dtype=torch.float64, device="cuda")

    def ms(cp):
        mg = tt.mgrid(11, 11, cp, 1)
        G = torch.zeros((1, 11, 11, cp), dtype=torch.float64, device="cuda")
        best = np.inf
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            tt.tt_mgrid_project(ctx, mg, K, G)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    assert ms(3) <= 1.3 * ms(11)
    ctx.close()


def test_short_hats_do_not_take_longer_than_long_ones_of_as_many_values():
    """Five grids of 11 x 11 x 200 against 11 x 11 x 100 at 101x201x201: twice the outputs, of hats of two
    nodes; 2.0 times the time with an unrolled remainder, 1.6 without."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (101, 201, 201)
    ctx = tt.tt_ctx_create(_grid(shape))
    K = torch.randn(shape, dtype=torch.float64, device="cuda")

    def ms(cp):
        G = torch.zeros((5, 11, 11, cp), dtype=torch.float64, device="cuda")
        best = np.inf
        for _ in range(10):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            tt.tt_mgrid_project(ctx, tt.mgrid(11, 11, cp, 5), K, G)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    assert ms(200) <= 1.8 * ms(100)
    ctx.close()
