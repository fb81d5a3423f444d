"""The expansion of the inversion grids on both sides of its rule (through rows of coarse nodes, or at
once where these are many), against dense FP64 sums; and the time of many coarse nodes along phi."""
import numpy as np
import pytest

from test_gpu_descent import _grid, _hats

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,cp,H", [((4, 5, 40), 50, 1), ((4, 5, 40), 51, 1), ((6, 4, 40), 35, 5), ((6, 4, 40), 36, 5),
                                        ((4, 4, 4), 3, 1), ((4, 4, 4), 900, 2), ((5, 6, 33), 27, 64)])
def test_expansion(shape, cp, H):
    import torch
    import paper_2412_00031_gb300 as tt
    coarse = (5, 3, cp)
    ctx = tt.tt_ctx_create(_grid(shape))
    G = np.random.default_rng(cp).standard_normal((H,) + coarse)
    W = [_hats(n, c, H) for n, c in zip(shape, coarse)]
    want = sum(np.einsum("ai,bj,ck,abc->ijk", W[0][h], W[1][h], W[2][h], G[h]) for h in range(H)) / H
    D = torch.full(shape, float("nan"), dtype=torch.float64, device="cuda")
    tt.tt_mgrid_expand(ctx, tt.mgrid(*coarse, H), torch.as_tensor(G, device="cuda"), D)
    # eight products of weights whose tables round at 1e-16 of a coarse index, and a mean over H
    assert np.abs(D.cpu().numpy() - want).max() <= 64 * 2.0 ** -53 * cp * np.abs(G).max()
    ctx.close()


def test_many_coarse_nodes_along_phi_do_not_take_longer():
    """4,096 coarse nodes along phi against 261 (1.3 times the nodes): 13 times as long through rows."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (101, 201, 201)
    ctx = tt.tt_ctx_create(_grid(shape))
    D = torch.empty(shape, dtype=torch.float64, device="cuda")

    def ms(cp):
        G = torch.ones((1, 3, 3, cp), dtype=torch.float64, device="cuda")
        best = np.inf
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            tt.tt_mgrid_expand(ctx, tt.mgrid(3, 3, cp, 1), G, D)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    assert ms(4096) <= 1.5 * ms(261)
    ctx.close()
