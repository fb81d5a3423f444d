"""Values at the ends of the range in the descent step's kernels: infinities and NaN in the phi
contraction."""
import numpy as np
import pytest

from test_gpu_descent import _grid, _hats

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,coarse,H", [((4, 5, 6), (3, 3, 3), 1), ((5, 4, 33), (4, 3, 40), 2),
                                            ((7, 7, 64), (3, 5, 7), 5)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_projection_of_values_that_are_not_finite(shape, coarse, H, value):
    """The dense sums' answer: infinite for the hats over the node, NaN (a zero weight times the
    value) for the others, and NaN in every coefficient for a NaN."""
    import torch
    import paper_2412_00031_gb300 as tt
    rng = np.random.default_rng(11)
    ctx = tt.tt_ctx_create(_grid(shape))
    K = rng.uniform(0.5, 1.0, shape)
    at = (2, 3, shape[2] // 2 + 1)
    K[at] = value
    mg = tt.mgrid(*coarse, H)
    G = torch.zeros((H,) + coarse, dtype=torch.float64, device="cuda")
    tt.tt_mgrid_project(ctx, mg, torch.as_tensor(K, device="cuda"), G)
    got = G.cpu().numpy()
    W = [_hats(n, c, H) for n, c in zip(shape, coarse)]
    w = np.einsum("ha,hb,hc->habc", *[v[:, :, q] for v, q in zip(W, at)])
    want = np.where(w > 0, value * np.ones_like(w), np.nan)
    assert ((got == want) | (np.isnan(got) & np.isnan(want))).all()
    ctx.close()
