"""Values at the ends of the range in the descent step's kernels: infinities and NaN in the phi
contraction, and powers of the normalisation that over- or underflow."""
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


@pytest.mark.parametrize("zeta", [0.5, 1.0, 2.0, 3.0])
def test_relative_normalisation_where_the_power_overflows(zeta):
    """Factors x^-zeta of densities from 1e-120 to 1e160, against the same power in extended
    precision: x^2 and x^3 overflow where their reciprocals are still FP64 numbers (subnormal ones
    among them), and a large kernel times the factor is an ordinary number."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (5, 6, 7)
    ctx = tt.tt_ctx_create(_grid(shape))
    rng = np.random.default_rng(5)
    for top in (1e-100, 1.0, 1e104, 1e155, 1e160):
        Kd = top * rng.uniform(0.1, 1.0, shape)
        x = Kd + 1e-3 * Kd.max()
        want = np.power(x.astype(np.longdouble), -np.longdouble(zeta))
        K0 = np.full(shape, 1e140 if top > 1e10 else 1.0)
        K = [torch.as_tensor(K0, device="cuda").clone() for _ in range(3)]
        tt.tt_kernel_normalize_rel(ctx, *K, torch.as_tensor(Kd, device="cuda"), 1e-3, zeta)
        got = K[0].cpu().numpy() / K0.astype(np.longdouble)
        # pow and rsqrt to 2 units in the last place, the sum x, the product and the division of
        # this check to one each (x's error zeta times); the factor's own spacing where subnormal
        tol = (8 + 2 * zeta) * 2.0 ** -53 * want + 2 * np.longdouble(5e-324)
        ok = np.abs(got - want) <= tol
        finite = want < np.finfo(np.float64).max
        assert ok[finite].all() and np.isinf(got[~finite]).all()
    ctx.close()


@pytest.mark.parametrize("zeta", [0.5, 0.75])
@pytest.mark.parametrize("rel", [False, True])
def test_normalisation_of_densities_that_are_not_positive(zeta, rel):
    """(Kd + eps)^-zeta of negative, infinite and NaN densities, by pow's rules."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (4, 4, 4)
    ctx = tt.tt_ctx_create(_grid(shape))
    Kd = np.ones(shape)
    Kd[0, 0] = [-2.0, -np.inf, np.nan, 1.0]
    K = [torch.ones(shape, dtype=torch.float64, device="cuda") for _ in range(3)]
    d = torch.as_tensor(Kd, device="cuda")
    if rel:
        tt.tt_kernel_normalize_rel(ctx, *K, d, 1e-16, zeta)   # the largest |Kd| is infinite
        want = [0.0, np.nan, np.nan, 0.0]
    else:
        tt.tt_kernel_normalize(ctx, *K, d, 1e-3, zeta)
        want = [np.nan, 0.0, np.nan, 1.001 ** -zeta]
    for k in K:
        assert np.allclose(k[0, 0].cpu().numpy(), want, rtol=1e-14, atol=0.0, equal_nan=True)
    ctx.close()
