"""The descent step's kernels at the edges of their layout: the normalisation with zeta = 1/2, the
sparse phi contraction and the two-step expansion against dense FP64 sums, rows around a
warp and coarse grids wider and narrower than it, values that are not finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _grid(shape):
    return dict(n_r=shape[0], n_t=shape[1], n_p=shape[2], depth_min_km=0.0, depth_max_km=40.0, lat_min_deg=10.0,
                lat_max_deg=11.0, lon_min_deg=0.0, lon_max_deg=1.0, earth_radius_km=6371.0, flat=0)


def _hats(n, c, H):
    x = np.arange(n) / (n - 1) * (c - 2)
    a = np.arange(c)[None, :, None] - np.arange(H)[:, None, None] / H
    return np.maximum(0.0, 1.0 - np.abs(x[None, None] - a))


@pytest.mark.parametrize("shape,coarse,H", [((4, 5, 6), (3, 3, 3), 1), ((5, 4, 33), (4, 3, 40), 2),
                                            ((6, 7, 64), (3, 5, 7), 5), ((4, 9, 31), (5, 11, 33), 3)])
def test_projection_and_expansion(shape, coarse, H):
    import torch
    import paper_2412_00031_gb300 as tt
    rng = np.random.default_rng(sum(shape) + H)
    g = _grid(shape)
    ctx = tt.tt_ctx_create(g)
    K = rng.standard_normal(shape)
    W = [_hats(n, c, H) for n, c in zip(shape, coarse)]
    r = 6371.0 - np.linspace(40.0, 0.0, shape[0])
    th = np.deg2rad(np.linspace(10.0, 11.0, shape[1]))
    vol = 40.0 / (shape[0] - 1) * np.deg2rad(1.0) / (shape[1] - 1) * np.deg2rad(1.0) / (shape[2] - 1)
    KV = K * (r ** 2)[:, None, None] * np.cos(th)[None, :, None] * vol
    want = np.stack([np.einsum("ai,bj,ck,ijk->abc", W[0][h], W[1][h], W[2][h], KV) for h in range(H)]) / H
    size = np.stack([np.einsum("ai,bj,ck,ijk->abc", W[0][h], W[1][h], W[2][h], np.abs(KV)) for h in range(H)]) / H
    mg = tt.mgrid(*coarse, H)
    G = torch.zeros((H,) + coarse, dtype=torch.float64, device="cuda")
    Kd = torch.as_tensor(K, device="cuda")
    tt.tt_mgrid_project(ctx, mg, Kd, G)
    # sums of at most prod(shape) products of a few roundings each, and weights of size 1
    # whose tables round at 1e-16 of a coarse index
    eps = 2.0 ** -53 * (np.sum(shape) + 64) * max(coarse)
    assert (np.abs(G.cpu().numpy() - want) <= eps * (size + np.abs(KV).max())).all()
    D = torch.zeros(shape, dtype=torch.float64, device="cuda")
    Gin = rng.standard_normal(G.shape)
    tt.tt_mgrid_expand(ctx, mg, torch.as_tensor(Gin, device="cuda"), D)
    ref = sum(np.einsum("ai,bj,ck,abc->ijk", W[0][h], W[1][h], W[2][h], Gin[h]) for h in range(H)) / H
    assert np.abs(D.cpu().numpy() - ref).max() <= 64 * 2.0 ** -53 * max(coarse) * np.abs(Gin).max()
    # a value that is not finite reaches every coefficient, as in the dense sums
    Kd[1, 1, 1] = float("inf")
    tt.tt_mgrid_project(ctx, mg, Kd, G)
    assert not bool(torch.isfinite(G).any())
    ctx.close()


@pytest.mark.parametrize("zeta", [0.0, 0.5, 1.0])
def test_normalisation_exponents(zeta):
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (5, 6, 7)
    rng = np.random.default_rng(3)
    ctx = tt.tt_ctx_create(_grid(shape))
    K0 = [rng.standard_normal(shape) for _ in range(3)]
    Kd = rng.uniform(0.0, 9.0, shape)
    Kd[0, 0, 0] = 0.0
    dev = lambda a: torch.as_tensor(a, device="cuda").clone()
    for rel in (False, True):
        K, d = [dev(k) for k in K0], dev(Kd)
        eps = 0.03 * Kd.max() if rel else 1e-3
        if rel:
            tt.tt_kernel_normalize_rel(ctx, *K, d, 0.03, zeta)
        else:
            tt.tt_kernel_normalize(ctx, *K, d, eps, zeta)
        for k, k0 in zip(K, K0):
            want = k0 / (Kd + eps) ** zeta
            # a few units in the last place of pow or rsqrt and two products
            assert (np.abs(k.cpu().numpy() - want) <= 16 * 2.0 ** -53 * np.abs(want)).all()
    ctx.close()
