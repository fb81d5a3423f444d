"""Kernel accumulation (Eqs. 6-8) at the sizes where its layout changes: batches around the
vector width and the warp, phi rows around the 32 nodes of a warp, both precisions, unaligned
fields. Reference: the same sums in FP64 by plain torch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _reference(g, s, T, P, re):
    import torch
    deg = np.pi / 180.0
    dev = T.device
    r = torch.linspace(re - g["depth_max_km"], re - g["depth_min_km"], g["n_r"], dtype=torch.float64, device=dev)
    th = torch.linspace(g["lat_min_deg"], g["lat_max_deg"], g["n_t"], dtype=torch.float64, device=dev) * deg
    dt = (g["lat_max_deg"] - g["lat_min_deg"]) * deg / (g["n_t"] - 1)
    dp = (g["lon_max_deg"] - g["lon_min_deg"]) * deg / (g["n_p"] - 1)
    T, P, s = T.double(), P.double(), s.double()

    def d(n, axis, h):
        up = torch.arange(n, device=dev).add(1).clamp(max=n - 1)   # indices: widened below
        dn = torch.arange(n, device=dev).sub(1).clamp(min=0)
        sh = [1, 1, 1, 1]
        sh[axis] = n
        return (T.index_select(axis, up) - T.index_select(axis, dn)) / ((up - dn).double() * h).view(sh)
    gt = d(g["n_t"], 1, dt) / r[:, None, None, None]
    gp = d(g["n_p"], 2, dp) / (r[:, None, None, None] * torch.cos(th)[None, :, None, None])
    terms = [P * (s * s)[..., None], P * (gt * gt - gp * gp), -2 * P * gt * gp]
    size = [(P * (s * s)[..., None]).abs(), P.abs() * (gt * gt + gp * gp), (2 * P * gt * gp).abs()]
    return [t.sum(-1) for t in terms], [t.sum(-1) for t in size]


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("B,n_p,shift", [(1, 31, 0), (3, 32, 0), (4, 33, 0), (4, 33, 1), (31, 40, 0),
                                         (36, 65, 0), (128, 5, 0), (130, 4, 0), (260, 7, 0)])
def test_kernel_sums_match_fp64(f64, B, n_p, shift):
    import torch
    import paper_2412_00031_gb300 as tt
    dt = torch.float64 if f64 else torch.float32
    g = dict(n_r=4, n_t=5, n_p=n_p, depth_min_km=0.0, depth_max_km=30.0, lat_min_deg=1.0, lat_max_deg=2.0,
             lon_min_deg=0.0, lon_max_deg=2.0, earth_radius_km=6371.0, flat=0)
    shape = (4, 5, n_p)
    gen = torch.Generator(device="cuda").manual_seed(100 * B + n_p)
    rnd = lambda *s: torch.rand(s, dtype=dt, device="cuda", generator=gen)
    n = 4 * 5 * n_p * B
    # shift: fields that start off a 16-byte boundary
    T = rnd(n + shift)[shift:].view(shape + (B,)).mul_(20.0)
    P = rnd(n + shift)[shift:].view(shape + (B,)).sub_(0.4)
    s = rnd(*shape) + 0.1
    z = torch.zeros_like(s)
    ctx = tt.tt_ctx_create(g)
    K = [torch.full(shape, 0.5, dtype=torch.float64, device="cuda") for _ in range(3)]
    tt.tt_kernel(ctx, (s, z, z), T, P, *K)
    ref, size = _reference(g, s, T, P, 6371.0)
    # each term: two differences, a metric factor of three roundings each, four products and a
    # difference (under 16 roundings of half a unit); the sums are compensated
    eps = 16 * (2.0 ** -53 if f64 else 2.0 ** -24)
    for a, r, z1 in zip(K, ref, size):
        assert bool(((a - 0.5 - r).abs() <= eps * z1 + 1e-15 * (1 + r.abs())).all())
    ctx.close()
