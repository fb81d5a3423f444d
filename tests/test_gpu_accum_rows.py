"""Kernel accumulation where a phi row is cut into other parts than 32 nodes: grids with few rows and
large batches (down to a node a warp), rows just longer than a multiple of 32, against FP64 sums;
and the time of few nodes with many sources."""
import numpy as np
import pytest

from test_gpu_accum import _reference

pytestmark = pytest.mark.gpu


def _fields(shape, B, dt, seed):
    import torch
    g = dict(n_r=shape[0], n_t=shape[1], n_p=shape[2], depth_min_km=0.0, depth_max_km=30.0, lat_min_deg=1.0,
             lat_max_deg=2.0, lon_min_deg=0.0, lon_max_deg=2.0, earth_radius_km=6371.0, flat=0)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.rand(s, dtype=dt, device="cuda", generator=gen)
    return g, rnd(*shape, B).mul_(20.0), rnd(*shape, B).sub_(0.4), rnd(*shape) + 0.1


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("shape,B", [((4, 4, 4), 1), ((4, 4, 4), 4096), ((5, 4, 11), 4095), ((4, 5, 13), 9),
                                     ((21, 21, 21), 255), ((40, 60, 33), 33), ((40, 60, 33), 5),
                                     ((4, 4, 161), 20), ((50, 80, 97), 2), ((4, 6, 700), 3)])
def test_kernel_sums_match_fp64(f64, shape, B):
    import torch
    import paper_2412_00031_gb300 as tt
    dt = torch.float64 if f64 else torch.float32
    g, T, P, s = _fields(shape, B, dt, 7 * B + shape[2])
    z = torch.zeros_like(s)
    ctx = tt.tt_ctx_create(g)
    K = [torch.full(shape, 0.5, dtype=torch.float64, device="cuda") for _ in range(3)]
    tt.tt_kernel(ctx, (s, z, z), T, P, *K)
    ref, size = _reference(g, s, T, P, 6371.0)
    # each term: two differences, a metric factor of three roundings each, four products and a
    # difference (under 16 roundings of half a unit); the sums are compensated, the reference's not
    eps = 16 * (2.0 ** -53 if f64 else 2.0 ** -24) + (2.0 ** -53 * B if f64 else 0.0)
    for a, r, z1 in zip(K, ref, size):
        assert bool(((a - 0.5 - r).abs() <= eps * z1 + 1e-15 * (1 + r.abs())).all())
    ctx.close()


def test_few_nodes_with_many_sources_do_not_take_longer():
    """The same number of values as 41^3 nodes x 79 sources on 11^3 x 4096, in FP64: six times as long
    with 11 nodes to a warp."""
    import torch
    import paper_2412_00031_gb300 as tt

    def ms(n, B):
        g, T, P, s = _fields((n, n, n), B, torch.float64, 1)
        ctx = tt.tt_ctx_create(g)
        K = [torch.zeros((n, n, n), dtype=torch.float64, device="cuda") for _ in range(3)]
        best = np.inf
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            tt.tt_kernel(ctx, (s, 0 * s, 0 * s), T, P, *K)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ctx.close()
        return best
    assert ms(11, 4096) <= 2.0 * ms(41, 79)
