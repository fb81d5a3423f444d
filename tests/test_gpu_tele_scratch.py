"""The 2-D teleseismic solve's scratch for the nodes' constants: what a large call takes is given
back, and events beyond the scratch's limit (in further launches, or without the constants where a
launch would hold too few of them) have the times of the same events in a small batch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def _setup(n_r, n_ev, dtype):
    import torch
    import paper_2412_00031_gb300 as tt
    ctx = tt.tt_ctx_create(dict(n_r=4, n_t=4, n_p=4, depth_min_km=0.0, depth_max_km=40.0, lat_min_deg=0.0,
                                lat_max_deg=1.0, lon_min_deg=0.0, lon_max_deg=1.0, earth_radius_km=6371.0, flat=0))
    r = np.linspace(5971.0, 6371.0, n_r)
    s_r = torch.as_tensor(1.0 / (5.8 + 3.0 * (6371.0 - r) / 400.0), dtype=dtype, device="cuda")
    return tt, ctx, s_r, np.random.default_rng(n_ev).uniform(6060.0, 6340.0, n_ev)


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_a_large_call_gives_its_scratch_back():
    import torch
    n_ev, n_r, n_d = 1000, 201, 401
    tt, ctx, s_r, radii = _setup(n_r, n_ev, torch.float64)
    T = torch.empty((n_ev, n_r, n_d), dtype=torch.float64, device="cuda")
    before = _free()
    tt.tt_tele2d(ctx, s_r, 5971.0, 6371.0, 20.0, radii, T, max_iter=1, allow_unconverged=True)
    kept = before - _free()
    # tau and a little more; the constants of all events are four times T
    assert kept < T.numel() * 8 + 1.5 * GIB, kept
    tt.tt_tele2d(ctx, s_r, 5971.0, 6371.0, 20.0, radii[:200], T[:200], max_iter=1, allow_unconverged=True)
    assert before - _free() < T.numel() * 8 + 1.5 * GIB
    ctx.close()


@pytest.mark.parametrize("n_r,n_d,n_ev", [(201, 401, 13500), (16384, 4096, 17)])
def test_events_beyond_the_scratch(n_r, n_d, n_ev):
    """34 GB of constants for 13,500 events (two launches); 17 events of 2 GiB each (16 fit: too few
    blocks, so no constants)."""
    import torch
    tt, ctx, s_r, radii = _setup(n_r, n_ev, torch.float64)
    T = torch.empty((n_ev, n_r, n_d), dtype=torch.float64, device="cuda")
    solve = lambda r, out: tt.tt_tele2d(ctx, s_r, 5971.0, 6371.0, 20.0, r, out, max_iter=1, allow_unconverged=True)
    solve(radii, T)
    for lo in (0, n_ev // 2, n_ev - 2):
        few = torch.empty((2, n_r, n_d), dtype=torch.float64, device="cuda")
        solve(radii[lo:lo + 2], few)
        assert bool(torch.isfinite(few).all()) and torch.equal(few, T[lo:lo + 2])
    ctx.close()
    del T, few
    _free()
