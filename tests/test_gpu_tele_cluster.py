"""The 2-D teleseismic solve with one, two, four and eight blocks an event: an event's times do not
depend on how many others share the launch (1, 30, 70 and 160 events), on grids whose diagonals
are shorter and longer than a cluster's threads."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("n_r,n_d", [(4, 4), (5, 37), (40, 11), (201, 140)])
def test_events_do_not_depend_on_the_batch(f64, n_r, n_d):
    import torch
    import paper_2412_00031_gb300 as tt
    dt = torch.float64 if f64 else torch.float32
    ctx = tt.tt_ctx_create(dict(n_r=4, n_t=4, n_p=4, depth_min_km=0.0, depth_max_km=40.0, lat_min_deg=0.0,
                                lat_max_deg=1.0, lon_min_deg=0.0, lon_max_deg=1.0, earth_radius_km=6371.0, flat=0))
    r = np.linspace(5971.0, 6371.0, n_r)
    s_r = torch.as_tensor(1.0 / (5.8 + 3.0 * (6371.0 - r) / 400.0), dtype=dt, device="cuda")
    radii = np.random.default_rng(n_r).uniform(6060.0, 6340.0, 160)
    ref = None
    for n in (160, 70, 30, 1):
        T = torch.empty((n, n_r, n_d), dtype=dt, device="cuda")
        it = tt.tt_tele2d(ctx, s_r, 5971.0, 6371.0, 20.0, radii[:n], T, tol=1e-9 if f64 else 1e-5)
        if ref is None:
            ref = (T, it)
            assert bool(torch.isfinite(T).all())
        assert torch.equal(T, ref[0][:n]) and np.array_equal(it, ref[1][:n])
    ctx.close()
