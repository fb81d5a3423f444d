"""The FP32 2-D teleseismic solve on both sides of its rules (the nodes' constants kept or computed at
every update, one block or eight for an event): the times of an event do not depend on how many
share the launch and agree with FP64, and few events take no longer than many."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,n_d", [(91, 90), (91, 91), (769, 769), (770, 768), (770, 769), (771, 900)])
def test_events_do_not_depend_on_the_batch(n_r, n_d):
    import torch
    import paper_2412_00031_gb300 as tt
    ctx = tt.tt_ctx_create(dict(n_r=4, n_t=4, n_p=4, depth_min_km=0.0, depth_max_km=40.0, lat_min_deg=0.0,
                                lat_max_deg=1.0, lon_min_deg=0.0, lon_max_deg=1.0, earth_radius_km=6371.0, flat=0))
    r = np.linspace(5971.0, 6371.0, n_r)
    s_r = torch.as_tensor(1.0 / (5.8 + 3.0 * (6371.0 - r) / 400.0), device="cuda")
    radii = np.random.default_rng(n_r).uniform(6060.0, 6340.0, 21)

    def solve(n, dt):
        T = torch.empty((n, n_r, n_d), dtype=dt, device="cuda")
        it = tt.tt_tele2d(ctx, s_r.to(dt), 5971.0, 6371.0, 20.0, radii[:n], T, tol=3e-5, max_iter=40,
                          allow_unconverged=True)
        return T, it
    many, itm = solve(21, torch.float32)      # 21 events: no room for eight blocks each
    for n in (19, 2):
        few, it = solve(n, torch.float32)
        assert torch.equal(few, many[:n]) and np.array_equal(it, itm[:n])
    # one iteration more or less moves tau by the tolerance; FP32 rounding of a path of n_r + n_d
    # updates, relative to the largest time
    ref, _ = solve(2, torch.float64)
    err = (many[:2].double() - ref).abs().max() / ref.abs().max()
    assert float(err) <= 3e-5 * 4 + 2.0 ** -23 * (n_r + n_d), float(err)
    ctx.close()


def test_few_events_do_not_take_longer_than_many():
    """24 events of 201x401 nodes against 150, one SM each: with clusters of blocks or the constants
    read back 24 took 1.7 times as long."""
    import torch
    import paper_2412_00031_gb300 as tt
    ctx = tt.tt_ctx_create(dict(n_r=4, n_t=4, n_p=4, depth_min_km=0.0, depth_max_km=40.0, lat_min_deg=0.0,
                                lat_max_deg=1.0, lon_min_deg=0.0, lon_max_deg=1.0, earth_radius_km=6371.0, flat=0))
    s_r = torch.as_tensor(1.0 / np.linspace(8.8, 5.8, 201), dtype=torch.float32, device="cuda")
    radii = np.random.default_rng(1).uniform(6060.0, 6340.0, 150)
    T = torch.empty((150, 201, 401), device="cuda")

    def ms(n):
        best = np.inf
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            tt.tt_tele2d(ctx, s_r, 5971.0, 6371.0, 20.0, radii[:n], T[:n], tol=1e-5, max_iter=6, allow_unconverged=True)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    assert ms(24) <= 1.25 * ms(150)
    ctx.close()
