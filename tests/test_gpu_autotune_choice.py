"""tt_autotune's choice against the default launch over whole solves in the batch order of repeated
calls: it is not slower by more than two runs of one launch differ."""
import numpy as np
import pytest

import tt_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n_src,scheme", [((81, 81, 81), 1024, 0), ((101, 121, 121), 256, 0), ((101, 121, 121), 256, 2)])
def test_the_choice_is_not_slower_than_the_default(shape, n_src, scheme):
    import torch
    import paper_2412_00031_gb300 as tt
    w = I.small_case(3, shape=shape, n_src=4, n_rec=4)
    u = np.random.default_rng(n_src).uniform(0.02, 0.98, (n_src, 3))
    g = w.grid
    src = np.stack([g.depth_min_km + u[:, 0] * (g.depth_max_km - g.depth_min_km),
                    g.lat_min_deg + u[:, 1] * (g.lat_max_deg - g.lat_min_deg),
                    g.lon_min_deg + u[:, 2] * (g.lon_max_deg - g.lon_min_deg)], 1)
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in (w.s, w.xi, w.eta))
    ctx = tt.tt_ctx_create(g.as_dict())
    tuned, plain = (tt.default_opts(tt.TT_F32, scheme=scheme) for _ in range(2))
    tt.tt_autotune(ctx, model, src, tuned)
    tau = torch.empty(shape + (n_src,), device="cuda")
    best = [np.inf, np.inf]
    for _ in range(3):
        for q, o in enumerate((tuned, plain)):
            tt.tt_forward(ctx, model, src, tau, None, o)
            best[q] = min(best[q], tt.tt_get_stats(ctx)["sweep_ms"])
    assert best[0] <= 1.015 * best[1], (best, tuned.sweep_schedule, tuned.fwd_groups)
    ctx.close()
