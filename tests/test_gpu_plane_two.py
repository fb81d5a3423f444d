"""The plane sweeps with two sources a thread: batches sized from the rule on the device's SMs, so that
every solver crosses it, even ones (neighbours by vector accesses), odd ones and fields off the
pair's alignment (scalar accesses). Their sources have the bits they have in small batches, one
to a thread, also with few blocks, three barrier groups and one iteration; and an odd batch costs
little more than the even one beside it."""
import numpy as np
import pytest

import tt_inputs as I

pytestmark = pytest.mark.gpu

# updates of a time step and SM from which on a thread holds two sources, by solver
LINE = {"lf": 1300, "iso": 2900, "aniso": 4300, "tele": 768, "adj": 2000}


def _steps(na, nb, nc):
    planes = na + nb + nc - 2
    start = [0]
    for o in range(1, 8):
        f = o ^ (o - 1)
        d = min(planes, 2 + (na - 1) * (f >> 2 & 1) + (nb - 1) * (f >> 1 & 1) + (nc - 1) * (f & 1))
        start.append(max(start[-1] + d, start[o - 3] + planes if o >= 3 else 0))
    return start[7] + planes


def _batch(kind, shape):
    """A batch 1.2 times beyond the rule of scalar accesses (which lies at or beyond the pairs')."""
    import torch
    a, b, c = shape if kind == "adj" else [n - 2 for n in shape]
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    n = int(1.2 * LINE[kind] * sm * _steps(a, b, c) / (8.0 * a * b * c)) // 2 * 2 + 2
    assert n <= 4095, (shape, n)
    return n


def _case(kind, shape, n_src):
    w = I.small_case(sum(shape), shape=shape, n_src=4, n_rec=4, aniso=0.0 if kind == "iso" else 0.03)
    u = np.random.default_rng(n_src).uniform(0.02, 0.98, (n_src, 3))
    w.grid = I.GridSpec(*shape, 0.0, 12.0, 0.0, 0.12, 0.0, 0.132)
    return w, np.stack([12.0 * u[:, 0], 0.12 * u[:, 1], 0.132 * u[:, 2]], 1)


def _field(shape, n, shift):
    import torch
    return torch.empty(int(np.prod(shape)) * n + shift, device="cuda")[shift:].view(shape + (n,))


def _check(solve, n, variants):
    """solve(lo, hi, shift, **options) -> (field, iterations, sources of a thread)"""
    import torch
    small = [(lo, min(lo + 20, n)) for lo in sorted({0, n // 3 // 2 * 2 + 1, n // 2 - 10, n - 20})]
    refs = [solve(lo, hi, 0) for lo, hi in small]
    assert all(r[2] == 1 for r in refs)
    for cut, shift, kw in variants:
        out, it, two = solve(0, n - cut, shift, **kw)
        assert two == 2, (cut, shift, kw)
        for (lo, hi), (ref, itr, _) in zip(small, refs):
            hi = min(hi, n - cut)
            assert torch.equal(out[..., lo:hi], ref[..., :hi - lo]), (cut, shift, kw, lo)
            assert np.array_equal(it[lo:hi], itr[:hi - lo]), (cut, shift, kw, lo)


# (sources left out of the even batch, field's offset, options)
VARIANTS = [(0, 0, {}), (1, 0, {}), (0, 1, {}), (1, 1, {}), (1, 0, dict(launch_blocks=7)), (0, 0, dict(launch_blocks=7))]


@pytest.mark.parametrize("kind,scheme", [("lf", 0), ("iso", 1), ("aniso", 2)])
@pytest.mark.parametrize("shape", [(26, 27, 29), (12, 40, 31)])
@pytest.mark.parametrize("max_iter", [1, 40])
def test_forward(kind, scheme, shape, max_iter):
    import torch
    import paper_2412_00031_gb300 as tt
    n = _batch(kind, shape)
    w, src = _case(kind, shape, n)
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in (w.s, w.xi, w.eta))

    def solve(lo, hi, shift, **kw):
        ctx = tt.tt_ctx_create(w.grid.as_dict())
        tau = _field(shape, hi - lo, shift)
        it = tt.tt_forward(ctx, model, src[lo:hi], tau, None,
                           tt.default_opts(tt.TT_F32, scheme=scheme, max_iter_fwd=max_iter, **kw), allow_unconverged=True)
        two = tt.tt_get_stats(ctx)["thread_sources"]
        ctx.close()
        return tau, it, two
    _check(solve, n, VARIANTS + [(c, s, dict(fwd_groups=3)) for c, s in ((0, 0), (1, 0), (0, 1))])


@pytest.mark.parametrize("shape", [(18, 19, 20), (9, 30, 29)])
@pytest.mark.parametrize("max_iter", [1, 40])
def test_teleseismic(shape, max_iter):
    import torch
    import paper_2412_00031_gb300 as tt
    n = _batch("tele", shape)
    w, _ = _case("tele", shape, n)
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in (w.s, w.xi, w.eta))
    gen = torch.Generator(device="cuda").manual_seed(n)
    start = 3.0 + torch.rand(shape + (n,), device="cuda", generator=gen)

    def solve(lo, hi, shift, **kw):
        ctx = tt.tt_ctx_create(w.grid.as_dict())
        T = _field(shape, hi - lo, shift)
        T.copy_(start[..., lo:hi])
        it = tt.tt_forward_tele(ctx, model, T, tt.default_opts(tt.TT_F32, max_iter_fwd=max_iter, tol_fwd=1e-5, **kw),
                                allow_unconverged=True)
        two = tt.tt_get_stats(ctx)["thread_sources"]
        ctx.close()
        return T, it, two
    _check(solve, n, VARIANTS + [(1, 0, dict(fwd_groups=3))])


@pytest.mark.parametrize("shape", [(18, 19, 20), (9, 30, 29)])
@pytest.mark.parametrize("max_iter", [1, 40])
def test_adjoint(shape, max_iter):
    import torch
    import paper_2412_00031_gb300 as tt
    n = _batch("adj", shape)
    w, src = _case("adj", shape, n)
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in (w.s, w.xi, w.eta))
    ctx = tt.tt_ctx_create(w.grid.as_dict())
    tau, T = _field(shape, n, 0), _field(shape, n, 0)
    tt.tt_forward(ctx, model, src, tau, T)
    rng = np.random.default_rng(n)
    rec = src[rng.integers(0, n, 5)] * np.array([0.0, 1.0, 1.0])
    R = torch.as_tensor(rng.standard_normal((n, 5)), device="cuda")

    def solve(lo, hi, shift, **kw):
        P = _field(shape, hi - lo, shift)
        it = tt.tt_adjoint(ctx, model, src[lo:hi], T[..., lo:hi].contiguous(), rec, R[lo:hi].contiguous(), P,
                           tt.default_opts(tt.TT_F32, max_iter_adj=max_iter, **kw), allow_unconverged=True)
        return P, it, tt.tt_get_stats(ctx, tt.TT_STATS_ADJOINT)["thread_sources"]
    _check(solve, n, VARIANTS + [(1, 0, dict(adj_groups=3)), (0, 0, dict(adj_groups=3))])
    ctx.close()


@pytest.mark.parametrize("kind,scheme,below,above", [("lf", 0, 550, 1000), ("iso", 1, 2000, 2600), ("aniso", 2, 2500, 3200)])
def test_even_batches_on_both_sides_of_the_line(kind, scheme, below, above):
    """A Godunov thread holds a pair only from larger batches on than an LF one; the bits do not tell."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (26, 27, 29)
    per = _batch(kind, shape) / (1.2 * LINE[kind])
    n, m = (int(x * per) // 2 * 2 for x in (above, below))
    w, src = _case(kind, shape, n)
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in (w.s, w.xi, w.eta))
    ctx = tt.tt_ctx_create(w.grid.as_dict())
    tau = []
    for k, want in ((n, 2), (m, 1)):
        tau.append(_field(shape, k, 0))
        tt.tt_forward(ctx, model, src[:k], tau[-1], None, tt.default_opts(tt.TT_F32, scheme=scheme))
        assert tt.tt_get_stats(ctx)["thread_sources"] == want
    assert torch.equal(tau[0][..., :m], tau[1])
    ctx.close()


@pytest.mark.parametrize("shift", [0, 1])
def test_an_odd_batch_costs_little_more(shift):
    """399 sources against 400 at 81^3: 1.34 times as long with a source a thread."""
    import torch
    import paper_2412_00031_gb300 as tt
    shape = (81, 81, 81)
    w, src = _case("lf", shape, 400)
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in (w.s, w.xi, w.eta))
    ctx = tt.tt_ctx_create(w.grid.as_dict())

    def ms(n, shift):
        tau = _field(shape, n, shift)
        o = tt.default_opts(tt.TT_F32, max_iter_fwd=3, fwd_order=1)
        best = np.inf
        for _ in range(3):
            tt.tt_forward(ctx, model, src[:n], tau, None, o, allow_unconverged=True)
            best = min(best, tt.tt_get_stats(ctx)["sweep_ms"])
        return best
    assert ms(400 - (1 - shift), shift) <= 1.2 * ms(400, 0)
    ctx.close()
