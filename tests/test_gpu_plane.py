"""The plane sweep (orderings in flight together, faces completed on the way, two sources a thread
in large batches) against the tile schedule, which waits for every ordering and extrapolates
the faces in passes: the same bits at the smallest and ragged extents, odd and even batches
on both sides of the pair rule, fields off the pair's alignment, few blocks and barrier groups."""
import numpy as np
import pytest

import tt_inputs as I

pytestmark = pytest.mark.gpu


def _case(seed, shape, n_src, aniso=0.03):
    """A small heterogeneous case with sources anywhere inside the grid, near its faces too."""
    w = I.small_case(seed, shape=tuple(max(n, 7) for n in shape), n_src=n_src, n_rec=4, aniso=aniso)
    rng = np.random.default_rng(seed)
    g = I.GridSpec(*shape, 0.0, 12.0, 0.0, 0.12, 0.0, 0.132)
    cut = tuple(slice(0, n) for n in shape)
    u = rng.uniform(0.02, 0.98, (n_src, 3))
    src = np.stack([12.0 * u[:, 0], 0.12 * u[:, 1], 0.132 * u[:, 2]], 1)
    w.grid, w.src = g, src
    w.s, w.xi, w.eta = (np.ascontiguousarray(a[cut]) for a in (w.s, w.xi, w.eta))
    return w


def _solve(tt, w, opts, shift=0, dtype=None):
    import torch
    dt = dtype or torch.float32
    model = tuple(torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda") for a in (w.s, w.xi, w.eta))
    ctx = tt.tt_ctx_create(w.grid.as_dict())
    n = int(np.prod(w.grid.shape)) * w.n_src
    buf = torch.empty(n + shift, dtype=dt, device="cuda")
    tau = buf[shift:].view(w.grid.shape + (w.n_src,))
    it = tt.tt_forward(ctx, model, w.src, tau, None, opts, allow_unconverged=True)
    out = tau.cpu().numpy()
    ctx.close()
    return out, it


@pytest.mark.parametrize("shape,n_src", [((4, 4, 4), 32), ((4, 5, 9), 36), ((5, 4, 4), 40), ((9, 4, 21), 32),
                                         ((4, 23, 5), 36), ((23, 6, 7), 32), ((18, 19, 20), 704),
                                         ((7, 30, 29), 900)])
@pytest.mark.parametrize("max_iter", [1, 60])
def test_plane_sweep_gives_the_tile_schedule_bits(shape, n_src, max_iter):
    import paper_2412_00031_gb300 as tt
    w = _case(40 + sum(shape), shape, n_src)
    o = lambda **kw: tt.default_opts(tt.TT_F32, max_iter_fwd=max_iter, **kw)
    ref, itr = _solve(tt, w, o(sweep_schedule=2))
    for kw, shift in (({}, 0), ({}, 1), ({"launch_blocks": 3}, 0), ({"fwd_groups": 3}, 0)):
        out, it = _solve(tt, w, o(**kw), shift)
        assert np.array_equal(it, itr), (kw, shift)
        assert np.array_equal(out, ref), (kw, shift)


@pytest.mark.parametrize("scheme", [0, 1, 2])
@pytest.mark.parametrize("n_src", [1, 3, 33, 700])
@pytest.mark.parametrize("f64", [False, True])
def test_plane_sweep_gives_the_refill_bits(scheme, n_src, f64):
    """Against the retire-and-refill sweep (one hyperplane at a time, 32 slots): sources of a batch
    do not see each other, so a batch that is padded by repeated sources to use it has the bits of
    the batch itself."""
    import torch
    import paper_2412_00031_gb300 as tt
    w = _case(90 + n_src, (12, 14, 17), n_src, 0.0 if scheme == 1 else 0.03)
    code, dt = (tt.TT_F64, torch.float64) if f64 else (tt.TT_F32, torch.float32)
    out, it = _solve(tt, w, tt.default_opts(code, scheme=scheme), dtype=dt)
    big = w.subset(list(range(n_src)) + [0] * 40)
    ref, itr = _solve(tt, big, tt.default_opts(code, scheme=scheme, fwd_slots=32), dtype=dt)
    assert np.array_equal(it, itr[:n_src])
    assert np.array_equal(out, ref[..., :n_src])


@pytest.mark.parametrize("shape,n_src", [((4, 4, 4), 40), ((4, 9, 5), 33), ((16, 18, 17), 800), ((7, 30, 29), 900)])
@pytest.mark.parametrize("max_iter", [1, 60])
def test_plane_adjoint_does_not_depend_on_the_batch(shape, n_src, max_iter):
    """The adjoint of a large batch (pairs of sources a thread above some hundred) has the bits of its
    sources in slices of 31 (a source a thread), at the smallest extents and with unaligned fields,
    source slices, barrier groups and few blocks."""
    import torch
    import paper_2412_00031_gb300 as tt
    w = _case(7 * sum(shape), shape, n_src)
    rng = np.random.default_rng(n_src)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")
    model = tuple(dev(a) for a in (w.s, w.xi, w.eta))
    ctx = tt.tt_ctx_create(w.grid.as_dict())
    tau, T = (torch.empty(shape + (n_src,), device="cuda") for _ in range(2))
    tt.tt_forward(ctx, model, w.src, tau, T)
    rec = w.src[rng.integers(0, n_src, 5)] * np.array([0.0, 1.0, 1.0])
    R = torch.as_tensor(rng.standard_normal((n_src, 5)), device="cuda")

    def solve(lo, hi, shift=0, **kw):
        buf = torch.empty(int(np.prod(shape)) * (hi - lo) + shift, device="cuda")
        P = buf[shift:].view(shape + (hi - lo,))
        it = tt.tt_adjoint(ctx, model, w.src[lo:hi], T[..., lo:hi].contiguous(), rec, R[lo:hi].contiguous(), P,
                           tt.default_opts(tt.TT_F32, max_iter_adj=max_iter, **kw), allow_unconverged=True)
        return P, it
    P, it = solve(0, n_src)
    for lo in range(0, n_src, 31 * (1 + n_src // 200)):
        hi = min(lo + 31, n_src)
        p, i = solve(lo, hi)
        assert torch.equal(p, P[..., lo:hi]) and np.array_equal(i, it[lo:hi])
    for kw in (dict(shift=1), dict(adj_chunk=64), dict(adj_groups=3), dict(launch_blocks=5)):
        p, i = solve(0, n_src, **kw)
        assert torch.equal(p, P) and np.array_equal(i, it), kw
    ctx.close()
