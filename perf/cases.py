"""What is measured of the traveltime library, as a user's program calls it.

A case is one call, or one short fixed sequence of calls, of the package's public binding:
  forward   tt_forward: the Eikonal solves of a batch of sources (or of stations, by reciprocity)
  adjoint   tt_adjoint: the adjoint solves of a batch for given times and adjoint sources
  step      tt_plan_run: a whole inversion step over a batch (forward, misfit, adjoint, kernels)
  kernel    tt_kernel: the sensitivity kernels of a batch, summed over its sources
  start     tt_net_start: the learned warm start of a batch
  train     tt_net_loss_grad_tc and tt_net_adam: one training step of the warm-start network
  descent   tt_kernel_normalize_rel, tt_mgrid_project, tt_mgrid_expand, tt_model_update:
            from kernels to the updated model
  tele      tt_tele2d, tt_tele_region_times, tt_forward_tele: teleseismic events

Grids are nr x nt x np nodes (depth, latitude, longitude), 0.8 km and 0.025 degrees apart.
Models are a velocity rising from 5 to 8 km/s with depth times a checkerboard of seeded
phases, with checkerboards of xi and eta where the case is anisotropic.
"""
import math

import numpy as np
import torch

import paper_2412_00031_gb300 as tt
from paper_2412_00031_gb300 import warmstart

RE = 6371.0
DEG = math.pi / 180.0
DR_KM, DLL_DEG = 0.8, 0.025
F64 = torch.float64


def listed():
    return [
        # the smallest call: one source on a 41^3 grid, double precision (a first solve, a check)
        dict(name="forward 41^3 1 src f64", kind="forward", nr=41, nt=41, np=41, src=1, f64=True,
             aniso=True, scheme=0, rec=0),
        # one event or station traced through the large region
        dict(name="forward 121x161x161 1 src", kind="forward", nr=121, nt=161, np=161, src=1,
             f64=False, aniso=True, scheme=2, rec=0),
        # an odd batch on a ragged grid with the default solver
        dict(name="forward 67x83x95 37 src", kind="forward", nr=67, nt=83, np=95, src=37,
             f64=False, aniso=True, scheme=0, rec=0),
        # double-precision adjoint of a few events
        dict(name="adjoint 41x61x67 6 src f64", kind="adjoint", nr=41, nt=61, np=67, src=6,
             f64=True, aniso=True, scheme=0, rec=64),
        # an inversion step of the isotropic checkerboard test
        dict(name="step 81^3 64 src", kind="step", nr=81, nt=81, np=81, src=64, f64=False,
             aniso=False, scheme=0, rec=100),
        # the same with anisotropy on a larger, ragged grid: the default solver's heaviest use
        dict(name="step 101x141x151 112 src", kind="step", nr=101, nt=141, np=151, src=112,
             f64=False, aniso=True, scheme=0, rec=200),
        # the headline region and batch with the Godunov solver
        dict(name="step godunov 121x161x161 256", kind="step", nr=121, nt=161, np=161, src=256,
             f64=False, aniso=True, scheme=2, rec=200),
        # kernels of a batch whose fields are kept
        dict(name="kernel 121x161x161 256 src", kind="kernel", nr=121, nt=161, np=161, src=256,
             f64=False, aniso=True, scheme=0, rec=0),
        # the warm start, and the training of its network
        dict(name="start 121x161x161 32 src", kind="start", nr=121, nt=161, np=161, src=32,
             f64=False, aniso=True, scheme=0, rec=0),
        dict(name="train 81^3 8 grids", kind="train", nr=81, nt=81, np=81, src=8, f64=False,
             aniso=True, scheme=0, rec=0),
        # from an inversion step's kernels to the next model
        dict(name="descent 101x201x201", kind="descent", nr=101, nt=201, np=201, src=1, f64=False,
             aniso=True, scheme=0, rec=0),
        # teleseismic events over a region
        dict(name="tele 81x101x101 24 events", kind="tele", nr=81, nt=101, np=101, src=24,
             f64=False, aniso=True, scheme=0, rec=0),
    ]


# Typical iteration counts of the sweeps (8 orderings each), for the work a solve cannot do
# without: Lax-Friedrichs, Godunov from above, adjoint.
_ITERS = {0: 40, 2: 5}
_ITERS_ADJ = 4


def draw(rng):
    """A case of the listed ranges: any kind, odd and even extents, batches from one source to
    the largest that costs no more than the listed ones of its kind."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forward", "forward", "forward", "adjoint", "step", "step", "kernel",
                       "start", "train", "descent", "tele"])
    f64 = kind in ("forward", "adjoint", "step", "kernel") and rng.random() < 0.25
    scheme = 2 if kind in ("forward", "step") and rng.random() < 0.4 else 0
    hi = {"train": 81, "tele": 101}.get(kind, 61 if f64 else 161)
    nr, nt, np_ = size(21, min(hi, 121)), size(21, hi), size(21, hi)
    # node-source products: bounded by the listed cases of each kind
    most = {"forward": 3e6 if f64 else 4e7, "adjoint": 2e6 if f64 else 6e7,
            "step": 2e6 if f64 else (4e8 if scheme else 2e8), "kernel": 2e8 if f64 else 8e8,
            "start": 1e8, "train": 4.2e6, "descent": 1e9, "tele": 2e7}[kind]
    top = {"train": 8, "start": 64, "tele": 48}.get(kind, 256)
    src = 1 if kind == "descent" else size(1, max(1, min(top, most / (nr * nt * np_))))
    rec = size(20, 200) if kind in ("step", "adjoint") else 0
    return dict(kind=kind, nr=nr, nt=nt, np=np_, src=src, f64=f64,
                aniso=kind in ("start", "train") or scheme == 2 or rng.random() < 0.7,
                scheme=scheme, rec=rec)


# ------------------------------------------------------------------------------ inputs

def _grid(c):
    return dict(n_r=c["nr"], n_t=c["nt"], n_p=c["np"], depth_min_km=0.0,
                depth_max_km=DR_KM * (c["nr"] - 1), lat_min_deg=0.0,
                lat_max_deg=DLL_DEG * (c["nt"] - 1), lon_min_deg=0.0,
                lon_max_deg=DLL_DEG * (c["np"] - 1), earth_radius_km=RE, flat=0)


def _axes(c):
    """Radius (km, ascending), latitude and longitude (radians) of the grid's nodes."""
    a = lambda n: torch.arange(n, dtype=F64, device="cuda")
    r = RE - DR_KM * (c["nr"] - 1) + DR_KM * a(c["nr"])
    return r, a(c["nt"]) * (DLL_DEG * DEG), a(c["np"]) * (DLL_DEG * DEG)


def _model64(c, rng):
    """(s, xi, eta) in double: the 1-D velocity with a seeded checkerboard."""
    x = [torch.linspace(0, 1, n, dtype=F64, device="cuda") for n in (c["nr"], c["nt"], c["np"])]

    def checker(n, phase):
        f = [torch.sin(2 * math.pi * (k * v + p)) for k, v, p in zip(n, x, phase)]
        return f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]

    ph = rng.uniform(0.0, 1.0, (3, 3))
    per = (1.5, 2.0, 2.0)
    v = (5.0 + 3.0 * (1 - x[0]))[:, None, None] * (1.0 + 0.045 * checker(per, ph[0]))
    amp = 0.04 if c["aniso"] else 0.0
    return [t.contiguous() for t in (1.0 / v, amp * checker(per, ph[1]), amp * checker(per, ph[2]))]


def _dtype(c):
    return F64 if c["f64"] else torch.float32


def _points(c, n, rng, surface):
    """n points (depth km, lat, lon) inside the grid, two cells from its sides."""
    g = _grid(c)
    u = rng.uniform(0.0, 1.0, (n, 3))
    depth = np.zeros(n) if surface else g["depth_max_km"] * (0.05 + 0.85 * u[:, 0])
    m = 2 * DLL_DEG
    return np.stack([depth, m + u[:, 1] * (g["lat_max_deg"] - 2 * m),
                     m + u[:, 2] * (g["lon_max_deg"] - 2 * m)], 1)


def _xyz(p):
    r, th, ph = RE - p[:, 0], p[:, 1] * DEG, p[:, 2] * DEG
    return np.stack([r * np.cos(th) * np.cos(ph), r * np.cos(th) * np.sin(ph), r * np.sin(th)], 1)


def _data(c, src, rng):
    """Observations of a batch: per source a seeded subset of the stations, absolute times
    and the common-source pairs closer than one degree."""
    rec = _points(c, c["rec"], rng, True)
    dist = np.linalg.norm(_xyz(src)[:, None] - _xyz(rec)[None], axis=2)
    tobs = dist / 6.2 + 0.05 * rng.standard_normal(dist.shape)
    close = np.hypot(rec[:, None, 1] - rec[None, :, 1], rec[:, None, 2] - rec[None, :, 2]) <= 1.0
    ar, cm, ci = [], [], []
    for n in range(len(src)):
        k = int(rng.integers(min(20, c["rec"]), c["rec"] + 1))
        sub = np.sort(rng.permutation(c["rec"])[:k])
        a, b = np.nonzero(np.triu(close[np.ix_(sub, sub)], 1))
        ar.append(sub)
        cm.append(sub[a])
        ci.append(sub[b])
    off = lambda parts: np.concatenate([[0], np.cumsum([len(p) for p in parts])])
    rows = lambda parts: np.repeat(np.arange(len(parts)), [len(p) for p in parts])
    A, M, I = np.concatenate(ar), np.concatenate(cm), np.concatenate(ci)
    return tt.DeviceData(rec, off(ar), A, tobs[rows(ar), A], np.ones(len(A)), off(cm), M, I,
                         tobs[rows(cm), M] - tobs[rows(cm), I], np.ones(len(M)))


def _smooth_times(c, src, dtype):
    """Times of each source in the medium v = 5 + g depth (closed form of a constant gradient
    along the chord), [nr, nt, np, src]."""
    r, th, ph = _axes(c)
    X = torch.stack([(r[:, None, None] * torch.cos(th)[None, :, None] * torch.cos(ph)).expand(
        c["nr"], c["nt"], c["np"]), (r[:, None, None] * torch.cos(th)[None, :, None]
                                     * torch.sin(ph)).expand(c["nr"], c["nt"], c["np"]),
        (r[:, None] * torch.sin(th)[None]).unsqueeze(-1).expand(c["nr"], c["nt"], c["np"])])
    gr = 3.0 / (DR_KM * (c["nr"] - 1))
    vx = (5.0 + gr * (RE - r))[:, None, None]
    T = torch.empty((c["nr"], c["nt"], c["np"], len(src)), dtype=dtype, device="cuda")
    for b, (p, s) in enumerate(zip(src, _xyz(src))):
        d2 = sum((X[a] - s[a]) ** 2 for a in range(3))
        T[..., b] = torch.arccosh(1.0 + gr * gr * d2 / (2.0 * vx * (5.0 + gr * p[0]))) / gr
    return T


def _inputs(c, seed):
    """The inputs of a case from the seed alone: what prepare() and exact() both start from."""
    rng = np.random.default_rng([int(seed), 7])
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    d = {"rng": rng, "gen": gen, "model64": _model64(c, rng)}
    # what the program holds, in the case's type; exact() starts from these values
    d["model"] = [t.to(_dtype(c)) for t in d["model64"]]
    d["src"] = _points(c, c["src"], rng, False)
    shape = (c["nr"], c["nt"], c["np"])
    if c["kind"] == "adjoint":
        d["rec"] = _points(c, c["rec"], rng, True)
        d["T"] = _smooth_times(c, d["src"], _dtype(c))
        d["R"] = 0.1 * torch.randn((c["src"], c["rec"]), dtype=F64, device="cuda", generator=gen)
    if c["kind"] == "kernel":
        d["T"] = _smooth_times(c, d["src"], _dtype(c))
        d["P"] = torch.randn(shape + (c["src"],), dtype=_dtype(c), device="cuda", generator=gen)
    if c["kind"] == "start":
        d["theta"] = torch.as_tensor(warmstart.init_params(int(seed) % (1 << 31)), device="cuda")
        d["theta"] *= 0.5      # predictions of the size that the clamp lets through
    if c["kind"] == "train":
        d["theta"] = torch.as_tensor(warmstart.init_params(int(seed) % (1 << 31)), device="cuda")
        u = [torch.linspace(0, 1, n, device="cuda") for n in shape]
        p = torch.rand((c["src"], 3), device="cuda", generator=gen)
        f = [torch.sin(2 * math.pi * (v[None] + p[:, a:a + 1])) for a, v in enumerate(u)]
        d["target"] = (1.05 + 0.2 * f[0][:, :, None, None] * f[1][:, None, :, None]
                       * f[2][:, None, None, :]).contiguous()
        d["mask"] = torch.ones_like(d["target"])
    if c["kind"] == "descent":
        d["K"] = [torch.randn(shape, dtype=F64, device="cuda", generator=gen) for _ in range(3)]
        d["Kd"] = 5.0 * torch.rand(shape, dtype=F64, device="cuda", generator=gen)
    if c["kind"] == "tele":
        n = c["src"]
        dist, az = rng.uniform(8.0, 20.0, n), rng.uniform(0.0, 2 * np.pi, n)
        d["events"] = np.stack([rng.uniform(30.0, 300.0, n),
                                0.5 * DLL_DEG * (c["nt"] - 1) + dist * np.cos(az),
                                0.5 * DLL_DEG * (c["np"] - 1) + dist * np.sin(az)], 1)
    return d


_MG = (11, 11, 11, 5)             # the inversion's five offset grids of 11^3
_TELE = (201, 401, 400.0, 25.0)   # 2-D grid of the 1-D model: radii, angles, depth km, degrees


def prepare(case, seed):
    c, d = case, _inputs(case, seed)
    dt = _dtype(c)
    shape = (c["nr"], c["nt"], c["np"])
    new = lambda s, t: torch.empty(s, dtype=t, device="cuda")
    st = {"case": c, "ctx": tt.tt_ctx_create(_grid(c)), "src": d["src"], "model": d["model"]}
    kind = c["kind"]
    opts = tt.default_opts(tt.TT_F64 if c["f64"] else tt.TT_F32)
    if c["scheme"] == 2:
        opts.scheme, opts.init = 2, tt.TT_INIT_ABOVE
    st["opts"] = opts
    if kind == "forward":
        st["tau"], st["T"] = (new(shape + (c["src"],), dt) for _ in range(2))
    elif kind == "adjoint":
        st.update(T=d["T"], R=d["R"], rec=d["rec"], P=new(shape + (c["src"],), dt))
    elif kind == "step":
        data = _data(c, d["src"], d["rng"])
        st["f"] = [new(shape + (c["src"],), dt) for _ in range(3)]
        st["chi"], st["R"] = new((c["src"], 2), F64), new((c["src"], c["rec"]), F64)
        st["K"] = [new(shape, F64) for _ in range(3)]
        st["plan"] = tt.tt_plan_create(st["ctx"], d["model"], d["src"], data, *st["f"], st["chi"],
                                       st["R"], *st["K"], opts=opts)
    elif kind == "kernel":
        st.update(T=d["T"], P=d["P"], K=[new(shape, F64) for _ in range(3)])
    elif kind == "start":
        tt.tt_net_set_stride(st["ctx"], 2)
        tt.tt_net_set_weights(st["ctx"], d["theta"])
        st["tau"] = new(shape + (c["src"],), dt)
    elif kind == "train":
        st["x"] = new((c["src"],) + shape + (tt.NET_FEATURES,), torch.float32)
        tt.tt_net_features(st["ctx"], d["model"], d["src"], st["x"])
        st.update(theta=d["theta"], target=d["target"], mask=d["mask"], step=0)
        st["grad"], st["m"], st["v"] = (torch.zeros_like(d["theta"]) for _ in range(3))
    elif kind == "descent":
        st.update(K0=d["K"], Kd=d["Kd"], model0=[t.clone() for t in d["model"]],
                  mg=tt.mgrid(*_MG), K=[new(shape, F64) for _ in range(3)],
                  D=[new(shape, F64) for _ in range(3)],
                  G=[new((_MG[3],) + _MG[:3], F64) for _ in range(3)])
    elif kind == "tele":
        n_r, n_d, depth, _ = _TELE
        r = np.linspace(RE - depth, RE, n_r)
        st.update(events=d["events"], s_r=torch.as_tensor(
            1.0 / (5.8 + 3.0 * (RE - r) / depth), device="cuda"))
        st["T2"], st["T2f"] = new((c["src"], n_r, n_d), F64), new((c["src"], n_r, n_d), torch.float32)
        st["T"] = new(shape + (c["src"],), torch.float32)
        # FP32 resolves times of a few hundred seconds to about 1.5e-5 s
        st["opts"] = tt.default_opts(tt.TT_F32, tol_fwd=3e-5)
    return st


def run(st):
    c, ctx, kind = st["case"], st["ctx"], st["case"]["kind"]
    if kind == "forward":
        it = tt.tt_forward(ctx, st["model"], st["src"], st["tau"], st["T"], st["opts"])
        return {"tau": st["tau"], "T": st["T"], "iters": it}
    if kind == "adjoint":
        it = tt.tt_adjoint(ctx, st["model"], st["src"], st["T"], st["rec"], st["R"], st["P"],
                           st["opts"])
        return {"P": st["P"], "iters": it}
    if kind == "step":
        itf, ita = tt.tt_plan_run(st["plan"])
        return {"tau": st["f"][0], "T": st["f"][1], "P": st["f"][2], "chi": st["chi"],
                "R": st["R"], "K": st["K"], "iters_fwd": itf, "iters_adj": ita}
    if kind == "kernel":
        for K in st["K"]:
            K.zero_()
        tt.tt_kernel(ctx, st["model"], st["T"], st["P"], *st["K"])
        return {"K": st["K"]}
    if kind == "start":
        tt.tt_net_start(ctx, st["model"], st["src"], st["tau"])
        return {"tau": st["tau"]}
    if kind == "train":
        loss = tt.tt_net_loss_grad_tc(ctx, st["theta"], st["x"], st["target"], st["mask"],
                                      st["grad"])
        st["step"] += 1
        tt.tt_net_adam(ctx, st["theta"], st["grad"], st["m"], st["v"], st["step"])
        return {"loss": loss, "grad": st["grad"], "theta": st["theta"]}
    if kind == "descent":
        # the kernels of an evaluation and the model that a refused step goes back to
        for a, b in zip(st["K"] + st["model"], st["K0"] + st["model0"]):
            a.copy_(b)
        tt.tt_kernel_normalize_rel(ctx, *st["K"], st["Kd"], 1e-2, 0.5)
        for K, G, D in zip(st["K"], st["G"], st["D"]):
            tt.tt_mgrid_project(ctx, st["mg"], K, G)
            tt.tt_mgrid_expand(ctx, st["mg"], G, D)
        tt.tt_model_update(ctx, st["model"], *st["D"], 0.02)
        return {"K": st["K"], "G": st["G"], "D": st["D"], "model": st["model"]}
    n_r, n_d, depth, dmax = _TELE
    it2 = tt.tt_tele2d(ctx, st["s_r"], RE - depth, RE, dmax, RE - st["events"][:, 0], st["T2"],
                       tol=1e-10)
    st["T2f"].copy_(st["T2"])
    tt.tt_tele_region_times(ctx, st["T2f"], RE - depth, RE, dmax, st["events"], st["T"])
    it3 = tt.tt_forward_tele(ctx, st["model"], st["T"], st["opts"])
    return {"T2": st["T2"], "T": st["T"], "iters_2d": it2, "iters": it3}


def work(case):
    """Bytes: each input read once, each output written once. Operations: those of the usual
    number of iterations (40 per Lax-Friedrichs, 120 per Godunov and 30 per adjoint update of
    a node and source); 27 taps x 2,272 channel pairs per node of the network."""
    c = case
    N, B, e = c["nr"] * c["nt"] * c["np"], c["src"], 8 if c["f64"] else 4
    kind = c["kind"]
    model = 3 * e * N
    fwd = 8.0 * N * B * _ITERS.get(c["scheme"], 40) * (120 if c["scheme"] else 40)
    adj = 8.0 * N * B * _ITERS_ADJ * 30
    net = 27 * 2272 * 2.0
    if kind == "forward":
        return {"bytes": model + 2 * e * N * B, "flops": fwd}
    if kind == "adjoint":
        return {"bytes": model + 2 * e * N * B, "flops": adj}
    if kind == "step":
        return {"bytes": model + 3 * e * N * B + 24 * N, "flops": fwd + adj + 12.0 * N * B}
    if kind == "kernel":
        return {"bytes": model + 2 * e * N * B + 24 * N, "flops": 12.0 * N * B}
    if kind == "start":
        Nn = math.prod((c[k] - 2) // 2 + 2 for k in ("nr", "nt", "np"))
        return {"bytes": model + e * N * B, "flops": net * Nn * B}
    if kind == "train":
        return {"bytes": N * B * 4 * 8, "flops": 3 * net * N * B}
    if kind == "descent":
        return {"bytes": 2 * 24 * N + 8 * N + 24 * N + 2 * model, "flops": 3.0 * N * (5 * 11 + 120)}
    n_r, n_d = _TELE[:2]
    return {"bytes": model + e * N * B + 8 * n_r * n_d * B, "flops": 8.0 * N * B * 20 * 40}


# ------------------------------------------------------------- the same in 64 bits, in torch

def _source_values(c, model, src):
    """s, xi, eta interpolated at the sources and the node nearest each source."""
    f = np.stack([(c["nr"] - 1) - src[:, 0] / DR_KM, src[:, 1] / DLL_DEG, src[:, 2] / DLL_DEG], 1)
    n = np.array([c["nr"], c["nt"], c["np"]])
    lo = np.clip(np.floor(f).astype(int), 0, n - 2)
    u = f - lo
    out = np.zeros((3, len(src)))
    for q in range(8):
        d = np.array([q >> 2 & 1, q >> 1 & 1, q & 1])
        w = np.prod(np.where(d, u, 1 - u), 1)
        i, j, k = (lo + d).T
        for a in range(3):
            out[a] += w * model[a][i, j, k].cpu().numpy()
    return out, np.clip(np.floor(f + 0.5).astype(int), 0, n - 1)


def _frames(th, ph):
    """Unit vectors up, north, east, [..., 3 (vector), 3 (xyz)]."""
    ct, st_, cp, sp = torch.cos(th), torch.sin(th), torch.cos(ph), torch.sin(ph)
    ct, st_, cp, sp = torch.broadcast_tensors(ct, st_, cp, sp)
    z = torch.zeros_like(ct)
    return torch.stack([torch.stack([ct * cp, ct * sp, st_], -1),
                        torch.stack([-st_ * cp, -st_ * sp, ct], -1),
                        torch.stack([-sp, cp, z], -1)], -2)


def _factor(c, model, src):
    """T0 and grad T0 (node components) of each source, [nr, nt, np, src], the offset D in the
    source's frame, the fixed set and s at the source."""
    r, th, ph = _axes(c)
    (s0, x0, e0), near = _source_values(c, model, src)
    En = _frames(th[:, None], ph[None, :])
    X = r[:, None, None, None] * En[None, :, :, 0]
    T0, G, Ds, fixed = [], [], [], []
    for b, p in enumerate(src):
        Es = _frames(torch.tensor(p[1] * DEG, dtype=F64, device="cuda"),
                     torch.tensor(p[2] * DEG, dtype=F64, device="cuda"))
        D = (X - (RE - p[0]) * Es[0]) @ Es.T
        M = torch.tensor([[1.0, 0, 0], [0, 1 - 2 * x0[b], 2 * e0[b]], [0, 2 * e0[b], 1 + 2 * x0[b]]],
                         dtype=F64, device="cuda")
        w = D @ torch.linalg.inv(M)
        t0 = s0[b] * torch.sqrt((D * w).sum(-1))
        g = torch.einsum("ijkx,jkax->ijka", w @ Es, En) * (s0[b] ** 2 / t0)[..., None]
        fx = torch.zeros_like(t0, dtype=torch.bool)
        i, j, k = near[b]
        fx[max(i - 1, 0):i + 2, max(j - 1, 0):j + 2, max(k - 1, 0):k + 2] = True
        T0.append(t0)
        G.append(g)
        Ds.append(D)
        fixed.append(fx)
    st = lambda v, a: torch.stack(v, a)
    return st(T0, 3), st(G, 3), st(Ds, 0), st(fixed, 3), s0


def _exact_forward(c, d):
    """The fixed point of the Lax-Friedrichs scheme on tau by Jacobi iterations (T = T0 tau,
    T = T0 on the 3x3x3 nodes of the source, faces max(2 t1 - t2, t2))."""
    s, xi, eta = (t.double()[..., None] for t in d["model"])
    T0, G, _, fixed, _ = _factor(c, [t.double() for t in d["model"]], d["src"])
    r, th, _ = _axes(c)
    r, th = r[:, None, None, None], th[None, :, None, None]
    h = DLL_DEG * DEG
    er = torch.full_like(r, 0.5 / DR_KM)
    et, ep = 0.5 / (h * r), 0.5 / (h * r * torch.cos(th))
    I = (slice(1, -1),) * 3
    inner = lambda t: t.expand(T0.shape)[I]
    er, et, ep, s, xi, eta = (inner(t) for t in (er, et, ep, s, xi, eta))
    t0, g, keep = T0[I], G[I], ~fixed[I]
    ct, cp = torch.sqrt(1 - 2 * xi), torch.sqrt(1 + 2 * xi)
    W = 2 * T0[I] * (er + ct * et + cp * ep)
    tau = torch.ones_like(T0)
    for it in range(40000):
        tc = tau[I]
        dn = [tau[:-2, 1:-1, 1:-1], tau[1:-1, :-2, 1:-1], tau[1:-1, 1:-1, :-2]]
        up = [tau[2:, 1:-1, 1:-1], tau[1:-1, 2:, 1:-1], tau[1:-1, 1:-1, 2:]]
        p = [tc * g[..., a] + t0 * (up[a] - dn[a]) * e for a, e in enumerate((er, et, ep))]
        H = torch.sqrt(p[0] ** 2 + (1 - 2 * xi) * p[1] ** 2 + (1 + 2 * xi) * p[2] ** 2
                       + 4 * eta * p[1] * p[2])
        vis = t0 * (er * (up[0] + dn[0]) + ct * et * (up[1] + dn[1]) + cp * ep * (up[2] + dn[2]))
        v = torch.where(keep, (s - H + vis) / W, tc)
        err = (v - tc).abs().max() if it % 50 == 0 else None
        tau[I] = v
        for a in range(3):
            for f0, f1, f2 in ((0, 1, 2), (-1, -2, -3)):
                t1, t2 = tau.select(a, f1), tau.select(a, f2)
                old, fx = tau.select(a, f0), fixed.select(a, f0)
                old.copy_(torch.where(fx, old, torch.maximum(2 * t1 - t2, t2)))
        if err is not None and float(err) < 1e-13:
            break
    T = torch.where(T0 > 0, T0 * tau, torch.zeros_like(T0))
    return {"tau": tau, "T": T, "iters": None}


def _exact_adjoint(c, d):
    """The upwind finite-volume adjoint by Jacobi iterations: face velocities -(M grad T) with M
    and the cross derivative averaged over a face's nodes, no flux through the outer faces,
    point sources spread to the cell's corners over the node volume, P = 0 around the source."""
    T, R = d["T"].double(), d["R"]
    xi, eta = (t.double()[..., None] for t in d["model"][1:])
    r, th, _ = _axes(c)
    h = DLL_DEG * DEG
    h2, cth = r[:, None, None, None], torch.cos(th)[None, :, None, None]

    def grad(a):     # central, one-sided on the faces, per radian
        n = T.shape[a]
        up = torch.arange(n, device="cuda").add(1).clamp(max=n - 1)
        dn = torch.arange(n, device="cuda").sub(1).clamp(min=0)
        sh = [1] * 4
        sh[a] = n
        return (T.index_select(a, up) - T.index_select(a, dn)) / ((up - dn) * h).view(sh)

    mean = lambda t, a: 0.5 * (t.narrow(a, 0, t.shape[a] - 1) + t.narrow(a, 1, t.shape[a] - 1))
    diff = lambda a: T.narrow(a, 1, T.shape[a] - 1) - T.narrow(a, 0, T.shape[a] - 1)
    rf = (r[:-1] + 0.5 * DR_KM)[:, None, None, None]
    cf = torch.cos(th[:-1] + 0.5 * h)[None, :, None, None]
    flux = [rf ** 2 * cth / DR_KM * -(diff(0) / DR_KM)]
    xh, eh = mean(xi, 1), mean(eta, 1)
    flux.append(h2 * cf / h * -((1 - 2 * xh) * diff(1) / (h * h2) + 2 * eh * mean(grad(2), 1) / (h2 * cf)))
    xh, eh = mean(xi, 2), mean(eta, 2)
    flux.append(h2 / h * -(2 * eh * mean(grad(1), 2) / h2 + (1 + 2 * xh) * diff(2) / (h * h2 * cth)))
    out = torch.zeros_like(T)
    for a in range(3):
        n = T.shape[a] - 1
        out.narrow(a, 0, n).add_(flux[a].clamp(min=0))
        out.narrow(a, 1, n).sub_(flux[a].clamp(max=0))
    S = torch.zeros_like(T)
    n3 = np.array([c["nr"], c["nt"], c["np"]])
    f = np.stack([(c["nr"] - 1) - d["rec"][:, 0] / DR_KM, d["rec"][:, 1] / DLL_DEG,
                  d["rec"][:, 2] / DLL_DEG], 1)
    lo = np.clip(np.floor(f).astype(int), 0, n3 - 2)
    for m in range(len(lo)):
        for q in range(8):
            e = np.array([q >> 2 & 1, q >> 1 & 1, q & 1])
            w = float(np.prod(np.where(e, f[m] - lo[m], 1 - (f[m] - lo[m]))))
            i, j, k = lo[m] + e
            S[i, j, k] += w * R[:, m] / (DR_KM * h * h)
    _, near = _source_values(c, [t.double() for t in d["model"]], d["src"])
    free = torch.ones_like(T, dtype=torch.bool)
    for b, (i, j, k) in enumerate(near):
        free[max(i - 1, 0):i + 2, max(j - 1, 0):j + 2, max(k - 1, 0):k + 2, b] = False
    free &= out > 1e-30
    P = torch.zeros_like(T)
    for it in range(4000):
        s = S.clone()
        for a in range(3):
            n = T.shape[a] - 1
            s.narrow(a, 0, n).sub_(flux[a].clamp(max=0) * P.narrow(a, 1, n))
            s.narrow(a, 1, n).add_(flux[a].clamp(min=0) * P.narrow(a, 0, n))
        v = torch.where(free, s / out, torch.zeros_like(P))
        done = it % 20 == 0 and float((v - P).abs().max()) <= 1e-13 * float(v.abs().max())
        P = v
        if done:
            break
    return {"P": P, "iters": None}


def _exact_kernel(c, d):
    s = d["model"][0].double()
    r, th, _ = _axes(c)
    h = DLL_DEG * DEG
    h2, h3 = r[:, None, None, None], r[:, None, None, None] * torch.cos(th)[None, :, None, None]
    K = [torch.zeros_like(s) for _ in range(3)]
    ends = lambda n: (torch.arange(n, device="cuda").add(1).clamp(max=n - 1),
                      torch.arange(n, device="cuda").sub(1).clamp(min=0))
    for b0 in range(0, c["src"], 16):
        T, P = d["T"][..., b0:b0 + 16].double(), d["P"][..., b0:b0 + 16].double()
        up, dn = ends(c["nt"])
        gt = (T[:, up] - T[:, dn]) / ((up - dn) * h)[None, :, None, None] / h2
        up, dn = ends(c["np"])
        gp = (T[:, :, up] - T[:, :, dn]) / ((up - dn) * h)[None, None, :, None] / h3
        K[0] += s * s * P.sum(-1)
        K[1] += (P * (gt * gt - gp * gp)).sum(-1)
        K[2] += (-2 * P * gt * gp).sum(-1)
    return {"K": K}


def _net(theta, x):
    """The network in double: x [n, D, H, W, 6] -> y [n, D, H, W], taps as matrix products."""
    off = 0
    for l, (ci, co) in enumerate(warmstart.LAYERS):
        w = theta[off:off + 27 * ci * co].view(27, ci, co)
        bias = theta[off + 27 * ci * co:off + 27 * ci * co + co]
        off += 27 * ci * co + co
        D, H, W = x.shape[1:4]
        p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
        y = bias
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            y = y + p[:, dz:dz + D, dy:dy + H, dx:dx + W] @ w[t]
        x = torch.relu(y) if l < 3 else y
    return x[..., 0]


def _features(c, d, b, idx):
    model = [t.double() for t in d["model"]]
    _, _, D, fixed, s0 = _factor(c, model, d["src"][b:b + 1])
    pick = lambda t: t[idx[0]][:, idx[1]][:, :, idx[2]]
    x = torch.stack([pick(model[0]) / s0[0] - 1, pick(model[1]), pick(model[2])], -1)
    return torch.cat([x, pick(D[0]) / 100.0], -1)[None], fixed[..., 0]


def _exact_start(c, d):
    shape = (c["nr"], c["nt"], c["np"])
    idx = [torch.clamp(2 * torch.arange((n - 2) // 2 + 2, device="cuda"), max=n - 1) for n in shape]
    up = []
    for n, ix in zip(shape, idx):
        i = torch.arange(n, device="cuda")
        a = (i // 2).clamp(max=len(ix) - 2)
        f = (i - ix[a]).double() / (ix[a + 1] - ix[a]).double()
        w = torch.zeros((n, len(ix)), dtype=F64, device="cuda")
        w[i, a], w[i, a + 1] = 1 - f, f
        up.append(w)
    tau = torch.empty(shape + (c["src"],), dtype=F64, device="cuda")
    for b in range(c["src"]):
        x, fixed = _features(c, d, b, idx)
        y = _net(d["theta"].double(), x)[0].clamp(-0.5, 1.0)
        y = torch.einsum("ia,jb,kc,abc->ijk", *up, y)
        tau[..., b] = torch.where(fixed, torch.ones_like(y), 1 + y)
    return {"tau": tau}


def _exact_train(c, d):
    idx = [torch.arange(n, device="cuda") for n in (c["nr"], c["nt"], c["np"])]
    theta = d["theta"].double().requires_grad_()
    total, grad = 0.0, torch.zeros_like(theta)
    count = float(d["mask"].double().sum())
    for b in range(c["src"]):
        x, _ = _features(c, d, b, idx)
        e = _net(theta, x) - (d["target"][b:b + 1].double() - 1)
        loss = (d["mask"][b:b + 1].double() * e * e).sum() / count
        grad += torch.autograd.grad(loss, theta)[0]
        total += float(loss)
    return {"loss": total, "grad": grad, "theta": None}


def _exact_descent(c, d):
    nc, H = _MG[0], _MG[3]
    r, th, _ = _axes(c)
    h = DLL_DEG * DEG
    dV = (r[:, None, None] ** 2 * torch.cos(th)[None, :, None] * DR_KM * h * h)
    f = (d["Kd"] + 1e-2 * d["Kd"].max()) ** -0.5
    W = []
    for n in (c["nr"], c["nt"], c["np"]):
        x = torch.arange(n, dtype=F64, device="cuda") / (n - 1) * (nc - 2)
        a = torch.arange(nc, dtype=F64, device="cuda")[None] - \
            torch.arange(H, dtype=F64, device="cuda")[:, None] / H
        W.append((1 - (x[None, None] - a[..., None]).abs()).clamp(min=0))   # [H, nc, n]
    Ks, Gs, Ds, model = [], [], [], []
    for q, K in enumerate(d["K"]):
        K = K * f
        G = torch.stack([torch.einsum("ai,bj,ck,ijk->abc", W[0][g], W[1][g], W[2][g], K * dV)
                         for g in range(H)]) / H
        D = sum(torch.einsum("ai,bj,ck,abc->ijk", W[0][g], W[1][g], W[2][g], G[g])
                for g in range(H)) / H
        m, step = d["model"][q].double(), 0.02 / float(D.abs().max())
        model.append(m * (1 - step * D) if q == 0 else m - step * D)
        Ks.append(K)
        Gs.append(G)
        Ds.append(D)
    return {"K": Ks, "G": Gs, "D": Ds, "model": model}


def exact(case, seed):
    c, kind = case, case["kind"]
    NB = c["nr"] * c["nt"] * c["np"] * c["src"]
    # the solves that an unaccelerated iteration in 64 bits reaches within some seconds
    if kind == "forward" and c["scheme"] == 0 and NB <= 2e5:
        return _exact_forward(c, _inputs(c, seed))
    if kind == "adjoint" and NB <= 4e6:
        return _exact_adjoint(c, _inputs(c, seed))
    if kind == "kernel":
        return _exact_kernel(c, _inputs(c, seed))
    if kind == "start" and NB <= 1.1e8:
        return _exact_start(c, _inputs(c, seed))
    if kind == "train":
        return _exact_train(c, _inputs(c, seed))
    if kind == "descent":
        return _exact_descent(c, _inputs(c, seed))
    return None
