"""The tensor-core convolutions walk windows of rows along the radius: against 64-bit convolutions of
the BF16-rounded operands, at one and two windows of a plane, the smallest grid, walks of one
plane and of all, and more walks than blocks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [((4, 4, 4), 1), ((4, 6, 17), 1), ((5, 6, 18), 3), ((41, 8, 13), 1), ((6, 8, 13), 170),
          ((7, 41, 39), 9), ((33, 20, 21), 40)]


def _setup(tt, shape, n):
    import torch
    g = dict(n_r=shape[0], n_t=shape[1], n_p=shape[2], depth_min_km=0.0, depth_max_km=10.0, lat_min_deg=0.0,
             lat_max_deg=0.5, lon_min_deg=0.0, lon_max_deg=0.5, earth_radius_km=6371.0, flat=0)
    from paper_2412_00031_gb300 import warmstart
    theta = torch.as_tensor(warmstart.init_params(sum(shape)), device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(n + shape[0])
    x = torch.randn((n,) + shape + (tt.NET_FEATURES,), device="cuda", generator=gen)
    return tt.tt_ctx_create(g), theta, x, gen


@pytest.mark.parametrize("shape,n", SHAPES)
def test_inference_matches_64_bit_convolutions(shape, n):
    """Operands and sums are alike but for the order of FP32 sums, which can turn the rounding of a
    layer's BF16 outputs here and there: one unit (2^-8) of the largest value in each of three layers."""
    import torch
    import paper_2412_00031_gb300 as tt
    ctx, theta, x, _ = _setup(tt, shape, n)
    tt.tt_net_set_weights(ctx, theta)
    y = torch.empty((n,) + shape, device="cuda")
    tt.tt_net_infer(ctx, x, y)
    bf = lambda t: t.to(torch.bfloat16).double().cpu()
    h, k = bf(x).movedim(-1, 1), 0
    for l, (ci, co) in enumerate(((6, 32), (32, 32), (32, 32), (32, 1))):
        w = bf(theta[k:k + 27 * ci * co]).view(3, 3, 3, ci, co).permute(4, 3, 0, 1, 2)
        b = bf(theta[k + 27 * ci * co:k + 27 * ci * co + co])
        k += 27 * ci * co + co
        h = torch.nn.functional.conv3d(h, w, b, padding=1)
        if l < 3:
            h = bf(h.clamp(min=0).float())
    err, top = (y.cpu().double() - h[:, 0]).abs().max().item(), h.abs().max().item()
    ctx.close()
    assert err <= 3 * 2.0 ** -8 * top


@pytest.mark.parametrize("shape,n", SHAPES)
def test_training_gradient_matches_the_fp32_path(shape, n):
    """Every entry of the gradient against the FP32 kernels, where all of a network's values are positive:
    the gates stay open and no sum cancels, so an entry is off by its BF16 roundings alone, of 2^-9 each:
    eight of y, one of dL/dy, three weights and three gradients on the way down, and the input row.
    The loss takes y's twice."""
    import torch
    import paper_2412_00031_gb300 as tt
    ctx, theta, x, gen = _setup(tt, shape, n)
    theta, x = theta.abs(), x.abs()
    target = torch.zeros((n,) + shape, device="cuda")
    mask = (torch.rand((n,) + shape, device="cuda", generator=gen) > 0.2).float()
    g, ref = torch.empty_like(theta), torch.empty_like(theta)
    loss = tt.tt_net_loss_grad_tc(ctx, theta, x, target, mask, g)
    want = tt.tt_net_loss_grad(ctx, theta, x, target, mask, ref)
    ctx.close()
    assert abs(loss / want - 1) <= 16 * 2.0 ** -9
    assert ((g - ref).abs() <= 16 * 2.0 ** -9 * ref).all()


@pytest.mark.parametrize("shape,n", [((4, 5, 4), 1), ((5, 4, 66), 33), ((6, 7, 68), 40), ((9, 8, 131), 3)])
def test_coarse_prediction_is_interpolated(shape, n):
    """The warm start from every other node (33 and 65 cells along phi, 33 and more sources, odd and even
    extents) against the network's own prediction, clamped and interpolated in 64 bits: eight products and
    sums of values up to 1 in FP32, and 1 + v."""
    import torch
    import paper_2412_00031_gb300 as tt
    ctx, theta, _, _ = _setup(tt, shape, n)
    rng = np.random.default_rng(n)
    src = rng.uniform(0.1, 0.9, (n, 3)) * np.array([10.0, 0.5, 0.5])
    model = [torch.full(shape, v, device="cuda") for v in (0.2, 0.01, -0.01)]
    tt.tt_net_set_stride(ctx, 2)
    tt.tt_net_set_weights(ctx, theta)
    net = tuple(s // 2 + 1 for s in shape)
    x = torch.empty((n, int(np.prod(net)), tt.NET_FEATURES), device="cuda")
    tt.tt_net_features(ctx, model, src, x)
    y = torch.empty((n, int(np.prod(net))), device="cuda")
    tt.tt_net_infer(ctx, x, y)
    tau = torch.empty(shape + (n,), device="cuda")
    tt.tt_net_start(ctx, model, src, tau)
    ctx.close()
    v = y.double().cpu().numpy().reshape((n,) + net).clip(-0.5, 1.0)
    for axis, s in enumerate(shape):
        at = np.minimum(2 * np.arange(net[axis]), s - 1)
        a = np.minimum(np.arange(s) // 2, net[axis] - 2)
        f = (np.arange(s) - at[a]) / (at[a + 1] - at[a])
        f = f.reshape([-1 if k == axis + 1 else 1 for k in range(4)])
        v = (1 - f) * v.take(a, axis + 1) + f * v.take(a + 1, axis + 1)
    # the nodes around a source are fixed at 1
    pos = np.stack([(10.0 - src[:, 0]) / 10.0, src[:, 1] / 0.5, src[:, 2] / 0.5], 1) * (np.array(shape) - 1)
    near = np.floor(pos + 0.5).astype(int)
    err = np.abs(tau.cpu().numpy() - 1 - np.moveaxis(v, 0, 3))
    for b in range(n):
        err[tuple(slice(max(c - 1, 0), c + 2) for c in near[b]) + (b,)] = 0
    assert err.max() <= 24 * 2.0 ** -24
