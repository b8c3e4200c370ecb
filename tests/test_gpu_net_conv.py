"""The network's convolutions at sizes and channel counts around their tiles, against the same
network in FP64 torch with the same BF16 weights: training in FP32 (forward, data gradient,
weight gradient) and inference on the tensor cores."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_01701_gb300 import build as B
    B.build()
    import paper_2305_01701_gb300 as P
    return P


def _reference(params, x, t, nd, cin, cout, base, levels):
    import torch
    F = torch.nn.functional
    conv, pool = (F.conv3d, F.avg_pool3d) if nd == 3 else (F.conv2d, F.avg_pool2d)
    leaves, at, terms = [], 0, 0

    def layer(a, ci, co, k):
        nonlocal at, terms
        m = ci * co * k ** nd
        w = params[at:at + m].bfloat16().double().view([co, ci] + [k] * nd).requires_grad_()
        b = params[at + m:at + m + co].double().requires_grad_()
        at += m + co
        terms = max(terms, ci * k ** nd, co * k ** nd)
        leaves.extend([w, b])
        return conv(a, w, b, padding=k // 2)

    skips, a, ci = [], x.double(), cin
    for lv in range(levels):
        o = base << lv
        a = torch.relu(layer(torch.relu(layer(a, ci, o, 3)), o, o, 3))
        ci = o
        if lv < levels - 1:
            skips.append(a)
            a = pool(a, 2)
    for lv in range(levels - 2, -1, -1):
        o = base << lv
        a = torch.cat([F.interpolate(a, scale_factor=2, mode="nearest"), skips[lv]], 1)
        a = torch.relu(layer(torch.relu(layer(a, 3 * o, o, 3)), o, o, 3))
    y = layer(a, base, cout, 1)
    loss = ((y - t.double()) ** 2).mean()
    loss.backward()
    return float(loss.detach()), torch.cat([q.grad.reshape(-1) for q in leaves]), terms


@pytest.mark.parametrize("nd,size,cin,cout,base,levels,N", [
    (2, (5, 3), 1, 1, 1, 1, 1),          # less than a tile of voxels and of channels
    (2, (16, 32), 9, 5, 16, 1, 2),       # exactly one tile
    (2, (20, 36), 9, 5, 16, 2, 3),       # one row and one run beyond it
    (2, (34, 66), 17, 33, 12, 2, 1),     # channels beyond a block of 16 / 32
    (3, (16, 8, 4), 4, 3, 16, 1, 1),
    (3, (17, 9, 5), 13, 9, 33, 1, 2),
    (3, (20, 12, 8), 13, 9, 16, 3, 1),
    (3, (6, 2, 14), 5, 2, 24, 2, 2),
])
def test_training_convolutions_match_fp64(P, nd, size, cin, cout, base, levels, N):
    import torch
    gen = torch.Generator().manual_seed(3)
    net = P.Net(nd, cin, cout, base=base, levels=levels)
    params = 0.1 * torch.randn(net.n_params(), generator=gen)
    net.set_params(params.numpy())
    dims = tuple(reversed(size))
    x = torch.randn((N, cin) + dims, generator=gen).cuda()
    t = torch.randn((N, cout) + dims, generator=gen).cuda()
    loss, g = net.gradients(x.data_ptr(), t.data_ptr(), N, list(size))
    loss2, g2 = net.gradients(x.data_ptr(), t.data_ptr(), N, list(size))
    assert loss == loss2 and np.array_equal(g, g2)      # sums in a fixed order
    ref_loss, ref, terms = _reference(params.cuda(), x, t, nd, cin, cout, base, levels)
    vox = N * int(np.prod(size))
    # FP32 sums of `terms` products per layer and `vox` per weight gradient, each rounding
    # 2^-24: their random growth, through the layers of both passes
    bound = 2.0 ** -24 * (np.sqrt(terms) + np.sqrt(vox)) * (4 * levels + 2)
    assert abs(loss - ref_loss) <= bound * ref_loss
    err = np.linalg.norm(g - ref.cpu().numpy()) / np.linalg.norm(ref.cpu().numpy())
    assert err <= bound, (err, bound)
    net.close()


@pytest.mark.parametrize("nd,size,cin,cout,base,levels,N", [
    (2, (8, 16), 9, 5, 16, 1, 1),         # one brick
    (2, (10, 18), 9, 5, 48, 1, 3),        # beyond it; 16-channel stages
    (2, (12, 36), 40, 17, 32, 3, 2),      # more than 12 head outputs
    (3, (8, 16, 4), 13, 9, 16, 1, 1),
    (3, (72, 68, 20), 13, 9, 16, 2, 1),   # four slabs per block
    (3, (9, 17, 3), 33, 2, 128, 1, 1),    # two slabs, the last one outside; all accumulator columns
    (3, (4, 12, 20), 13, 9, 32, 3, 2),
])
def test_tensor_core_convolutions_at_brick_edges(P, nd, size, cin, cout, base, levels, N):
    """The inference pass (blocked BF16 tensors between the layers, pooling, upsampling and head in
    the convolutions) against FP64 torch with the convolutions' inputs rounded to BF16: what is
    left is FP32 accumulation moving a value across a BF16 rounding boundary (2^-8 relative in a
    few values, carried on through the layers)."""
    import torch
    F = torch.nn.functional
    gen = torch.Generator().manual_seed(4)
    net = P.Net(nd, cin, cout, base=base, levels=levels)
    net.set_output_scale(0.5)
    params = torch.randn(net.n_params(), generator=gen)
    at, spans = 0, []
    for ci, co, k in _layers(nd, cin, cout, base, levels):
        params[at:at + ci * co * k ** nd] *= (2.0 / (ci * k ** nd)) ** 0.5
        params[at + ci * co * k ** nd:at + ci * co * k ** nd + co] *= 0.05
        spans.append((at, ci, co, k))
        at += ci * co * k ** nd + co
    net.set_params(params.numpy())
    dims = tuple(reversed(size))
    x = torch.randn((N, cin) + dims, generator=gen).cuda()
    y = torch.full((N, cout) + dims, float("nan"), device="cuda")
    net.forward(x.data_ptr(), N, list(size), y.data_ptr())
    conv, pool = (F.conv3d, F.avg_pool3d) if nd == 3 else (F.conv2d, F.avg_pool2d)
    p = params.cuda()
    it = iter(spans)

    def layer(a):
        o, ci, co, k = next(it)
        m = ci * co * k ** nd
        w = p[o:o + m].bfloat16().double().view([co, ci] + [k] * nd)
        a = a.float().bfloat16().double() if k == 3 else a
        return conv(a, w, p[o + m:o + m + co].double(), padding=k // 2)

    skips, a = [], x.double()
    for lv in range(levels):
        a = torch.relu(layer(torch.relu(layer(a))))
        if lv < levels - 1:
            skips.append(a)
            a = pool(a, 2)
    for lv in range(levels - 2, -1, -1):
        a = torch.cat([F.interpolate(a, scale_factor=2, mode="nearest"), skips[lv]], 1)
        a = torch.relu(layer(torch.relu(layer(a))))
    ref = 0.5 * layer(a)
    err = (y.double() - ref).abs().max() / ref.abs().max()
    assert torch.isfinite(y).all() and err <= 6e-3, float(err)
    net.close()


def _layers(nd, cin, cout, base, levels):
    out, c = [], cin
    for lv in range(levels):
        out += [(c, base << lv, 3), (base << lv, base << lv, 3)]
        c = base << lv
    for lv in range(levels - 2, -1, -1):
        out += [(3 * (base << lv), base << lv, 3), (base << lv, base << lv, 3)]
    return out + [(base, cout, 1)]


@pytest.mark.parametrize("call", ["gradients", "train_step", "forward"])
def test_a_shape_that_does_not_fit_fails_each_time_and_leaves_the_network_usable(P, call):
    """A batch whose first tensor is far beyond the device's memory: refused, refused again, and
    the next shape that fits gives what an untouched network gives.  The inputs are never read."""
    import torch
    gen = torch.Generator().manual_seed(5)
    nets = [P.Net(2, 9, 5, base=16, levels=2) for _ in range(2)]
    params = 0.1 * torch.randn(nets[0].n_params(), generator=gen)
    x = torch.randn((1, 9, 16, 16), generator=gen).cuda()
    t = torch.randn((1, 5, 16, 16), generator=gen).cuda()
    torch.cuda.synchronize()
    for n in nets:
        n.set_params(params.numpy())

    def run(net, N, size):
        if call == "forward":
            y = torch.empty((1, 5, 16, 16), device="cuda")
            net.forward(x.data_ptr(), N, size, y.data_ptr())
            return y.cpu().numpy()
        if call == "gradients":
            return net.gradients(x.data_ptr(), t.data_ptr(), N, size)[1]
        net.train_step(x.data_ptr(), t.data_ptr(), N, size, 1e-3)
        return net.get_params()

    for _ in range(2):
        with pytest.raises(P.EPError, match="out of memory"):
            run(nets[0], 60000, [2048, 2048])
    np.testing.assert_array_equal(run(nets[0], 1, [16, 16]), run(nets[1], 1, [16, 16]))
    for n in nets:
        n.close()


@pytest.mark.parametrize("nd,size,N", [(2, (64, 64), 8), (2, (256, 128), 2), (3, (32, 32, 16), 2)])
def test_partial_sums_of_a_gradient_add_without_their_roundings(P, nd, size, N):
    """The head's bias gradient of a zero head is -2 / n times the sum of the targets: with n a
    power of two its terms are exact in FP32.  A block's threads add runs of 16 to 64 of them
    (random roundings, averaged over hundreds of runs), and the hundreds of partial sums add
    without theirs: the result is within 2^-23, one rounding and as much again."""
    import torch
    worst = 0.0
    for seed in range(6):
        gen = torch.Generator().manual_seed(seed)
        net = P.Net(nd, 3, 4, base=16, levels=1)
        params = net.get_params().copy()
        params[-4 - 4 * 16:] = 0.0
        net.set_params(params)
        dims = tuple(reversed(size))
        x = torch.randn((N, 3) + dims, generator=gen).cuda()
        t = (torch.rand((N, 4) + dims, generator=gen) + 0.1).cuda()
        torch.cuda.synchronize()
        g = net.gradients(x.data_ptr(), t.data_ptr(), N, list(size))[1][-4:]
        n = t.numel()
        assert n & (n - 1) == 0
        want = (-2.0 / n * t.double().transpose(0, 1).reshape(4, -1).sum(1)).cpu().numpy()
        worst = max(worst, np.abs(g / want - 1.0).max())
        net.close()
    assert worst <= 2.0 ** -23, worst * 2.0 ** 23
