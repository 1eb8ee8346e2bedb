"""GPU parity of the learned warm start network (BF16 kernels, FP32
accumulation) against the FP64 network oracle, through the C ABI.

The oracle is fed the BF16-rounded weights and inputs, so the remaining
difference is the BF16 rounding of activations and gradients inside the
network: about 2^-9 relative per stored value, accumulated over 21 layers.
Bars (relative L2): output <= 2e-2, loss <= 1e-2, each layer's weight and
bias gradient <= 5e-2.  A wrong tap, transposed weight, missing bias or a
skip connection in the wrong place gives errors of order 1.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

from oracle import unet_oracle as U
from paper_2601_00822_gb300 import _lib, api, workloads as W

pytestmark = pytest.mark.gpu

DIMS = (24, 16, 16)   # (nx, ny, nz); coarsest level 3 x 2 x 2; untiled convolutions only
# (32, 16, 16): levels 0 and 1 run the shared-memory tiled convolution (16 x 8 x 2 tiles)
GRIDS = [DIMS, (32, 16, 16)]


def rel(a, b):
    a = np.asarray(a, dtype=np.float64).ravel()
    b = np.asarray(b, dtype=np.float64).ravel()
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def bf16(t):
    return torch.as_tensor(t).to(torch.bfloat16).to(torch.float64)


def params(seed):
    """He-initialised weights with small random biases (so every bias path is exercised)."""
    flat = U.init_params(seed)
    g = torch.Generator().manual_seed(seed + 100)
    for name, (w, b) in U.unpack(flat).items():
        b.copy_((torch.rand(b.shape, generator=g, dtype=torch.float64) - 0.5) * 0.2)
    return flat


def inputs(seed, batch, dims=DIMS, ch=4):
    g = torch.Generator().manual_seed(seed)
    nx, ny, nz = dims
    return torch.rand((batch, ch, nz, ny, nx), generator=g, dtype=torch.float64) * 2 - 1


def layer_slices():
    i = 0
    for name, kind, cin, cout in U.LAYERS:
        w = int(np.prod(U.weight_shape(kind, cin, cout)))
        yield name, slice(i, i + w), slice(i + w, i + w + cout)
        i += w + cout


@pytest.mark.parametrize("dims", GRIDS)
def test_forward_matches_oracle(dims):
    flat = params(3)
    x = inputs(5, 2, dims)
    net = api.Net(dims, max_batch=2)
    y = net.forward(flat.float().cuda(), x.float().cuda()).double().cpu()
    net.status()
    ref = U.forward(bf16(flat), bf16(x))
    for s in range(2):
        assert rel(y[s], ref[s]) <= 2e-2, (s, rel(y[s], ref[s]))


def test_forward_full_training_size_matches_oracle():
    dims = (64, 64, 64)
    flat = params(4)
    x = inputs(6, 1, dims)
    net = api.Net(dims, max_batch=1)
    y = net.forward(flat.float().cuda(), x.float().cuda()).double().cpu()
    net.status()
    assert rel(y, U.forward(bf16(flat), bf16(x))) <= 2e-2


@pytest.mark.parametrize("dims", GRIDS)
def test_gradients_match_oracle(dims):
    flat = params(7)
    x = inputs(8, 2, dims)
    t = inputs(9, 2, dims, ch=6)
    net = api.Net(dims, max_batch=2, train=True)
    g, loss = net.grad(flat.float().cuda(), x.float().cuda(), t.float().cuda())
    g = g.double().cpu()
    p = bf16(flat).requires_grad_(True)
    lo = U.loss(U.forward(p, bf16(x)), t.float().double())
    gref, = torch.autograd.grad(lo, p)
    lo = float(lo.detach())
    assert abs(float(loss.item()) - lo) <= 1e-2 * lo
    for name, ws, bs in layer_slices():
        assert rel(g[ws], gref[ws]) <= 5e-2, (name, "weight", rel(g[ws], gref[ws]))
        assert rel(g[bs], gref[bs]) <= 5e-2, (name, "bias", rel(g[bs], gref[bs]))


def test_gradient_is_deterministic():
    flat = params(10).float().cuda()
    x = inputs(11, 2).float().cuda()
    t = inputs(12, 2, ch=6).float().cuda()
    net = api.Net(DIMS, max_batch=2, train=True)
    g1, l1 = net.grad(flat, x, t)
    g1 = g1.clone()
    g2, l2 = net.grad(flat, x, t)
    assert torch.equal(g1, g2) and torch.equal(l1, l2)


def test_adam_matches_oracle():
    gen = torch.Generator().manual_seed(13)
    n = _lib.NET_PARAMS
    w, g, m = (torch.randn(n, generator=gen, dtype=torch.float64) for _ in range(3))
    v = torch.rand(n, generator=gen, dtype=torch.float64)
    w, g, m, v = (a.float().double() for a in (w, g, m, v))
    dev = [a.float().cuda() for a in (w, g, m, v)]
    net = api.Net((8, 8, 8))
    net.adam(dev[0], dev[1], dev[2], dev[3], 3, 1e-3)
    U.adam_step(w, g, m, v, 3, lr=1e-3)
    assert rel(dev[0].cpu(), w) <= 1e-6
    assert rel(dev[2].cpu(), m) <= 1e-6 and rel(dev[3].cpu(), v) <= 1e-6


def test_training_steps_reduce_the_loss():
    flat = params(14).float().cuda()
    xc = inputs(15, 2)
    x = xc.float().cuda()
    t = U.forward(params(16), xc).float().cuda()     # a target the network can represent
    net = api.Net(DIMS, max_batch=2, train=True)
    grad = torch.empty_like(flat)
    m = torch.zeros_like(flat)
    v = torch.zeros_like(flat)
    losses = [float(net.train_step(flat, grad, m, v, k, 1e-3, x, t).item()) for k in range(1, 31)]
    assert np.isfinite(losses).all() and losses[-1] < 0.8 * losses[0], losses


def test_prepare_predict_and_surrogate_match_oracle_features():
    p = W.config_c5_sample(3, n=32)
    phases = [tuple(q) for q in p.phases]
    mus = [q[1] for q in phases]
    ph = api.voxelize(p.dims, p.cell, p.spheres)
    b = api.body_force(p.dims, p.bf_centre, p.bf_radius, "fp64")
    eps = torch.randn((6,) + tuple(b.shape[1:]), dtype=torch.float64, device="cuda")
    net = api.Net(p.dims, max_batch=2)
    x, tgt = net.prepare(b, ph, phases, eps=eps)
    xr, s = U.features(b.cpu(), ph.cpu(), mus)
    assert rel(x.cpu(), xr) <= 1e-6
    assert rel(tgt.cpu(), U.targets(eps.cpu(), b.cpu(), mus)) <= 1e-6
    flat = params(17)
    fl = flat.float().cuda()
    pred = net.predict(fl, [b, b], [ph, ph], phases)
    y = net.forward(fl, x[None])
    want = y[0].double() * (s / max(mus))
    assert rel(pred[0].cpu(), want.cpu()) <= 1e-6 and torch.equal(pred[0], pred[1])
    assert rel(pred[0].cpu(), U.forward(bf16(flat), bf16(xr[None]))[0] * (s / max(mus))) <= 2e-2
    with api.Plan(p.dims, "mixed") as plan:
        sur = plan.surrogate_infer(fl, b, ph, phases)
    assert torch.equal(sur, pred[0])


def test_trained_warm_start_reduces_sweeps_and_matches_cold_solver():
    """The committed trained network, on held-out 64^3 samples (seeds 0..7; the
    training seeds start at 1000000): its prediction is within 35% relative L2 of
    the solution, the warm-started batched ladder needs fewer FP32 sweeps than
    the cold one, and both land within the tolerance of each other (the cold
    solver is the reference)."""
    from paper_2601_00822_gb300 import surrogate as S
    params = S.load(S.DEFAULT_WEIGHTS)
    res = S.warm_start_benchmark(params, list(range(8)), 64, tol=1e-6, batch=8, plain=False)
    assert res["prediction_rel_l2_mean"] < 0.35, res
    assert res["batched_warm"]["mean_sweeps"] < res["batched_cold"]["mean_sweeps"], res
    assert res["batched_warm"]["max_resid"] <= 1e-6 and res["batched_cold"]["max_resid"] <= 1e-6
    assert res["warm_vs_cold_eps_rel_l2_max"] < 1e-5, res


@pytest.mark.parametrize("dims,batch", [((8, 8, 8), 1), ((40, 24, 16), 2), ((16, 8, 72), 3), ((24, 56, 8), 1),
                                        ((64, 48, 64), 5)])
def test_tensor_core_convolutions_equal_the_warp_level_ones(dims, batch, monkeypatch):
    """Both forms of a convolution sum each output's products in the same order (taps, then
    blocks of 16 channels, FP32 accumulators), so partial tiles, tiles that cross a column of
    planes, blocks with one tile and blocks with many must reproduce the plain kernels bit for
    bit: outputs and loss.  Weight and bias gradients add the same terms in another order: FP32 sums of up to 10^6 terms of either sign,
    2^-24 a step growing as its square root against a sum that does too, a few 1e-7; 1e-5."""
    flat = params(21).float().cuda()
    x = inputs(22, batch, dims).float().cuda()
    t = inputs(23, batch, dims, ch=6).float().cuda()
    net = api.Net(dims, max_batch=batch, train=True)
    out = []
    for on in ("1", "0"):
        monkeypatch.setenv("BFCS_NET_TCGEN05", on)
        g, loss = net.grad(flat, x, t)
        out.append((net.forward(flat, x).clone(), g.clone(), loss.clone()))
    net.status()
    (y1, g1, l1), (y0, g0, l0) = out
    assert torch.equal(y1, y0) and torch.equal(l1, l0)
    for name, ws, bs in layer_slices():
        assert rel(g1[ws].cpu(), g0[ws].cpu()) <= 1e-5, name
        assert rel(g1[bs].cpu(), g0[bs].cpu()) <= 1e-5, name


@pytest.mark.parametrize("scale", [1.0, 1e-14, 1e-20, 1e18])
def test_loss_and_its_gradient_over_the_range_of_the_fields(scale):
    """The loss of the network's own output, written out in FP64, for targets and outputs
    far below and above 1 (squares outside the FP32 range); the head's bias gradient is the
    sum of the loss gradient over the voxels."""
    dims = (24, 8, 16)
    flat = params(31).float()
    wslice, bslice = list(layer_slices())[-1][1:]
    flat[wslice] *= scale
    flat[bslice] *= scale
    flat = flat.cuda()
    x = inputs(32, 2, dims).float().cuda()
    t = (scale * inputs(33, 2, dims, ch=6)).float().cuda()
    t[:, 3] = 0.0
    net = api.Net(dims, max_batch=2, train=True)
    y = net.forward(flat, x).double()
    g, loss = net.grad(flat, x, t)
    d = y - t.double()
    den = (t.double() ** 2).sum((1, 2, 3, 4))
    want = ((d ** 2).sum((1, 2, 3, 4)) / den).mean()
    assert abs(float(loss) - float(want)) <= 1e-12 * float(want)
    db = (2.0 * d / (2 * den.view(-1, 1, 1, 1, 1))).sum((0, 2, 3, 4))
    assert rel(g[bslice].double().cpu(), db.cpu()) <= 1e-2     # BF16 terms, 2^-9 each


@pytest.mark.parametrize("dims,batch", [((8, 8, 8), 1), ((32, 16, 24), 3)])
def test_captured_passes_equal_the_direct_ones(dims, batch):
    """Forward pass, strain prediction and gradient recorded in a CUDA graph and replayed
    with other parameters and inputs: the chained launches keep their order, and the
    layers' early parameter loads see the values of the replay."""
    r = np.random.default_rng(41)
    flat = params(42).float().cuda()
    x = inputs(43, batch, dims).float().cuda()
    t = inputs(44, batch, dims, ch=6).float().cuda()
    b = [torch.tensor(r.standard_normal((3,) + dims[::-1]), dtype=torch.float32, device="cuda") for _ in range(batch)]
    ph = [torch.tensor(r.integers(0, 2, dims[::-1]), dtype=torch.int8, device="cuda") for _ in range(batch)]
    phases = [(1.0, 0.5), (0.3, 2.0)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        net = api.Net(dims, max_batch=batch, train=True, stream=side)

        def passes():
            y = net.forward(flat, x)
            p = net.predict(flat, b, ph, phases)
            g, loss = net.grad(flat, x, t)
            return [y, *p, g, loss]

        passes()
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            got = passes()
        for k in range(3):
            flat.copy_(params(45 + k).float())
            x.copy_(inputs(48 + k, batch, dims).float())
            b[0].copy_(torch.tensor(r.standard_normal(b[0].shape), dtype=torch.float32))
            graph.replay()
            replayed = [v.clone() for v in got]
            want = passes()
            assert all(torch.equal(u, v) for u, v in zip(replayed, want))
        net.status()
        side.synchronize()


def constant_output(bias):
    """Parameters whose output is `bias` at every voxel (FP32, exactly): zero head weights."""
    flat = params(51).float()
    ws, bs = list(layer_slices())[-1][1:]
    flat[ws] = 0.0
    flat[bs] = torch.tensor(bias, dtype=torch.float32)
    return flat.cuda()


@pytest.mark.parametrize("n,roundings", [(8, 13), (64, 43)])
def test_the_loss_is_summed_to_fp64(n, roundings):
    """Constant output and target: every voxel has the same terms, so that what is lost on
    one of them is lost on all, and the sums over voxels are multiples of one number.  Each
    of the two sums rounds a voxel (2), k v for k up to the voxels of a thread (15 at 64^3)
    and for 3, 5, 6, 7 warps; then the quotient: 2 (2 + 4) + 1 or 2 (2 + 15 + 4) + 1 roundings
    of 2^-53.  The values are such that sums of 48 bits miss by 1.6e-14."""
    p = [float.fromhex(v) for v in ("-0x1.5bd8e8p+0", "0x1.094478p+1", "0x1.78f4p+0", "-0x1.581092p-2",
                                    "-0x1.85381ap-1", "0x1.1108bcp+0")]
    q = [float.fromhex(v) for v in ("0x1.18d16ep-2", "-0x1.afdb24p-2", "0x1.c6bcb6p-10", "0x1.081ab6p-10",
                                    "0x1.8f6894p-8", "-0x1.79607p-11")]
    net = api.Net((n, n, n), max_batch=1, train=True)
    t = torch.tensor(q, dtype=torch.float32, device="cuda").view(1, 6, 1, 1, 1).expand(1, 6, n, n, n).contiguous()
    _, loss = net.grad(constant_output(p), inputs(52, 1, (n, n, n)).float().cuda(), t)
    want = sum((Fraction(a) - Fraction(b)) ** 2 for a, b in zip(p, q)) / sum(Fraction(b) ** 2 for b in q)
    assert abs(Fraction(float(loss)) - want) <= roundings * Fraction(1, 2 ** 53) * want


def test_the_loss_gradient_rounds_as_fp64_does():
    """The loss gradient (p - t) 2 / den is rounded to FP32 and then to BF16.  Here the
    product lies between a tie of two BF16 values and the next float, 2^-46 from where FP32
    decides between them: 48 bits give the other neighbour.  512 voxels with the same value:
    den and the head's bias gradient, 512 times the value, are exact."""
    p, q = float.fromhex("0x1.429116p+7"), float.fromhex("0x1.23aaap-1")
    net = api.Net((8, 8, 8), max_batch=1, train=True)
    t = torch.zeros((1, 6, 8, 8, 8), device="cuda")
    t[:, 5] = q
    g, _ = net.grad(constant_output([p, 0.0, 0.0, 0.0, 0.0, q]), inputs(53, 1, (8, 8, 8)).float().cuda(), t)
    want = torch.tensor(p * (2.0 / (512.0 * q * q)), dtype=torch.float64).float().to(torch.bfloat16).double()
    bias = g[list(layer_slices())[-1][2]].double().cpu()
    assert float(bias[0]) == 512.0 * float(want), (float(bias[0]) / 512.0, float(want))
    assert torch.equal(bias[1:], torch.zeros(5, dtype=torch.float64))


@pytest.mark.parametrize("s,y", [("0x1.d16d7p-1", "0x1.98p+0"), ("0x1.8p+0", "-0x1.fffffep+3"), ("0x1.4p-30", "0x1.23456p-60"),
                                 ("0x1.4p+20", "0x1.23456p-60")])
def test_the_fp32_prediction_rounds_as_fp64_does(s, y):
    """Predicted strain y s / mu_max, one FP64 product rounded to FP32.  The first
    product lies 2^-47 from where FP32 decides between two values."""
    s, y = float.fromhex(s), float.fromhex(y)
    net = api.Net((8, 8, 8), max_batch=1)
    b = torch.zeros((3, 8, 8, 8), device="cuda")
    b[1, 2, 3, 4], b[1, 5, 3, 4] = s, -s
    ph = torch.zeros((8, 8, 8), dtype=torch.int8, device="cuda")
    got = net.predict(constant_output([y, -y, 0.5, y, y, y]), [b], [ph], [(1.0, 3.0)])[0].cpu()
    want = torch.tensor([v * (s / 3.0) for v in (y, -y, 0.5, y, y, y)], dtype=torch.float64).float()
    assert torch.equal(got.view(torch.int32), want.view(6, 1, 1, 1).expand(6, 8, 8, 8).contiguous().view(torch.int32))


def layer_spans():
    return {name: (ws, bs) for name, ws, bs in layer_slices()}


def set_identity(flat, name, cin, cout=32, first=0):
    """Layer `name` passes its input channels first .. first + cout - 1 through unchanged: the
    centre tap of a 3^3 layer, every sub-voxel of an up-convolution, the six rows of the head."""
    ws, bs = layer_spans()[name]
    w = torch.zeros_like(flat[ws])
    if name.startswith("u"):
        w.view(cin, cout, 8)[first:first + cout][torch.arange(cout), torch.arange(cout)] = 1.0
    elif name == "head":
        w.view(6, 32)[torch.arange(min(6, 32 - first)), first + torch.arange(min(6, 32 - first))] = 1.0
    else:
        w.view(cout, cin, 27)[torch.arange(cout), first + torch.arange(cout), 13] = 1.0
    flat[ws] = w
    flat[bs] = 0.0


def pass_through_from(flat, level):
    """Everything after the up-convolution of `level` hands its output on: the decoder's
    convolutions and the finer up-convolutions are identities (for positive values)."""
    for k in range(level, -1, -1):
        set_identity(flat, f"d{k}a", 64)
        set_identity(flat, f"d{k}b", 32)
        if k > 0:
            set_identity(flat, f"u{k - 1}", 32)


def read_channels(net, flat, x, level):
    """The 32 channels that reach the head, at the resolution of `level` (replicated above it)."""
    out = []
    for first in range(0, 32, 6):
        f = flat.clone()
        set_identity(f, "head", 32, first=first)
        y = net.forward(f.cuda(), x).double().cpu()
        out.append(y[:, :min(6, 32 - first)])
    s = 2 ** level
    y = torch.cat(out, 1)
    return y[:, :, ::s, ::s, ::s]


@pytest.mark.parametrize("dims,batch", [((8, 8, 8), 1), ((24, 16, 8), 3), ((40, 8, 24), 2)])
@pytest.mark.parametrize("level", [2, 1, 0])
def test_pointwise_layers_against_fp64_sums(dims, batch, level):
    """The up-convolutions and the head against FP64 sums of the BF16 operands that they get
    (rows in numbers that are no multiples of a warp's 32 or a block's 256 at levels 2 and 1).
    With identities after the up-convolution of `level` the output shows what it writes, and
    with an identity in its place what it reads.  Values stay positive, so that no activation
    or its derivative changes them.  Forward: rounded to BF16 from an FP32 sum of up to 48
    products within 1e-5.  Weight and bias gradients: FP32 sums of BF16 products, 1e-5.  The gradient it hands down, rounded to
    BF16 (a few values the other way), through the bias gradient of the layer below: 1e-3."""
    cin = 48 if level == 2 else 32
    below = {2: "e3b", 1: "d2b", 0: "d1b"}[level]
    g = torch.Generator().manual_seed(60 + level)
    flat = params(61).float()
    ws, bs = layer_spans()[f"u{level}"]
    pass_through_from(flat, level)
    flat[layer_spans()[below][1]] += 8.0
    w = (torch.rand(cin, 32, 8, generator=g) * 0.1 - 0.05).float()
    bias = 40.0 + torch.rand(32, generator=g)
    x = inputs(62, batch, dims).float().cuda()
    t = (40.0 + 4.0 * inputs(63, batch, dims, ch=6)).float()
    net = api.Net(dims, max_batch=batch, train=True)
    # what the layer reads, 32 channels at a time
    got_in = []
    for first in range(0, cin, 16 if cin == 48 else 32):
        if first + 32 > cin:
            break
        f = flat.clone()
        set_identity(f, f"u{level}", cin, first=first)
        got_in.append(read_channels(net, f, x, level + 1))
    u = got_in[0] if cin == 32 else torch.cat([got_in[0], got_in[1][:, 16:]], 1)
    assert (u > 0).all()
    # what it writes
    flat[ws] = w.reshape(-1)
    flat[bs] = bias
    wb = bf16(w)
    nz, ny, nx = u.shape[2:]

    def spread(v):                                   # (b, 32, 8, z, y, x) -> fine grid
        return v.view(batch, 32, 2, 2, 2, nz, ny, nx).permute(0, 1, 5, 2, 6, 3, 7, 4).reshape(batch, 32, 2 * nz, 2 * ny, 2 * nx)

    want = spread(torch.einsum("bizyx,ico->bcozyx", u, wb) + bias.double().view(1, 32, 1, 1, 1, 1))
    got = read_channels(net, flat, x, level)
    assert ((bf16(want * (1 - 1e-5)) <= got) & (got <= bf16(want * (1 + 1e-5)))).all()
    # the head with weights of its own, on what reaches it
    fine = got
    for _ in range(level):
        fine = fine.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
    f = flat.clone()
    hw = (torch.rand(6, 32, generator=g) - 0.5).float()
    f[layer_spans()["head"][0]] = hw.reshape(-1)
    y = net.forward(f.cuda(), x).double().cpu()
    want = torch.einsum("bczyx,hc->bhzyx", fine, bf16(hw)) + f[layer_spans()["head"][1]].double().view(1, 6, 1, 1, 1)
    assert ((y - want).abs() <= 1e-5 * torch.einsum("bczyx,hc->bhzyx", fine, bf16(hw).abs())).all()
    # gradients with the head on six of the channels
    set_identity(f, "head", 32, first=13)
    y = net.forward(f.cuda(), x).double().cpu()
    grad, _ = net.grad(f.cuda(), x, t.cuda())
    grad = grad.double().cpu()
    d = y - t.double()
    den = (t.double() ** 2).sum((1, 2, 3, 4)).view(-1, 1, 1, 1, 1)
    dout = bf16((d * (2.0 / (den * batch))).float())
    assert rel(grad[layer_spans()["head"][1]], dout.sum((0, 2, 3, 4))) <= 1e-5
    assert rel(grad[layer_spans()["head"][0]], torch.einsum("bhzyx,bczyx->hc", dout, fine)) <= 1e-5
    dy = torch.zeros_like(fine)
    dy[:, 13:19] = dout
    for _ in range(level):                           # the identity up-convolutions add their eight sub-voxels
        b_, c_, z_, y_, x_ = dy.shape
        dy = bf16(dy.view(b_, c_, z_ // 2, 2, y_ // 2, 2, x_ // 2, 2).sum((3, 5, 7)).float())
    dyo = dy.view(batch, 32, nz, 2, ny, 2, nx, 2).permute(0, 1, 3, 5, 7, 2, 4, 6).reshape(batch, 32, 8, nz, ny, nx)
    assert rel(grad[bs], dy.sum((0, 2, 3, 4))) <= 1e-5
    assert rel(grad[ws], torch.einsum("bcozyx,bizyx->ico", dyo, u)) <= 1e-5
    du = bf16(torch.einsum("bcozyx,ico->bizyx", dyo, wb).float())
    assert rel(grad[layer_spans()[below][1]], du.sum((0, 2, 3, 4))) <= 1e-3
    net.status()


def test_batches_beyond_one_launch_of_pointers():
    """More samples than travel in one launch's arguments (64), and predictions of more
    samples than the context holds: equal to smaller batches bit for bit."""
    dims, n = (8, 8, 8), 70
    r = np.random.default_rng(71)
    flat = params(72).float().cuda()
    x = inputs(73, n, dims).float().cuda()
    b = [torch.tensor(r.standard_normal((3, 8, 8, 8)), dtype=torch.float32, device="cuda") for _ in range(n)]
    ph = [torch.tensor(r.integers(0, 2, (8, 8, 8)), dtype=torch.int8, device="cuda") for _ in range(n)]
    phases = [(1.0, 0.5), (0.3, 2.0)]
    big, small = api.Net(dims, max_batch=n), api.Net(dims, max_batch=9)
    want = torch.cat([small.forward(flat, x[i:i + 9]) for i in range(0, n, 9)])
    assert torch.equal(big.forward(flat, x), want)
    alone = [small.predict(flat, [bi], [pi], phases)[0].clone() for bi, pi in zip(b, ph)]
    for net in (big, small):
        assert all(torch.equal(p, a) for p, a in zip(net.predict(flat, b, ph, phases), alone))
        net.status()
