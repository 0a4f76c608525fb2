"""The network's gradients layer by layer, and its sums and special values.

test_layers_at_tile_edges: weights whose taps add up to zero and large positive
biases leave every ReLU open, so no decision hangs on a BF16 rounding, and the
gradient of each layer's weights and biases is compared on its own.  Tolerance 5e-3
(relative, 2-norm): activations and weights are BF16 on both sides, and stored values
can differ by one unit, 2^-8, where the FP32 sums straddle a rounding (few do: the
reference with FP32 sums moves by 2e-3 at most).  Two taps exchanged move the least
sensitive layer by 8e-3, the others by 6e-2 or more.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from oracle import guessnet as G  # noqa: E402
from test_gpu_guessnet import _bf16_weights, _flat_grads, _to_oracle  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(8, (5, 13, 30, 50), 2), (24, (24, 48, 96, 192), 1), (40, (17, 24, 33, 49), 3), (16, (48, 9, 8, 25), 1),
          (64, (3, 5, 7, 9), 1)]


def _open_net(arch, rng):
    """Flat parameters: zero-sum taps, biases that keep every ReLU open."""
    flat = []
    for _, cin, cout, kind in arch:
        if kind in "cs":
            w = rng.normal(0.0, 0.25 / math.sqrt(9 * cin), (9, cin, cout))
            flat += [(w - w.mean(0)).ravel(), rng.uniform(3.0, 5.0, cout)]
        elif kind == "h":
            flat += [rng.normal(0.0, 1.0 / math.sqrt(cin), cin), rng.normal(size=1)]
    return np.concatenate(flat).astype(np.float32)


def _reference(params, arch, x, noise):
    """Targets (the outputs plus noise), the loss's gradients and the smallest value
    any ReLU gets."""
    total, low, targets = 0.0, np.inf, []
    for b in range(len(x)):
        out, cache = G.forward(params, arch, x[b].astype(np.float64), store=G.round_bf16)
        low = min([low] + [c[1][1].min() for c, a in zip(cache, arch) if a[3] in "cs"])
        targets.append((out[0] + noise[b]).astype(np.float32))
        _, gout = G.h1_loss(out, targets[-1][None], 0.0)
        grads, _ = G.backward(params, arch, cache, gout / len(x))
        total = total + _flat_grads(grads, arch)
    return np.stack(targets), total, low


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()


@pytest.mark.parametrize("hw,ch,batch", SHAPES)
def test_layers_at_tile_edges(hw, ch, batch):
    _cuda()
    arch = G.architecture(ch=ch)
    rng = np.random.default_rng(hw)
    flat = _open_net(arch, rng)
    params = _bf16_weights(_to_oracle(flat, arch), arch)
    x = rng.normal(size=(batch, 3, hw, hw)).astype(np.float32)
    t, want, low = _reference(params, arch, x, rng.normal(size=(batch, hw, hw)))
    assert low > 0.1
    net = P.ax_guessnet_create(hw, ch, batch_capacity=batch + 1, seed=3)
    try:
        P.ax_guessnet_set_params(net, flat)
        _, got = P.ax_guessnet_gradients(net, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), batch)
    finally:
        P.ax_guessnet_destroy(net)
    off = 0
    for name, cin, cout, kind in arch:
        if kind not in "csh":
            continue
        for part, n in (("w", (9 if kind != "h" else 1) * cin * cout), ("b", cout)):
            a, r = got[off:off + n], want[off:off + n]
            off += n
            assert np.linalg.norm(a - r) <= 5e-3 * np.linalg.norm(r), (name, part)


def _constant_net(ch, value, bias, head, head_bias):
    """Every weight `value`, every bias `bias`, the head's weights `head`."""
    flat = []
    for _, cin, cout, kind in G.architecture(ch=ch):
        if kind in "cs":
            flat += [np.full(9 * cin * cout, value), np.full(cout, bias)]
        elif kind == "h":
            flat += [np.full(cin, head), [head_bias]]
    return np.concatenate(flat).astype(np.float32)


@pytest.mark.parametrize("ch,hw,batch", [((24, 8, 8, 8), 64, 1), ((6, 8, 8, 8), 64, 2), ((48, 8, 8, 8), 128, 1)])
def test_sums_that_cancel(ch, hw, batch):
    """With zero weights, biases and activations of one and an output of zero, the
    head's gradients and those of the biases before it are all sum(gy), gy = -2 t / n
    exactly.  t = +-1e4 cancels but for its noise.  Each sample's sum may be off by its
    rounding to FP32 and by n roundings to FP64 on the way, and they are added in FP32."""
    _cuda()
    net = P.ax_guessnet_create(hw, ch, batch_capacity=batch, seed=3)
    try:
        P.ax_guessnet_set_params(net, _constant_net(ch, 0.0, 1.0, 1.0, -ch[0]))
        rng = np.random.default_rng(hw)
        t = np.stack([rng.permutation(np.resize([1e4, -1e4], hw * hw)) + rng.normal(size=hw * hw) for _ in range(batch)])
        t = t.astype(np.float32)
        x = torch.zeros((batch, 3, hw, hw), dtype=torch.float32, device="cuda")
        _, grad = P.ax_guessnet_gradients(net, x, torch.from_numpy(t).cuda().view(batch, hw, hw), batch)
    finally:
        P.ax_guessnet_destroy(net)
    gy = t.astype(np.float64) * (-2.0 / t.size)  # exact where n is a power of two
    each = [math.fsum(g) for g in gy]
    tol = 2.0 ** -24 * (sum(abs(e) for e in each) + abs(sum(each))) + t.size * 2.0 ** -53 * np.abs(gy).sum()
    c = ch[0]
    got = grad[-(2 * c + 1):]  # biases of the last convolution, the head's weights and bias
    assert np.abs(got - math.fsum(each)).max() <= tol


@pytest.mark.parametrize("value", [float("inf"), 3.4e38])
def test_an_infinite_input_stays_visible(value):
    """3.4e38 is infinite in BF16.  All weights are positive, so the outputs that
    depend on the value are infinite."""
    _cuda()
    ch, hw = (8, 8, 8, 8), 64
    net = P.ax_guessnet_create(hw, ch, batch_capacity=1, seed=3)
    try:
        P.ax_guessnet_set_params(net, _constant_net(ch, 0.125, 1.0, 1.0, 0.0))
        x = torch.zeros((1, 3, hw, hw), dtype=torch.float32, device="cuda")
        x[0, 1, 20, 30] = value
        y = torch.zeros((1, hw, hw), dtype=torch.float32, device="cuda")
        P.ax_guessnet_forward(net, x, y, 1)
        assert torch.isinf(y[0, 17:24, 27:34]).all()
        assert not torch.isnan(y).any()
    finally:
        P.ax_guessnet_destroy(net)
