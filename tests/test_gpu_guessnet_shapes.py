"""The network's tensor-core kernels at the edges of their tiles, against the
FP64 reference on the same BF16 values (see test_gpu_guessnet.py): channels that
fill no 16-channel chunk, 24-channel weight-gradient block or 8-channel vector,
lattices that end inside a 16 x 16 patch, and the default channels.

Tolerances (relative, 2-norm): forward 5e-3; the whole gradient 1e-1, since on
lattices this small one ReLU decision that BF16 rounding flips changes it by
several percent (up to 5e-2 at 16 x 16), while a wrong tile, tap or channel
changes it by its own size.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from oracle import guessnet as G  # noqa: E402
from test_gpu_guessnet import _bf16_weights, _flat_grads, _to_oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hw,ch,batch", [(8, (5, 13, 30, 50), 2), (24, (24, 48, 96, 192), 1), (40, (17, 24, 33, 49), 3),
                                         (16, (48, 9, 8, 25), 1), (64, (3, 5, 7, 9), 1)])
def test_shapes(hw, ch, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    arch = G.architecture(ch=ch)
    net = P.ax_guessnet_create(hw, ch, batch_capacity=batch + 1, seed=3)
    try:
        rng = np.random.default_rng(hw)
        flat = P.ax_guessnet_get_params(net)
        flat = flat + rng.normal(0, 0.05, size=flat.size).astype(np.float32) * (np.abs(flat) == 0)  # non-zero biases
        P.ax_guessnet_set_params(net, flat)
        params = _bf16_weights(_to_oracle(flat, arch), arch)
        x = rng.normal(size=(batch, 3, hw, hw)).astype(np.float32)
        t = rng.normal(size=(batch, hw, hw)).astype(np.float32)
        xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        y = torch.zeros((batch, hw, hw), dtype=torch.float32, device="cuda")
        P.ax_guessnet_forward(net, xd, y, batch)
        got = y.cpu().numpy()
        _, grad = P.ax_guessnet_gradients(net, xd, td, batch)
        want = 0.0
        for b in range(batch):
            ref, cache = G.forward(params, arch, x[b].astype(np.float64), store=G.round_bf16)
            assert np.linalg.norm(got[b] - ref[0]) <= 5e-3 * np.linalg.norm(ref[0])
            _, gout = G.h1_loss(ref, t[b][None], 0.0)
            grads, _ = G.backward(params, arch, cache, gout / batch)
            want = want + _flat_grads(grads, arch)
        assert np.linalg.norm(grad - want) <= 1e-1 * np.linalg.norm(want)
    finally:
        P.ax_guessnet_destroy(net)
