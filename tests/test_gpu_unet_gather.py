"""Whole-volume inference with the convolutions forced to the gather kernel
(NM_CONV_GATHER=1), which lays out no operand images: on a fresh handle, and
after a pass of the other form and a change of the weights, against the FP64
oracle U-Net (2 % in norm: BF16 activations, as in test_gpu_unet.py)."""
import numpy as np
import pytest

from tests.test_gpu_unet import _oracle_box, _random_net, _volume, env, to_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def test_apply_without_images_matches_oracle(env, monkeypatch):  # noqa: F811
    torch, nm, dn = env
    shape, body = (20, 28, 36), ((4, 16), (6, 22), (5, 31))
    (z0, z1), (y0, y1), (x0, x1) = body
    dose, den, act = _volume(np.random.default_rng(11), shape, body)
    m = den >= 0.1
    s, a = (np.float32(v[m].astype(np.float64).mean()) for v in (dose, act))
    dev = [torch.from_numpy(v).cuda() for v in (dose, den, act)]
    out = torch.empty(shape, dtype=torch.float32, device="cuda")
    names = [n for n, _, _ in dn.unet_layers(8, (16, 32, 64, 128))]

    def check(net, flat, layers):
        net.apply(*dev, out)
        params = to_oracle(flat, layers, (16, 32, 64, 128), names)
        y = _oracle_box(torch, dn, params, dose, den, act, s, a, (x0 - 8, y0 - 8, z0 - 8), (48, 32, 32))
        exp = s * y[8:8 + z1 - z0, 8:8 + y1 - y0, 8:8 + x1 - x0]
        got = out.cpu().numpy()[z0:z1, y0:y1, x0:x1]
        assert np.linalg.norm(got - exp) < 2e-2 * np.linalg.norm(exp)

    monkeypatch.setenv("NM_CONV_GATHER", "1")
    net, flat, layers = _random_net(torch, nm, 4)
    check(net, flat, layers)
    monkeypatch.delenv("NM_CONV_GATHER")
    check(net, flat, layers)                                 # leaves images of these weights
    other, flat, _ = _random_net(torch, nm, 7)
    other.close()
    net.params(set=flat)
    monkeypatch.setenv("NM_CONV_GATHER", "1")
    check(net, flat, layers)
    net.close()
