"""The tile of a forward convolution follows how full the layer leaves the chip
(16 x 16 x 2, 16 x 16 x 1 or 16 x 8 x 1 voxels).  An output's additions come in
one order whichever tile holds it, so a volume alone and the same volume in a
large batch give the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,h,w,cin,cout,many", [
    (1, 1, 1, 16, 16, 400),
    (3, 9, 17, 48, 16, 100),
    (2, 8, 16, 8, 16, 300),
    (5, 16, 33, 32, 32, 60),
    (4, 17, 15, 16, 48, 80),
    (16, 16, 16, 64, 64, 20),
    (3, 7, 18, 128, 64, 160),
    (6, 10, 12, 32, 96, 60),
    (8, 8, 8, 64, 192, 80),
])
def test_a_volume_alone_and_in_a_batch_give_the_same_bits(d, h, w, cin, cout, many):
    import torch

    from paper_2111_11687_gb300 import build, nmdose as nm
    build.build()
    g = torch.Generator(device="cuda").manual_seed(d * 1000 + cout)
    kpad = nm.load().nm_conv3d_kpad(cin)
    wt = torch.zeros((cout, kpad), dtype=torch.bfloat16, device="cuda")
    wt[:, :27 * cin] = torch.randn((cout, 27 * cin), generator=g, device="cuda") / np.sqrt(27 * cin)
    bias = torch.randn(cout, generator=g, device="cuda")
    x = torch.randn((4, d, h, w, cin), generator=g, device="cuda").bfloat16()
    out = []
    for n in (1, 4, many):
        xn = x.repeat(-(-n // 4), 1, 1, 1, 1)[:n].contiguous()
        # the middle one at an odd multiple of 16 bytes: two stores a thread instead of one
        off = 8 if n == 4 else 0
        y = torch.empty(n * d * h * w * cout + off, dtype=torch.bfloat16, device="cuda")[off:].view(n, d, h, w, cout)
        nm.nm_conv3d_fwd(nm._desc(n, d, h, w, cin, cout=cout), xn, None, wt, bias, y, True)
        out.append(y)
    assert torch.equal(out[0][0].view(torch.int16), out[2][0].view(torch.int16))
    for i in range(many):
        assert torch.equal(out[1][i % 4].view(torch.int16), out[2][i].view(torch.int16))
