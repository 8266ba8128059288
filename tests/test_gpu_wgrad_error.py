"""The weight gradient of layers with 64 and 128 outputs, by rows or by the
gather kernel: its error against 64 bits is no larger than the gather kernel's,
at layers on both sides of the line between the two, near it and far, and with
an input group that is not full."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,h,w,cin,cout", [
    (2, 8, 16, 16, 64, 64), (2, 2, 32, 16, 64, 64), (4, 16, 16, 16, 64, 64), (2, 20, 33, 33, 32, 64),
    (3, 21, 23, 25, 80, 64), (2, 40, 60, 60, 16, 64), (2, 40, 60, 60, 64, 64), (1, 7, 20, 17, 96, 128),
    (4, 30, 40, 60, 16, 128), (4, 30, 26, 26, 64, 128), (4, 24, 24, 24, 128, 128)])
def test_error_is_no_larger_than_the_gather_kernels(monkeypatch, n, d, h, w, cin, cout):
    import torch

    from paper_2111_11687_gb300 import build, nmdose as nm
    build.build()
    torch.manual_seed(n * d * h * w + cin)
    x = torch.randn(n, d, h, w, cin, device="cuda").relu().bfloat16()
    dy = (0.1 * torch.randn(n, d, h, w, cout, device="cuda")).bfloat16()
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    flat = dy.double().reshape(-1, cout)
    ref = torch.stack([flat.T @ xp[:, t // 9:t // 9 + d, t // 3 % 3:t // 3 % 3 + h, t % 3:t % 3 + w].reshape(-1, cin)
                       for t in range(27)], 1)
    dw = torch.empty(cout, nm.load().nm_conv3d_kpad(cin), device="cuda")

    def error():
        nm.nm_conv3d_wgrad(nm._desc(n, d, h, w, cin, cout=cout), x, None, dy, dw)
        return float((dw[:, :27 * cin].reshape(ref.shape).double() - ref).norm() / ref.norm())

    mine = error()
    monkeypatch.setenv("NM_CONV_GATHER", "1")
    assert mine <= error() and mine < 1e-5
