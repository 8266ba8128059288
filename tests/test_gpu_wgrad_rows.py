"""The row kernel of the weight gradient (14 x 8 x 2-voxel tiles, groups of
input chunks, z-taps by pass) against the FP64 oracle on the same BF16-rounded
operands, at the edges of its tiles and of its groups.

BF16 x BF16 products are exact in FP32 and the data are >= 0, so the error is
the FP32 accumulation's: at most (chain of additions) 2^-24 of the value, times
four for the tensor core's internal order.  The chain is a CTA's tiles x 16
rows x 16 voxels, then the CTAs; the bias gradient's is at most the voxels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,h,w,cin,cout", [
    (1, 1, 1, 1, 32, 16),        # one voxel
    (2, 2, 8, 14, 32, 16),       # exactly one tile an item; z-taps must not reach the other item
    (2, 3, 9, 15, 48, 16),       # one voxel over in every direction
    (1, 2, 7, 13, 80, 16),       # five chunks in groups of two: the last group half empty
    (1, 5, 17, 29, 32, 32),      # a z-tap a pass
    (2, 1, 9, 1, 144, 32),       # columns; nine chunks by three
    (2, 28, 33, 36, 16, 64),     # one chunk
    (1, 10, 13, 15, 80, 64),     # 64 outputs, the last group half empty
    (2, 52, 70, 73, 8, 128),     # half a chunk
    (1, 20, 64, 70, 48, 128),
    (3, 16, 48, 70, 32, 32),     # more tiles than SMs: several tiles a CTA
    (4, 24, 73, 99, 32, 16),     # 3840 tiles, 26 a CTA: two sums each, added to the partial in turn
    (2, 22, 40, 43, 128, 64),    # the SMs shared among the passes
])
def test_weight_gradient_by_rows(n, d, h, w, cin, cout):
    import torch

    from oracle import denoise
    from paper_2111_11687_gb300 import build, nmdose as nm
    build.build()
    rng = np.random.default_rng([n, d, h, w, cin, cout])
    draw = lambda c: torch.from_numpy(rng.random((n, d, h, w, c), np.float32)).to(torch.bfloat16)
    x, dy = draw(cin), draw(cout)
    kpad = nm.load().nm_conv3d_kpad(cin)
    dw = torch.full((cout, kpad), 7.0, device="cuda")
    db = torch.full((cout,), 7.0, device="cuda")
    nm.nm_conv3d_wgrad(nm._desc(n, d, h, w, cin, cout=cout), x.cuda(), None, dy.cuda(), dw, db)
    got, gotb = dw.cpu().numpy().astype(np.float64), db.cpu().numpy().astype(np.float64)
    ref, refb = denoise.conv3d_wgrad(x.float().numpy().astype(np.float64), dy.float().numpy().astype(np.float64))
    tiles = n * -(-d // 2) * -(-h // 8) * -(-w // 14)
    ctas = min(152, tiles) if cout <= 32 else min(25, -(-tiles // 4))     # fewest that the split makes
    bound = 4 * 2.0 ** -24 * (-(-tiles // ctas) * 256 + ctas)
    assert np.all(got[:, 27 * cin:] == 0.0)                              # padding columns
    assert np.all(np.abs(got[:, :27 * cin].reshape(ref.shape) - ref) <= bound * ref)
    assert np.all(np.abs(gotb - refb) <= 4 * 2.0 ** -24 * n * d * h * w * refb)


@pytest.mark.parametrize("cin,cout,other", [(32, 32, "NM_WGRAD_TILE_UNPACKED"), (64, 64, "NM_CONV_GATHER")])
def test_infinite_inputs_give_the_general_kernels_result(monkeypatch, cin, cout, other):
    """An infinity at the edge of the volume and one inside: bit for bit what the kernel that serves other layers gives."""
    import torch

    from paper_2111_11687_gb300 import build, nmdose as nm
    build.build()
    n, d, h, w = 1, 8, 16, 30
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(n, d, h, w, cin, generator=g, device="cuda").bfloat16()
    dy = torch.randn(n, d, h, w, cout, generator=g, device="cuda").bfloat16()
    x[0, 3, 5, 0, 1] = x[0, 4, 7, 13, 3] = float("inf")
    out = []
    for env in ("", other):
        if env:
            monkeypatch.setenv(env, "1")
        dw = torch.zeros(cout, nm.load().nm_conv3d_kpad(cin), device="cuda")
        nm.nm_conv3d_wgrad(nm._desc(n, d, h, w, cin, cout=cout), x, None, dy, dw)
        out.append(dw.view(torch.int32))
    assert not torch.isfinite(dw).all()
    assert torch.equal(out[0], out[1])
