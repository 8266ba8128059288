"""The order of the organ sums, which the variance of an organ's mean needs kept:
it cancels, so that the last bits of the sums are leading bits of a small sigma.
Columns of 64 voxels, 128 to a tile of 8192, a warp's tree over them, tiles
32-strided: formed here in numpy from the batches' own tallies and from the
maps, and equal bit for bit to Eq. 2 and 3 and the batch sigma, on grids around
the fold's forms (organ sums by tile and slot, whole tiles with columns for 32,
16, 8 and 4 labels) and with more labels in a tile than columns."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SHAPE = dict(block_threads=128, chunk=32, warp_aggregate=0, regroup=1, regroup_lanes=12)
A = 1e6


@pytest.fixture(scope="module")
def nm():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    nmdose.load()
    return nmdose


def _tree(s):
    for o in (16, 8, 4, 2, 1):
        s = s + s[..., np.arange(32) ^ o]
    return s[..., 0]


def _label_sums(x, labels, g=None):
    """x (times g, if given: whole x below 2^40 and an FP32 g, added with one rounding) [voxels] summed per label,
    in the order of the kernels."""
    tiles = -(-x.size // 8192)
    tile = lambda a: np.pad(a, (0, tiles * 8192 - a.size)).reshape(tiles, 64, 128)
    x, g, lab = tile(x), tile(np.ones(x.size) if g is None else g), tile(labels.ravel())
    acc = np.zeros((tiles, 32, 128))
    t, c = np.ogrid[:tiles, :128]
    for k in range(64):
        old = acc[t, lab[:, k], c]
        new = old + x[:, k] * g[:, k]
        for i in np.argwhere(x[:, k] >= 1 << 29):           # the product may have more than 53 bits
            i = tuple(i)
            new[i] = float(Fraction(old[i]) + Fraction(x[:, k][i]) * Fraction(g[:, k][i]))
        acc[t, lab[:, k], c] = new
    a = acc.reshape(tiles, 32, 4, 32)
    part = _tree(((a[:, :, 0] + a[:, :, 1]) + a[:, :, 2]) + a[:, :, 3])      # [tile, label]
    part = np.pad(part, ((0, -tiles % 32), (0, 0)))
    lanes = np.zeros((32, 32))
    for row in part.reshape(-1, 32, 32):
        lanes += row
    return _tree(lanes.T)


def _sigma(s1, s2, n, batches, count):
    mbar = s1 / (n * count)
    nm = n * mbar
    out = []
    for a, b, m in zip(s2 / (count * count), nm, mbar):
        var = max(float(Fraction(a) - Fraction(b) * Fraction(m)), 0.0) / ((batches - 1.0) * n)
        out.append(np.sqrt(var) * A)
    return np.array(out)


@pytest.mark.parametrize("shape,batches,n", [((31, 33, 29), 2, 9_001), ((31, 33, 29), 10, 20_003),
                                             ((113, 110, 107), 2, 300_001), ((113, 110, 107), 10, 200_001),
                                             ((174, 171, 173), 1, 150_001), ((174, 171, 173), 5, 400_003),
                                             ((174, 171, 173), 10, 400_003)])
def test_organ_sums_keep_their_order(nm, shape, batches, n):
    from paper_2111_11687_gb300 import inputs
    spacing = tuple(a / b for a, b in zip((51.2, 51.2, 90.0), shape[::-1]))
    ph = inputs.adult_phantom(shape=shape, spacing=spacing, seed=3)
    r = np.random.default_rng(2)
    fine = r.integers(0, 32, ph.shape).astype(np.uint8)
    labels = np.where(np.arange(shape[0])[:, None, None] % 3 == 0, fine, ph.labels)   # 1 to 32 labels a tile
    den = np.empty(ph.shape, np.float32)
    mat = np.empty(ph.shape, np.uint8)
    nm.nm_ct_to_phantom(ph.hu, den, mat)
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    make = lambda b: nm.Dose(den, mat, ph.spacing, gm, activity=ph.activity, labels=labels, batches=b, n_labels=31,
                             activity_bq=A, **SHAPE)
    runs = 2 if batches == 1 else 1                         # the uncertainty takes two batches
    sizes = [n // batches + (b < n % batches) for b in range(batches)] * runs
    with make(batches) as d, make(1) as one:
        for _ in range(runs):
            d.run(n, seed=4)
        tallies = [np.zeros(ph.shape, np.int64)]
        for s in sizes:
            one.run(s, seed=4)
            tallies.append(one.tally())
        dose, sigma = d.get()
        mean, eps, sg, count = d.organs()
        mean_b, _, sg_b, _ = d.organs(eps=False)
        mapped = d.map_organs(dose)
    dx, dy, dz = (float(np.float32(s)) for s in ph.spacing)
    gy = np.float32(1.602176634e-19 / 64.0 / (1e-3 * dx * dy * dz))
    g = (gy / den).astype(np.float64).ravel()
    total = float(n * runs)
    s1, s2 = np.zeros(32), np.zeros(32)
    for a, b, m in zip(tallies, tallies[1:], sizes):
        o = _label_sums((b - a).ravel().astype(np.float64), labels, g)
        s1, s2 = s1 + o, s2 + o * o / m
    assert np.array_equal(count, np.bincount(labels.ravel(), minlength=32)) and count.min() > 0
    count = count.astype(np.float64)
    assert np.array_equal(mean_b, s1 / (total * count) * A)
    assert np.array_equal(sg, _sigma(s1, s2, total, len(sizes), count))
    # the host's compiler may or may not fuse the last product into the difference
    assert np.allclose(sg_b, sg, rtol=1e-6, atol=1e-9 * mean.max())
    d32, s32 = np.asarray(dose).ravel(), np.asarray(sigma).ravel()
    assert np.array_equal(mean, _label_sums(d32.astype(np.float64), labels) / count)
    with np.errstate(divide="ignore", invalid="ignore"):
        e = np.where(d32 > 0, s32 / d32, np.float32(1))
    assert np.array_equal(eps, np.sqrt(_label_sums((e * e).astype(np.float64), labels) / count))
    assert np.array_equal(mapped, mean)
