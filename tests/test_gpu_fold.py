"""Batches that share a launch: each has a tally of its own and one pass folds
them all, which must leave the bits that a launch and a fold per batch leave,
at batch counts around the fold's variants (1, 2, 5, 10, 16 slots and several
launches), with sizes that do not divide, and with organ labels that fill a
tile with one label, a few, or more than the kernel keeps columns for."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SHAPE = dict(block_threads=128, chunk=32, warp_aggregate=0, regroup=1, regroup_lanes=12)


@pytest.fixture(scope="module")
def nm():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    nmdose.load()
    return nmdose


@pytest.fixture(scope="module")
def phantom(nm):
    from paper_2111_11687_gb300 import inputs
    ph = inputs.adult_phantom(shape=(29, 33, 31), spacing=(1.65, 1.55, 3.1), seed=3)
    den = np.empty(ph.shape, np.float32)
    mat = np.empty(ph.shape, np.uint8)
    nm.nm_ct_to_phantom(ph.hu, den, mat)
    return ph, den, mat


def _labels(ph, kind):
    r = np.random.default_rng(1)
    return {"organs": ph.labels, "none": None, "one": np.full(ph.shape, 3, np.uint8),
            "random": r.integers(0, 32, ph.shape).astype(np.uint8)}[kind]


def _make(nm, phantom, labels, batches, **kw):
    from paper_2111_11687_gb300 import inputs
    ph, den, mat = phantom
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    return nm.Dose(den, mat, ph.spacing, gm, activity=ph.activity, labels=labels, batches=batches,
                   n_labels=0 if labels is None else 31, activity_bq=1e6, **SHAPE, **kw)


@pytest.mark.parametrize("kind", ["organs", "none", "one", "random"])
@pytest.mark.parametrize("batches,n", [(1, 4_001), (2, 4_001), (3, 3_999), (5, 5_003), (7, 100), (10, 50_009),
                                       (11, 9_000), (16, 20_000), (20, 20_013), (33, 40_001)])
def test_shared_launch_equals_a_launch_per_batch(nm, phantom, batches, n, kind):
    ph, den, _ = phantom
    labels = _labels(ph, kind)
    sizes = [n // batches + (b < n % batches) for b in range(batches)]
    with _make(nm, phantom, labels, batches) as d, _make(nm, phantom, labels, 1) as one:
        d.run(n - 1 if batches == 1 else n, seed=4)
        tallies = []
        for s in (sizes if batches > 1 else [n - 1]):
            one.run(s, seed=4)
            tallies.append(one.tally())
        if batches == 1:                      # the uncertainty takes two batches
            d.run(1, seed=4)
            one.run(1, seed=4)
            tallies.append(one.tally())
            sizes = [n - 1, 1]
        assert np.array_equal(d.tally(), one.tally())
        c, c1 = d.counters(), one.counters()
        for k in ("histories", "batches", "deposited", "escaped", "steps", "compton", "photo", "escapes"):
            assert c[k] == c1[k], k
        assert c["emitted"] == c["deposited"] + c["escaped"]
        (dose, sigma), (dose1, sigma1) = d.get(), one.get()
        assert np.array_equal(dose, dose1) and np.array_equal(sigma, sigma1)
        # S2 in 64 bits from the batches' own tallies (sum, then FP32 rounding of the map: 2^-23)
        t = np.diff(np.stack([np.zeros_like(tallies[0])] + tallies), axis=0).astype(np.float64)
        s2 = sum(x * x / m for x, m in zip(t, sizes))
        tot = t.sum(0)
        var = np.maximum(s2 - tot * tot / n, 0.0) / ((len(sizes) - 1) * n)
        mass = den.astype(np.float64) * np.prod(ph.spacing) * 1e-3
        ref = np.sqrt(var) * 1.602176634e-19 / 64.0 * 1e6 / mass
        assert np.allclose(sigma, ref, rtol=1e-5, atol=1e-6 * ref.max())
        if labels is not None:
            for a, b in zip(d.organs(), one.organs()):
                assert np.allclose(a, b, rtol=1e-9, atol=0)
            for a, b in zip(d.organs(eps=False), one.organs(eps=False)):
                if a is not None:
                    assert np.allclose(a, b, rtol=1e-9, atol=0)
