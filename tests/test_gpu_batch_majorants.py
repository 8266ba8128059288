"""nm_dose_run_batch with patients whose densest voxels differ, and with them the
majorants that flight lengths are drawn from: every patient's tally and
counters are those of a run of its own, whoever else is in the list."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nm():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    nmdose.load()
    return nmdose


@pytest.mark.parametrize("kw", [{}, dict(kn_sampler=1), dict(regroup=0)])
def test_majorants_of_a_patient_are_its_own(nm, kw):
    from paper_2111_11687_gb300 import inputs
    ph = inputs.adult_phantom(shape=(30, 24, 24), spacing=(2.13, 2.13, 3.0), seed=1)
    den = np.empty(ph.shape, np.float32)
    mat = np.empty(ph.shape, np.uint8)
    nm.nm_ct_to_phantom(ph.hu, den, mat)
    thin = np.where(den > 0.9, 0.8 * den, den).astype(np.float32)
    soft = np.minimum(den, np.float32(1.03)), np.minimum(mat, np.uint8(3))      # no bone
    haze = den.copy()
    haze[:, :2] = 0.15                                                          # denser outside the tracking box
    patients = [(den, mat), (thin, mat), soft, (haze, mat)]
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    make = lambda p: nm.Dose(*p, ph.spacing, gm, activity=ph.activity, labels=ph.labels, n_labels=27, batches=3,
                             block_threads=128, chunk=64, warp_aggregate=0, **{"regroup": 1, "regroup_lanes": 12, **kw})
    keys = ("histories", "emitted", "deposited", "escaped", "steps", "compton", "photo", "cutoff", "escapes")
    batch = [make(p) for p in patients]
    try:
        nm.nm_dose_run_batch(batch, [50_000] * 4, 7)
        tallies = []
        for p, d in zip(patients, batch):
            with make(p) as one:
                one.run(50_000, seed=7)
                assert np.array_equal(d.tally(), one.tally())
                a, b = d.counters(), one.counters()
                for k in keys:
                    assert a[k] == b[k], k
                assert all(np.array_equal(x, y) for x, y in zip(d.organs(), one.organs()))
            tallies.append(d.tally())
        assert not any(np.array_equal(tallies[0], t) for t in tallies[1:])
    finally:
        for d in batch:
            d.close()
