"""Densities below FP32's normal range are accepted, and the transport, which
flushes them, tallies what it does with the smallest normal ones: nothing there
interacts either way (probabilities of 1e-27 and less)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("whole", [False, True])
@pytest.mark.parametrize("kw", [{}, dict(regroup=0), dict(history_sigma=1), dict(beta_max_mev=0.6335),
                                dict(kn_sampler=1)])
def test_denormal_density_is_as_good_as_vacuum(kw, whole):
    from paper_2111_11687_gb300 import build, inputs
    from paper_2111_11687_gb300 import nmdose as nm
    build.build()
    shape = (16, 16, 16)
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    thin = np.zeros(shape, bool)
    thin[4:9, 3:12, 6:] = True
    thin |= whole
    mat = np.where(thin, 0, 3).astype(np.uint8)
    res = []
    for rho in (1e-39, 1.2e-38):
        den = np.where(thin, np.float32(rho), np.float32(1.03))
        with nm.Dose(den, mat, (0.4, 0.4, 0.4), gm, activity=np.ones(shape, np.float32), batches=3, block_threads=128,
                     chunk=32, **{"regroup": 1, "regroup_lanes": 12, "warp_aggregate": 0, **kw}) as d:
            d.run(30_000, seed=5)
            c = d.counters()
            assert c["emitted"] == c["deposited"] + c["escaped"] and c["killed"] == 0
            res.append([d.tally()] + [c[k] for k in ("steps", "compton", "photo", "escapes", "escaped")])
    assert all(np.array_equal(a, b) for a, b in zip(*res))
