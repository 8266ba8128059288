"""The ring transport (photons handed between the lanes of a warp) against the
lane kernel (regroup = 0): the same histories give the same tally and counters
bit for bit, from a single decay to more than a warp's ring holds, with every
sampler and physics option, from sources inside and outside the tracking box,
across the 2^32 boundary of the history ids, when photons hit the step limit,
and for decays with tracked positrons or gamma lines (more lines per decay than
the site queue holds included)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KEYS = ("histories", "emitted", "deposited", "escaped", "killed", "steps", "compton", "photo", "rayleigh", "cutoff",
        "escapes")


@pytest.fixture(scope="module")
def nm():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    nmdose.load()
    return nmdose


@pytest.fixture(scope="module")
def phantom(nm):
    from paper_2111_11687_gb300 import inputs
    ph = inputs.adult_phantom(shape=(37, 30, 33), spacing=(1.55, 1.7, 2.4), seed=7)
    den = np.empty(ph.shape, np.float32)
    mat = np.empty(ph.shape, np.uint8)
    nm.nm_ct_to_phantom(ph.hu, den, mat)
    return ph, den, mat


def _run(nm, phantom, n, regroup, first=0, rayleigh=0, everywhere=False, decay=None, **kw):
    from paper_2111_11687_gb300 import inputs, nuclides
    if decay:
        kw.update(DECAYS[decay] if isinstance(DECAYS[decay], dict) else getattr(nuclides, DECAYS[decay]))
    ph, den, mat = phantom
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP,
                      rayleigh=rayleigh, rayleigh_coeff=1e-4)
    act = np.ones_like(ph.activity) if everywhere else ph.activity
    shape = dict(block_threads=64, chunk=32, warp_aggregate=0, regroup_lanes=12, batches=2)
    shape.update(kw)
    with nm.Dose(den, mat, ph.spacing, gm, activity=act, regroup=regroup, **shape) as d:
        d.seek(first)
        try:
            d.run(n, seed=9)
            status = 0
        except nm.NmError as e:
            status = e.status
        c = d.counters()
        return d.tally(), {k: c[k] for k in KEYS}, status


CASES = ([dict(n=n) for n in (1, 2, 31, 32, 33, 64, 65, 127, 1000, 70_001)] +
         [dict(n=20_000, **kw) for kw in (
             dict(rayleigh=1), dict(kn_sampler=1), dict(rayleigh=1, kn_sampler=1), dict(warp_aggregate=1),
             dict(warp_aggregate=1, rayleigh=1), dict(everywhere=True), dict(block_threads=512, chunk=1024),
             dict(first=2**32 - 7_001), dict(max_steps=3), dict(max_steps=4, kn_sampler=1), dict(batches=1),
             dict(source_mode=1, point=(20.0, 25.0, 40.0)), dict(source_mode=1, point=(0.5, 0.5, 0.5)),
             dict(positron_mev=0.0))])


EIGHT = dict(no_annihilation=1, positron_mev=0.1, gamma_lines=[(0.05 + 0.1 * j, 1.0) for j in range(8)])
DECAYS = {"18F tracked": "F18_TRACKED", "177Lu": "LU177", "131I": "I131", "eight lines": EIGHT,
          "no photon": dict(no_annihilation=1, positron_mev=0.2),
          "pair and line": dict(gamma_lines=[(0.9, 0.7)])}
CASES += [dict(n=n, decay=d) for d in DECAYS for n in (1, 33, 9_001)]
CASES += [dict(n=9_001, decay=d, **kw) for d in ("18F tracked", "131I", "eight lines")
          for kw in (dict(rayleigh=1), dict(kn_sampler=1), dict(everywhere=True), dict(first=2**32 - 3_001),
                     dict(block_threads=256, chunk=64), dict(max_steps=4))]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()))
def test_ring_equals_lane_kernel(nm, phantom, case):
    t0, c0, s0 = _run(nm, phantom, regroup=0, **case)
    t1, c1, s1 = _run(nm, phantom, regroup=1, **case)
    assert s0 == s1 and (s0 == nm.NM_ERR_DEVICE) == ("max_steps" in case)
    if "max_steps" in case:
        # a photon stopped by the limit in the step that found its scatter: the
        # lane kernel has tallied the scatter by then, a regrouped one has not
        for c in (c0, c1):
            assert c["killed"] > 0 and c["emitted"] == c.pop("killed") + c.pop("deposited") + c["escaped"]
        c0.pop("cutoff"), c1.pop("cutoff")
    else:
        assert np.array_equal(t0, t1)
    assert c0 == c1
