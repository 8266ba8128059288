"""A run that fails on the host between the steps it hands to the device: the
handle then holds the launches before the failed one, histories, counters, maps
and organs alike, and goes on from there; or, past the start of a fold, it
refuses runs and read-outs until reset."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BATCHES, N = 33, 3300            # launches of 11 batches: three groups of 1100 histories
GROUP = 1100
SHAPE = dict(block_threads=128, chunk=32, warp_aggregate=0, regroup=1, regroup_lanes=12)


@pytest.fixture(scope="module")
def nm():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    nmdose.load()
    return nmdose


def _make(nm, batches, history):
    from paper_2111_11687_gb300 import inputs
    ph = inputs.adult_phantom(shape=(20, 16, 16), spacing=(3.2, 3.2, 4.5), seed=3)
    den = np.empty(ph.shape, np.float32)
    mat = np.empty(ph.shape, np.uint8)
    nm.nm_ct_to_phantom(ph.hu, den, mat)
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    return nm.Dose(den, mat, ph.spacing, gm, activity=ph.activity, labels=ph.labels, n_labels=27, batches=batches,
                   history_sigma=int(history), **SHAPE)


def _results(d, history):
    c = d.counters()
    out = [np.array([c[k] for k in ("histories", "batches", "emitted", "deposited", "escaped", "steps", "compton",
                                    "photo", "cutoff", "escapes")]), d.tally()]
    assert c["emitted"] == c["deposited"] + c["escaped"]
    if c["histories"]:
        out += [*d.get(), *d.organs()]
        if history:
            out.append(d.history_sigma())
    return out


def _fail(nm, step, run):
    """Whether the run failed at the step (False: it has fewer)."""
    nm.load().nm_debug_fail_enqueue(step)
    try:
        run()
    except nm.NmError as e:
        assert e.status == nm.NM_ERR_CUDA
        return True
    finally:
        nm.load().nm_debug_fail_enqueue(0)
    return False


def _check(nm, d, after, history):
    """True if the handle holds whole launches and goes on, False if it refuses until reset."""
    done = d.counters()["histories"]
    try:
        got = _results(d, history)
    except nm.NmError as e:
        assert e.status == nm.NM_ERR_STATE
        for call in (lambda: d.run(100, seed=2), d.get, d.organs, d.tally, d.checkpoint):
            with pytest.raises(nm.NmError) as e:
                call()
            assert e.value.status == nm.NM_ERR_STATE
        d.reset()
        d.run(N, seed=2)
        assert all(np.array_equal(a, b) for a, b in zip(_results(d, history), after[N]))
        return False
    assert done in after
    for a, b in zip(got, after[done]):
        assert np.array_equal(a, b)
    if done < N:
        d.run(N - done, seed=2)
    assert np.array_equal(d.tally(), after[N][1])
    return True


def _after(nm, history):
    """Results after 0 .. 3 launches of 11 batches, each a run of its own."""
    after = {}
    with _make(nm, 11, history) as d:
        for g in range(4):
            if g:
                d.run(GROUP, seed=2)
            after[g * GROUP] = _results(d, history)
    return after


@pytest.mark.parametrize("history", [False, True])
def test_run_that_fails_on_the_host(nm, history):
    after = _after(nm, history)
    whole, refused, step = 0, 0, 1
    while True:
        with _make(nm, BATCHES, history) as d:
            if not _fail(nm, step, lambda: d.run(N, seed=2)):
                assert all(np.array_equal(a, b) for a, b in zip(_results(d, history), after[N]))
                break
            if _check(nm, d, after, history):
                whole += 1
            else:
                refused += 1
        step += 1
    assert whole >= 15 and refused == (3 if history else 0)   # a launch's squares, after its fold


def test_batched_run_that_fails_on_the_host(nm):
    after = _after(nm, False)
    step, failed = 1, 0
    while True:
        with _make(nm, BATCHES, False) as a, _make(nm, BATCHES, False) as b:
            if not _fail(nm, step, lambda: nm.nm_dose_run_batch([a, b], [N, N], 2)):
                break
            failed += 1
            for d in (a, b):
                _check(nm, d, after, False)
        step += 1
    assert failed >= 30
