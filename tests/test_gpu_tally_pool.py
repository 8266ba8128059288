"""The batch tallies that runs share: one buffer serves the handles that run one
after the other, whatever their grids and batches, and is clear for each; runs
of several threads, and patients side by side, have their own; nothing is held
by the handles, and the library gives the memory back."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TALLY = 96 * 128 * 128 * 8       # bytes of one at the largest grid here


@pytest.fixture(scope="module")
def nm():
    from paper_2111_11687_gb300 import build, nmdose
    build.build()
    nmdose.load()
    return nmdose


def _make(nm, shape, batches, **kw):
    from paper_2111_11687_gb300 import inputs
    r = np.random.default_rng(shape[0])
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    return nm.Dose(r.uniform(0.9, 1.1, shape).astype(np.float32), np.full(shape, 3, np.uint8), (0.3, 0.3, 0.3), gm,
                   activity=np.ones(shape, np.float32), labels=r.integers(0, 5, shape).astype(np.uint8), n_labels=4,
                   batches=batches, block_threads=128, chunk=32, warp_aggregate=0, regroup=1, regroup_lanes=12, **kw)


def _results(d):
    return [d.tally(), *d.get(), *d.organs()]


def test_handles_share_one_buffer(nm):
    import torch
    free = lambda: torch.cuda.mem_get_info()[0]
    shape = (96, 128, 128)
    with _make(nm, shape, 10) as d:                # loads the kernels
        d.run(20_000, seed=1)
        first = _results(d)
    nm.nm_release_cached_memory()
    ds = [_make(nm, shape, 10) for _ in range(4)]
    try:
        f0 = free()
        ds[0].run(20_000, seed=1)
        f1 = free()
        assert f0 - f1 > 9 * TALLY
        for d in ds[1:]:
            d.run(20_000, seed=1)
        assert f1 - free() < 2 * TALLY             # the organs' partial sums, not ten tallies a handle
        for d in ds:
            assert all(np.array_equal(a, b) for a, b in zip(_results(d), first))
    finally:
        for d in ds:
            d.close()
    nm.nm_release_cached_memory()
    assert free() - f1 > 9 * TALLY


@pytest.mark.parametrize("fail", [False, True])
def test_buffer_is_clear_for_the_next_run(nm, fail):
    """Grids and batch counts in turn in one buffer, with runs in between that fail at every step."""
    forms = [((24, 40, 40), 10), ((17, 19, 23), 16), ((24, 40, 40), 3), ((9, 11, 13), 33), ((30, 33, 31), 10)]
    ref = []
    for shape, batches in forms:
        nm.nm_release_cached_memory()
        with _make(nm, shape, batches) as d:
            d.run(6_600, seed=3)
            ref.append(_results(d))
    nm.nm_release_cached_memory()
    with _make(nm, (30, 33, 31), 16) as big:
        big.run(20_000, seed=2)                    # the buffer that all take
        for step in range(1, 25):
            (shape, batches), want = forms[step % 5], ref[step % 5]
            if fail:
                nm.load().nm_debug_fail_enqueue(step)
                try:
                    big.reset()
                    big.run(33_000, seed=5)
                except nm.NmError:
                    pass
                finally:
                    nm.load().nm_debug_fail_enqueue(0)
            with _make(nm, shape, batches) as d:
                d.run(6_600, seed=3)
                assert all(np.array_equal(a, b) for a, b in zip(_results(d), want))


def test_threads_and_patients_have_their_own(nm):
    import torch
    shapes = [(24, 40, 40), (17, 19, 23), (20, 30, 31), (9, 11, 13), (30, 33, 31), (16, 16, 16)]
    ref = []
    for shape in shapes:
        with _make(nm, shape, 10) as d:
            d.run(9_000, seed=3)
            ref.append(_results(d))
    bad = []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with _make(nm, shapes[i], 10, stream=stream.cuda_stream) as d:
                for _ in range(8):
                    d.reset()
                    d.run(9_000, seed=3)
                    if not all(np.array_equal(a, b) for a, b in zip(_results(d), ref[i])):
                        bad.append(i)
        except Exception as e:                     # noqa: BLE001: reported by the main thread
            bad.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    ds = [_make(nm, shape, 10) for shape in shapes]
    try:
        nm.nm_dose_run_batch(ds, [9_000] * len(ds), 3)
        for d, want in zip(ds, ref):
            assert all(np.array_equal(a, b) for a, b in zip(_results(d), want))
    finally:
        for d in ds:
            d.close()
