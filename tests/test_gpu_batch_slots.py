"""Device memory of a handle's batch tallies: none beyond the first for a run
whose batches share no launch, one per batch from a run that can use them, and
given back to the library with the handle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_tallies_are_taken_when_a_launch_can_use_them():
    import torch

    from paper_2111_11687_gb300 import build, inputs
    from paper_2111_11687_gb300 import nmdose as nm
    build.build()
    shape = (96, 128, 128)                           # 12.6 MB a tally
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    free = lambda: torch.cuda.mem_get_info()[0]
    nm.nm_release_cached_memory()
    with nm.Dose(np.ones(shape, np.float32), np.full(shape, 3, np.uint8), (0.4, 0.4, 0.4), gm,
                 activity=np.ones(shape, np.float32), batches=10) as d:
        f0 = free()
        d.run(630, seed=1)                           # 63 a batch
        assert f0 - free() < 12 << 20
        first = d.tally()
        d.reset()
        d.run(100_000, seed=1)
        assert f0 - free() > 9 * (12 << 20)
        d.reset()
        d.run(630, seed=1)
        assert np.array_equal(d.tally(), first)
    nm.nm_release_cached_memory()
