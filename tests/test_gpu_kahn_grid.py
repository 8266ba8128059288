"""The grid of a handle with Kahn's sampler is that of the kernel it launches,
the one that also takes Rayleigh scattering, not the tabulated sampler's, whose
warps need less shared memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [128, 256, 512])
def test_kahn_and_rayleigh_launch_the_same_grid(block):
    from paper_2111_11687_gb300 import build, inputs
    from paper_2111_11687_gb300 import nmdose as nm
    build.build()
    shape = (8, 8, 8)
    grids = []
    for kw, ray in ((dict(kn_sampler=1), {}), ({}, dict(rayleigh=1, rayleigh_coeff=1e-4))):
        gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP, **ray)
        with nm.Dose(np.ones(shape, np.float32), np.full(shape, 3, np.uint8), (1.0, 1.0, 1.0), gm,
                     activity=np.ones(shape, np.float32), block_threads=block, chunk=64, warp_aggregate=0, regroup=1,
                     regroup_lanes=12, **kw) as d:
            d.run(1000, seed=1)
            grids.append(d.counters()["grid_blocks"])
    assert grids[0] == grids[1] > 0
