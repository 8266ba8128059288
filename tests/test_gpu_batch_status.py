"""A device check that fires for one patient of nm_dose_run_batch marks that
patient alone: the call reports it and names the handle, the other handles'
status stays clean, and all are folded."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_flag_of_one_patient_stays_its_own():
    from paper_2111_11687_gb300 import build, inputs
    from paper_2111_11687_gb300 import nmdose as nm
    build.build()
    shape, spacing = (32, 32, 32), (1.0, 1.0, 1.0)
    act = np.ones(shape, np.float32)
    gm = nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    make = lambda rho, m: nm.Dose(np.full(shape, rho, np.float32), np.full(shape, m, np.uint8), spacing, gm,
                                  activity=act, batches=2, max_steps=8)
    with make(0.0012, 0) as air, make(1.03, 3) as water, make(0.0012, 0) as air2:
        with pytest.raises(nm.NmError) as e:             # a photon in air crosses the cube in a step or two
            nm.nm_dose_run_batch([air, water, air2], [20_000] * 3, 1)
        assert e.value.status == nm.NM_ERR_DEVICE and "handles 1)" in str(e.value)
        assert [d.counters()["device_status"] != 0 for d in (air, water, air2)] == [False, True, False]
        assert all(d.counters()["histories"] == 20_000 for d in (air, water, air2))
        nm.nm_dose_run_batch([air, air2], [1000] * 2, 1)
