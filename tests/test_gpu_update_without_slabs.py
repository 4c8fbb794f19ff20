"""A phantom that has a tally but no batch slabs (a run that asked for more batches
than fit the context's budget gave up the smaller slabs): contents that are refused
leave its tally as it was, and valid ones replace it."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_refused_contents_leave_a_tally_without_slabs():
    ph = W.blob_phantom(40, 41, 43, 0.5, 5)
    src = W.axial_source(ph, W.PHOTON, W.SPEC_6MV, 6.0, 90.0, 100.0, 6.0, 6.0)
    few = dict(n_batches=2, kernel=dpm.KERNEL_HISTORY)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        pid = d.load_phantom(ph)
        d.run(pid, src, 20000, 3, **few)
        d.read(pid)
        room = dpm.dpm_device_bytes(d.ctx)[0]
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS, hbm_budget_bytes=room + (8 << 20)) as d:
        pid = d.load_phantom(ph)
        d.run(pid, src, 20000, 3, **few)
        want = d.read(pid)
        with pytest.raises(dpm.DpmError) as e:
            d.run(pid, src, 20000, 4, n_batches=1000, kernel=dpm.KERNEL_HISTORY)
        assert e.value.code == dpm.DPM_ENOMEM
        bad = W.Phantom(ph.nx, ph.ny, ph.nz, ph.dx, ph.dy, ph.dz, ph.mat.copy(), ph.rho.copy())
        for mat, rho in ((16, 1.0), (0, np.nan)):
            bad.mat[-1], bad.rho[-1] = mat, rho
            with pytest.raises(dpm.DpmError) as e:
                dpm.dpm_update_phantom(d.ctx, pid, bad)
            assert e.value.code == dpm.DPM_EINVAL
        got = d.read(pid)
        assert want[2].any() and all(np.array_equal(a, b) for a, b in zip(want[:3], got[:3]))
        assert got[3]["n_histories"] == 20000 and got[3]["deposited"] == want[3]["deposited"]
        d.update_phantom(pid, ph)
        assert not d.read(pid)[2].any()
        d.run(pid, src, 20000, 3, **few)
        assert np.array_equal(d.read(pid)[2], want[2])
