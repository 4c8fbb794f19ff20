"""Phantom contents on both sides of the size up to which the host looks them over:
the same majorant for the same largest densities, wherever they stand, the same
refusals, and caller arrays that may change once the call has returned."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ENERGIES = np.geomspace(0.06, 20.0, 23)
SIZES = [(3, 1, 1), (20, 20, 30), (11, 1091, 1), (40, 41, 43)]  # 3, 12000, 12001 and 70520 voxels


def phantom(dims, at):
    n = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(n + at)
    mat = rng.integers(0, 3, n).astype(np.uint8)
    rho = rng.uniform(0.01, 0.2, n).astype(np.float32)
    for k, r in enumerate((1.0, 0.3, 1.85)):  # the largest densities, in turn from one end
        mat[(at + k) % n], rho[(at + k) % n] = k, r
    return W.Phantom(*dims, 0.5, 0.5, 0.5, mat, rho)


@pytest.mark.parametrize("dims", SIZES)
def test_majorant_and_refusals_do_not_depend_on_the_size(dims):
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        table = lambda q: dpm.dpm_diag_table(d.ctx, 9, q, ENERGIES)
        want = table(d.load_phantom(phantom((64, 64, 64), 77)))
        n = dims[0] * dims[1] * dims[2]
        low = phantom(dims, 0)
        low.rho[:] = 0.1
        q = d.load_phantom(low)
        assert np.all(table(q) < want)
        for at in (0, 1, n - 1, n - 2):
            ph = phantom(dims, at)
            assert np.array_equal(table(d.load_phantom(ph)), want)
            keep = ph.mat.copy(), ph.rho.copy()
            d.update_phantom(q, ph)
            ph.mat[:], ph.rho[:] = 2, 19.0  # the call is over: the arrays are the caller's
            assert np.array_equal(table(q), want)
            for m, r in ((16, 1.0), (255, 1.0), (0, 0.0), (0, -1.0), (0, np.nan), (0, np.inf)):
                ph.mat[:], ph.rho[:] = keep
                ph.mat[at], ph.rho[at] = m, r
                for call in (lambda: d.update_phantom(q, ph), lambda: d.load_phantom(ph)):
                    with pytest.raises(dpm.DpmError) as e:
                        call()
                    assert e.value.code == dpm.DPM_EINVAL
                    assert ("material" if m > 15 else "density") in str(e.value)
            assert np.array_equal(table(q), want)
