"""Phantom contents validated and packed on the device: what is refused leaves the
phantom as it was, whether it has run before or not, and D_max is found in the
voxel that exact arithmetic names, ties and faint densities included."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def bad_arrays(ph):
    n = ph.n_vox
    for at, m, r in ((0, 16, 1.0), (n - 1, 255, 1.0), (n // 2, 0, 0.0), (n - 1, 0, -1.0), (3, 0, np.nan), (n - 2, 0, np.inf)):
        mat, rho = ph.mat.copy(), ph.rho.copy()
        mat[at], rho[at] = m, r
        yield W.Phantom(ph.nx, ph.ny, ph.nz, ph.dx, ph.dy, ph.dz, mat, rho)


@pytest.mark.parametrize("ran", [False, True])
def test_refused_contents_change_nothing(ran):
    ph = W.blob_phantom(17, 13, 19, 0.6, 5)
    src = W.axial_source(ph, W.PHOTON, W.SPEC_6MV, 6.0, 90.0, 100.0, 6.0, 6.0)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        pid, ref = d.load_phantom(ph), d.load_phantom(ph)
        d.run(ref, src, 5000, 3)
        want = d.read(ref)[2]
        if ran:
            d.run(pid, src, 5000, 3)
        for bad in bad_arrays(ph):
            with pytest.raises(dpm.DpmError) as e:
                dpm.dpm_update_phantom(d.ctx, pid, bad)
            assert e.value.code == dpm.DPM_EINVAL
            with pytest.raises(dpm.DpmError) as e:
                d.load_phantom(bad)
            assert e.value.code == dpm.DPM_EINVAL
        got = d.read(pid)[2]
        assert np.array_equal(got, want if ran else 0 * want)
        d.reset(pid)
        d.run(pid, src, 5000, 3)
        assert np.array_equal(d.read(pid)[2], want)


@pytest.mark.parametrize("shape", [(1, 1, 1), (33, 1, 1), (64, 64, 65)])
def test_dmax_is_the_largest_dose_of_the_tally(shape):
    nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(2)
    rho = rng.uniform(0.2, 2.0, n).astype(np.float32)
    rho[::7] = 1e-33  # faint voxels: the largest doses, where they are hit at all
    ph = W.Phantom(nx, ny, nz, 0.5, 0.5, 0.5, np.zeros(n, np.uint8), rho)
    X, Y, _ = ph.extent
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        for tiny in (True, False):
            if not tiny:
                ph.rho[::7] = 1.0
            pid = d.load_phantom(ph)
            assert list(dpm.dpm_dmax_sigma(d.ctx, [pid])[0]) == [0.0, 0.0, -1.0]
            d.run(pid, W.Source(W.ELECTRON, W.SPEC_MONO, 6.0, (X / 2, Y / 2, 0.0), 100.0, X, Y), 20000, 4)
            dose, sigma, raw, _ = d.read(pid)
            out = dpm.dpm_dmax_sigma(d.ctx, [pid])[0]
            # the search compares doses as floats; among equal ones the last voxel wins
            s = raw.astype(np.float64) * 1.602176634e-13 / (ph.rho.astype(np.float64) * (ph.dx * ph.dy * ph.dz) * 1e-3)
            f = s.astype(np.float32)
            if not raw.any():
                assert list(out) == [0.0, 0.0, -1.0]
                continue
            v = int(np.flatnonzero(f == f.max())[-1])
            assert int(out[2]) == v
            assert abs(out[0] - dose[v]) <= 1e-15 * dose[v] and abs(out[1] - sigma[v]) <= 1e-12 * max(sigma[v], 1e-300)
