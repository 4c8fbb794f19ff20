"""Particles with very many steps that the step limit lets through: electrons of
some 120000 steps that nearly all end in a hard event (a Moller cut of a few eV in a
material of small mean excitation energy), and photons of some 10^5 virtual
collisions between two real ones (one voxel 12000 times as dense as the others)."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_electrons_whose_steps_end_in_hard_events():
    ph = W.slab_phantom(3, 3, 3, 20.0, [(0, 1e9, 0, 1.0)])
    mat = dict(W.MATERIALS[W.MAT_WATER], i_ev=0.05, rho_de=0.0)
    src = W.Source(W.ELECTRON, W.SPEC_MONO, 20.0, (30.0, 30.0, 0.0), 100.0, 1.0, 1.0)
    n, out = 8, []
    with dpm.Dpm(0, [mat], dict(W.DEFAULT_PARAMS, wcc=4e-6)) as d:
        for kernel in (dpm.KERNEL_QUEUE, dpm.KERNEL_HISTORY):
            pid = d.load_phantom(ph)
            d.run(pid, src, n, 5, kernel=kernel, count_events=1)
            _, _, raw, st = d.read(pid)  # raises on the step limit
            assert 100_000 < st["n_e_steps"] / n < 200_000
            out.append((raw, st["n_e_steps"], st["escaped"]))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1:] == out[1][1:]


def test_photons_between_whose_collisions_lie_many_virtual_ones():
    ph = W.slab_phantom(40, 40, 40, 3.0, [(0, 1e9, W.MAT_WATER, 1.0)])
    ph.rho[0] = 12000.0
    src = W.Source(W.PHOTON, W.SPEC_MONO, 1.0, (60.0, 60.0, 0.0), 100.0, 1.0, 1.0)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        pid = d.load_phantom(ph)
        d.run(pid, src, 300, 5, kernel=dpm.KERNEL_HISTORY)
        _, _, raw, st = d.read(pid)
    assert st["n_g_flights"] / 300 > 80_000
    assert raw.sum() / 2.0 ** 32 + st["escaped"] == pytest.approx(st["emitted"], rel=1e-9)


def test_photons_that_need_their_limit_more_than_once():
    """At twice that density some photons take more blocks in all than they may between
    two scatters."""
    ph = W.slab_phantom(40, 40, 40, 3.0, [(0, 1e9, W.MAT_WATER, 1.0)])
    ph.rho[0] = 24000.0
    src = W.Source(W.PHOTON, W.SPEC_MONO, 1.0, (60.0, 60.0, 0.0), 100.0, 1.0, 1.0)
    out = []
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        for runs in ([(0, 300)], [(0, 113), (113, 187)]):
            pid = d.load_phantom(ph)
            for first, n in runs:
                d.run(pid, src, n, 5, first=first, kernel=dpm.KERNEL_HISTORY)
            _, _, raw, st = d.read(pid)  # raises on the step limit
            assert st["n_histories"] == 300 and st["n_g_flights"] / 300 > 160_000
            out.append(raw)
    assert out[0].any() and np.array_equal(*out)
