"""Electrons that enter within rounding of an edge of the phantom start in the
voxel at that edge.  The beam comes in over an edge at 45 degrees, and one entry
coordinate of a few in a thousand is a few 1e-6 cm outside.  Without hard events
and deflections the tracks are straight and shorter than 2 cm, so that no energy
can be further than that from the edge."""
import math

import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N, D, E0 = 46, 0.25, 2.0


def far_from_edge(ph, at_x, at_z, r):
    """Voxels whose nearest point is further than r from the edge x = at_x, z = at_z."""
    lo = np.arange(N) * D
    gap = lambda at: np.maximum(np.maximum(lo - at, at - (lo + D)), 0.0)
    far = np.hypot(gap(at_x)[None, :], gap(at_z)[:, None]) > r  # [z, x]
    return np.broadcast_to(far[:, None, :], (ph.nz, ph.ny, ph.nx)).reshape(-1)


@pytest.mark.parametrize("kernel", ["queue", "history", "paper", "f64", "batch"])
@pytest.mark.parametrize("gantry", [45.0, 135.0, 225.0, 315.0])
def test_a_beam_over_an_edge_stays_at_the_edge(gantry, kernel):
    ph = W.slab_phantom(N, 9, N, D, [(0, 1e9, W.MAT_WATER, 1.0)])
    X, Y, Z = ph.extent
    g = math.radians(gantry)
    at_x, at_z = (0.0 if math.sin(g) > 0 else X), (0.0 if math.cos(g) > 0 else Z)
    src = W.Source(W.ELECTRON, W.SPEC_MONO, E0, (at_x, Y / 2, at_z), 100.0, 0.002, 1.0, gantry)
    straight = dpm.NO_MSC | dpm.NO_HARD
    n = 100_000
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        # the path at 2 MeV without hard losses is shorter than 2 cm of water
        assert dpm.dpm_diag_table(d.ctx, 3, W.MAT_WATER, [E0])[0] < 1.9
        pid = d.load_phantom(ph)
        if kernel == "batch":
            dpm.dpm_run_batch(d.ctx, [(pid, src, 0, n, 11)], dpm.run_opts(physics_flags=straight))
        else:
            k = {"queue": dpm.KERNEL_QUEUE, "history": dpm.KERNEL_HISTORY, "paper": dpm.KERNEL_PAPER_F32,
                 "f64": dpm.KERNEL_HISTORY_F64}[kernel]
            d.run(pid, src, n, 11, kernel=k, physics_flags=straight)
        raw = d.read(pid)[2]
    far = far_from_edge(ph, at_x, at_z, 2.0)
    near = raw[~far].sum() / 2.0 ** 32
    assert far.any() and near > 0.5 * n * E0
    assert not raw[far].any(), f"{raw[far].sum() / 2.0 ** 32} MeV far from the edge"
