"""Table values above the grid are those of its last node, also with so many nodes
that the position's clamp rounds to the last node (no node follows it)."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_e", [64, 2048, 65536])
def test_values_above_the_grid_are_those_at_its_end(n_e):
    top = 1.01 * W.DEFAULT_PARAMS["e_max"]
    with dpm.Dpm(0, W.MATERIALS, dict(W.DEFAULT_PARAMS, n_e=n_e)) as d:
        pid = d.load_phantom(W.blob_phantom(9, 8, 7, 0.5, 2))
        for which in (0, 1, 2, 3, 4, 5, 6, 7, 9):
            for m in (pid,) if which == 9 else range(len(W.MATERIALS)):
                end, above = dpm.dpm_diag_table(d.ctx, which, m, np.array([0.9999 * top, 3 * top]))
                # 0.9999 of the last energy and the clamp's 1e-3 of a node lie within
                # 2e-4 in ln E of the end (64 nodes: 1e-3 of a spacing of 0.095);
                # the quantities change by less than ten times that
                assert np.isfinite(above) and abs(above - end) <= 2e-3 * abs(end), (which, m, above, end)
