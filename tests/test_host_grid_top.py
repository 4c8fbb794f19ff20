"""The largest position at which the kernels read a per-material table: within a
node's end of the grid, and with a node of the grid after it, for every number of
nodes (in FP32 the last node less 1e-3 is the last node itself from 32770 nodes up)."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W


@pytest.mark.parametrize("n_e", [64, 2048, 16385, 16386, 32769, 32770, 65535, 65536])
def test_the_last_position_has_a_node_after_it(n_e):
    with dpm.HostTables([W.MATERIALS[0]], dict(W.DEFAULT_PARAMS, n_e=n_e)) as t:
        for name, width in (("ph", 4), ("el", 4), ("pmol", 1)):
            tab, meta = t.get(name)
            top = meta[4]
            assert len(tab) == width * n_e and top == np.float32(top)
            # 1e-3 and half an ulp of a position below 2^16, or one ulp
            assert n_e - 1 - 1e-3 - 2.0 ** -8 <= top < n_e - 1
            assert int(top) + 1 <= n_e - 1
            if n_e <= 32769:
                assert top == np.float32(n_e - 1) - np.float32(1e-3)
