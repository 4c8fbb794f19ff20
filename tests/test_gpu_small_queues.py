"""Runs that fill and drain small particle queues many times (the secondary
phase ends at a backlog of a few particles per shard, one at least): the same
integer tally as with the default queues, and no error.  The smallest queues are
too small for some of these runs, which then say so (DPM_EQUEUE_OVERFLOW)."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("queue_log2", [7, 8, 10, 12])
@pytest.mark.parametrize("particle", [W.ELECTRON, W.PHOTON])
def test_small_queues_change_nothing_but_the_schedule(particle, queue_log2):
    ph = W.blob_phantom(33, 29, 37, 0.4, 3)
    src = W.axial_source(ph, particle, W.SPEC_MONO, 18.0, 90.0, 100.0, 6.0, 6.0)
    out = []
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        for o in ({}, dict(queue_log2=queue_log2), dict(queue_log2=queue_log2, blocks_per_sm=1)):
            pid = d.load_phantom(ph)
            try:
                d.run(pid, src, 300_000, 19, **o)
                _, _, raw, st = d.read(pid)
            except dpm.DpmError as e:
                assert queue_log2 < 9 and "DPM_EQUEUE_OVERFLOW" in str(e)
                continue
            assert st["error_flags"] == 0
            out.append(raw)
    assert out and all(np.array_equal(out[0], x) for x in out[1:])
