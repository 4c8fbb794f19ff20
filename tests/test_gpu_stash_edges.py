"""The queue kernel's per-warp stashes and out buffers at their edges: launches
of one history, of a warp's 32 and of the stash and buffer sizes plus or minus
one, on the smallest and the default queues, against the per-history kernel,
whose integer tally must be the same."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def beams():
    ph = W.blob_phantom(23, 19, 31, 0.41, 6)
    X, Y, Z = ph.extent
    return ph, {
        "electron": W.axial_source(ph, W.ELECTRON, W.SPEC_MONO, 20.0, 90.0, 100.0, 5.0, 5.0),
        "6mv": W.Source(W.PHOTON, W.SPEC_6MV, 6.0, (X / 2, Y / 2, Z / 2), 100.0, 12.0, 12.0, 140.0),
        "pairs": W.axial_source(ph, W.PHOTON, W.SPEC_MONO, 20.0, 90.0, 100.0, 0.3, 0.3),
    }


@pytest.mark.parametrize("queue_log2", [0, 9])
@pytest.mark.parametrize("beam", ["electron", "6mv", "pairs"])
def test_small_launches_equal_the_history_kernel(beam, queue_log2):
    ph, srcs = beams()
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        for n in (1, 31, 32, 33, 47, 49, 1000, 40000):
            tallies = []
            for kernel in (dpm.KERNEL_QUEUE, dpm.KERNEL_HISTORY):
                pid = d.load_phantom(ph)
                d.run(pid, srcs[beam], n, 77, first=3, kernel=kernel, count_events=1, queue_log2=queue_log2, n_batches=7)
                _, _, raw, st = d.read(pid)
                tallies.append((raw, st))
                dpm.dpm_free_phantom(d.ctx, pid)
            (a, sa), (b, sb) = tallies
            assert np.array_equal(a, b)
            for k in ("emitted", "escaped", "missed", "n_e_steps", "n_g_flights", "n_g_interactions", "n_pushed"):
                assert sa[k] == sb[k], k
            assert sa["error_flags"] == sb["error_flags"] == 0


@pytest.mark.parametrize("refill_pause", [-1, 1])
@pytest.mark.parametrize("refill_min", [1, 32])
def test_options_change_nothing_but_the_schedule(refill_pause, refill_min):
    ph, srcs = beams()
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        out = []
        for o in ({}, dict(refill_pause=refill_pause, refill_min=refill_min, blocks_per_sm=3)):
            pid = d.load_phantom(ph)
            d.run(pid, srcs["electron"], 30000, 5, **o)
            out.append(d.read(pid)[2])
        assert np.array_equal(*out)
