"""The particle queues stay as one launch left them for the next: runs with
other beams, queue sizes and block counts, a failed run, and graph replays in
between give the tallies of fresh contexts."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def inputs():
    ph = W.blob_phantom(24, 20, 28, 0.5, 9)
    e = W.axial_source(ph, W.ELECTRON, W.SPEC_MONO, 15.0, 90.0, 100.0, 6.0, 6.0)
    g = W.axial_source(ph, W.PHOTON, W.SPEC_6MV, 6.0, 90.0, 100.0, 8.0, 8.0)
    return ph, e, g


def test_layouts_and_failures_in_turn():
    ph, e, g = inputs()
    steps = [(g, 30000, {}), (e, 8000, {}), (g, 30000, {}), (e, 8000, dict(blocks_per_sm=2)), (g, 20000, dict(queue_log2=9)),
             (e, 8000, dict(queue_log2=16)), (g, 30000, {})]
    want = []
    for src, n, _ in steps:
        with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
            pid = d.load_phantom(ph)
            d.run(pid, src, n, 3)
            want.append(d.read(pid)[2])
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        pid = d.load_phantom(ph)
        for turn in range(2):
            for (src, n, o), w in zip(steps, want):
                d.reset(pid)
                d.run(pid, src, n, 3, **o)
                assert np.array_equal(d.read(pid)[2], w), (turn, n, o)
            # a launch that gives up its waits leaves the queues in disorder
            d.run(pid, g, 2_000_000, 3, timeout_s=1e-9)
            with pytest.raises(dpm.DpmError):
                d.read(pid)


def test_graph_replay_after_other_layouts():
    ph, e, g = inputs()
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        pids = [d.load_phantom(ph) for _ in range(3)]
        jobs = [(pids[0], g, 0, 20000, 5), (pids[1], e, 0, 4000, 6)]
        first = None
        for o in ({}, dict(blocks_per_sm=1), dict(queue_log2=15), dict(queue_log2=8)):
            for pid in pids:
                d.reset(pid)
            dpm.dpm_run_batch(d.ctx, jobs, dpm.run_opts(use_graph=1))
            got = [d.read(pid)[2] for pid in pids[:2]]
            first = first or got
            assert all(np.array_equal(a, b) for a, b in zip(got, first)), o
            d.run(pids[2], e, 3000, 7, **o)  # another layout before the next replay
            d.read(pids[2])
