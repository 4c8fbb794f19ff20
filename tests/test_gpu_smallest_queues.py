"""Queues of 2^7 and 2^8 slots per shard, the smallest that dpm_run_opts takes:
photon beams on 256-slot shards run at any length, and shorter runs on all of
them, electron beams included, to the tally of the default queues."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu
PH = dict(blob=W.blob_phantom(33, 29, 37, 0.4, 3), slab=W.c1_photon_wbw().phantom)


def tally(d, ph, src, n, seed, **opts):
    pid = d.load_phantom(ph)
    d.run(pid, src, n, seed, n_batches=5, **opts)
    _, _, raw, st = d.read(pid)  # raises on an overflow
    assert st["error_flags"] == 0
    dpm.dpm_free_phantom(d.ctx, pid)
    return raw


@pytest.mark.parametrize("n", [100_000, 300_000, 1_000_000, 5_000_000])
@pytest.mark.parametrize("energy,phantom", [(1.0, "blob"), (18.0, "blob"), (6.0, "slab")])
def test_photon_beams_fit_256_slot_shards(energy, phantom, n):
    ph = PH[phantom]
    src = W.axial_source(ph, W.PHOTON, W.SPEC_MONO, energy, 90.0, 100.0, 6.0, 6.0)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        for seed in range(8):
            want = tally(d, ph, src, n, seed)
            for blocks in (0, 1) if seed == 0 and n <= 1_000_000 else (0,):
                assert np.array_equal(tally(d, ph, src, n, seed, queue_log2=8, blocks_per_sm=blocks), want)


@pytest.mark.parametrize("queue_log2,blocks,n", [(7, 0, 10_000), (7, 1, 1_500), (8, 0, 20_000), (8, 1, 3_000)])
@pytest.mark.parametrize("particle", [W.ELECTRON, W.PHOTON])
def test_short_runs_fit_every_queue(particle, queue_log2, blocks, n):
    ph = PH["blob"]
    src = W.axial_source(ph, particle, W.SPEC_MONO, 18.0, 90.0, 100.0, 6.0, 6.0)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        assert np.array_equal(tally(d, ph, src, n, 4, queue_log2=queue_log2, blocks_per_sm=blocks), tally(d, ph, src, n, 4))


def test_overflow_of_the_smallest_queues_is_an_error():
    ph = PH["blob"]
    src = W.axial_source(ph, W.PHOTON, W.SPEC_MONO, 18.0, 90.0, 100.0, 6.0, 6.0)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        with pytest.raises(dpm.DpmError) as e:
            tally(d, ph, src, 100_000, 4, queue_log2=7, queue_limit=1)
        assert e.value.code == dpm.DPM_EQUEUE_OVERFLOW
