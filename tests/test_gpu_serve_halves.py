"""A server round in two halves (dpm_server_round_begin / _end) gives what
dpm_server_round gives, and takes requests in while it is in flight."""
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def beam(ph, angle):
    X, Y, Z = ph.extent
    return W.Source(W.PHOTON, W.SPEC_6MV, 6.0, (X / 2, Y / 2, Z / 2), 100.0, 0.5, 0.5, angle)


def test_halves_equal_whole_rounds_and_admit_in_between():
    ph = W.blob_phantom(40, 40, 40, 0.4, 100)
    got = []
    for halves in (False, True):
        with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
            g = d.load_phantom(ph)
            s = dpm.Server(d.ctx, dpm.serve_opts(target=0.05, first_chunk=20000))
            assert s.round_begin() == 0 and s.round_end() == 0 and s.round_ready()  # nothing to run
            ids = [s.submit(g, beam(ph, 30.0), 5)]
            late = False
            while any(s.status(i)["state"] in (dpm.REQ_PENDING, dpm.REQ_ACTIVE) for i in ids) or not late:
                if not halves:
                    s.round()
                else:
                    assert s.round_begin() >= 1
                    with pytest.raises(dpm.DpmError) as e:
                        s.round_begin()
                    assert e.value.code == dpm.DPM_ESTATE
                if not late:
                    ids.append(s.submit(g, beam(ph, 200.0), 6))
                    late = True
                    if halves:
                        s.admit()  # gets its slot while the first round is in flight
                        assert s.status(ids[1])["state"] == dpm.REQ_ACTIVE
                if halves:
                    while not s.round_ready():
                        pass
                    s.round_end()
            got.append([{k: s.status(i)[k] for k in ("histories", "rounds", "rel_sigma", "dose_max", "dmax_voxel")}
                        for i in ids])
            s.close()
    assert got[0] == got[1]
