"""A server destroyed with a round in flight: another one takes over on its context,
and it may be destroyed after its context (it then holds host state only)."""
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_a_server_may_go_with_a_round_in_flight():
    ph = W.blob_phantom(40, 40, 40, 0.4, 100)
    X, Y, Z = ph.extent
    src = W.Source(W.PHOTON, W.SPEC_6MV, 6.0, (X / 2, Y / 2, Z / 2), 100.0, 0.5, 0.5, 30.0)
    new = lambda d: dpm.Server(d.ctx, dpm.serve_opts(target=0.05, first_chunk=20000))
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        g = d.load_phantom(ph)
        a, b = new(d), new(d)
        for s in (a, b):
            s.submit(g, src, 5)
        assert a.round_begin() == 1
        with pytest.raises(dpm.DpmError) as e:
            b.round_begin()
        assert e.value.code == dpm.DPM_ESTATE
        a.close()
        assert b.round_begin() == 1
        with pytest.raises(dpm.DpmError):
            b.round_begin()
        b.round_end()
        assert b.status(0)["histories"] == 20000
        assert b.round_begin() == (b.status(0)["state"] == dpm.REQ_ACTIVE)
    b.close()
