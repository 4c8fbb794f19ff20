"""The batch fold and the tally's sum on the device: sigma and the deposited
energy against exact integer arithmetic on the batches' tallies, at batch
counts around the fold's group of ten loads, on a ragged phantom with dense and
empty voxels."""
from fractions import Fraction

import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm
from paper_0910_0329_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("nb,n", [(1, 500), (2, 501), (10, 1000), (11, 1003), (12, 1200), (21, 2000), (50, 49)])
def test_sigma_and_deposited_energy_from_exact_batches(nb, n):
    ph = W.blob_phantom(13, 11, 9, 0.7, 4)
    src = W.axial_source(ph, W.ELECTRON, W.SPEC_MONO, 9.0, 90.0, 100.0, 2.0, 2.0)
    with dpm.Dpm(0, W.MATERIALS, W.DEFAULT_PARAMS) as d:
        pid, one = d.load_phantom(ph), d.load_phantom(ph)
        d.run(pid, src, n, 8, n_batches=nb)
        dose, sigma, raw, st = d.read(pid)
        bs = -(-n // min(nb, n))
        sizes = [min(bs, n - b) for b in range(0, n, bs)]
        batches = []
        for k, m in enumerate(sizes):
            d.reset(one)
            d.run(one, src, m, 8, first=k * bs, n_batches=1)
            batches.append([int(x) for x in d.read(one)[2]])
    B = len(sizes)
    assert st["n_batches"] == B
    s1 = [sum(x) for x in zip(*batches)]
    assert s1 == [int(x) for x in raw] and any(x == 0 for x in s1)
    assert st["deposited"] == float(sum(s1)) / 2.0 ** 32
    conv = 1.602176634e-13 / (ph.rho.astype(np.float64) * ph.dx * ph.dy * ph.dz * 1e-3) / 2.0 ** 32
    for v, s in enumerate(s1):
        assert abs(dose[v] - float(Fraction(s, n)) * conv[v]) <= 8 * U * abs(dose[v])
        q = sum(Fraction(b[v] ** 2, m) for b, m in zip(batches, sizes))
        x = q - Fraction(s * s, n)  # B - 1 times the variance per history
        if B == 1 or s == 0:
            assert sigma[v] == 0.0
            continue
        got = (sigma[v] / conv[v]) ** 2 * n * (B - 1)
        # Q carries at most four roundings, S1^2/n three, and what follows eight
        assert abs(got - float(x)) <= 16 * U * float(q + Fraction(s * s, n))
