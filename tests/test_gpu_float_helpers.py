"""The transport's single-precision functions: reciprocal, quotient and square root
give the nearest float (NumPy's, by IEEE 754) over the ranges stated beside them,
truncation and face positions are exact, and the hardware functions keep to the
errors that PTX states for them (FP64 references on the same float arguments)."""
import numpy as np
import pytest

from paper_0910_0329_gb300 import dpm

pytestmark = pytest.mark.gpu
F = np.float32
ENDS = np.array([0, 1, 2, 3, 0x3504F2, 0x3504F3, 0x3504F4, 0x3FFFFF, 0x400000, 0x400001, 0x7FFFFD, 0x7FFFFE, 0x7FFFFF],
                np.uint32)  # mantissas: the ends, the middle and the root of two


def floats(lo, hi, per, seed):
    """`per` random mantissas and the ends at every binary exponent in [lo, hi)."""
    rng = np.random.default_rng(seed)
    e = np.arange(lo + 127, hi + 127, dtype=np.uint32)[:, None] << 23
    m = np.concatenate([rng.integers(0, 1 << 23, (len(e), per), dtype=np.uint32),
                        np.broadcast_to(ENDS, (len(e), len(ENDS)))], axis=1)
    return (e | m).reshape(-1).view(F)


def run(ctx, which, x, e=1.0, aux=0.0):
    return dpm.dpm_diag_sample(ctx, which, float(e), aux, x.astype(np.float64))


def test_reciprocal_is_the_nearest_float(tables_ctx):
    x = floats(-126, 126, 4096, 1)
    assert np.array_equal(run(tables_ctx.ctx, 10, x), (F(1) / x).astype(np.float64))


def test_quotient_is_the_nearest_float(tables_ctx):
    b = floats(-40, 40, 512, 2)
    num = np.concatenate([floats(-40, 40, 0, 0)[::29], floats(-40, 40, 1, 3)[::9], F([0, 1, 0.2, 0.511, 3.2974426, 20])])
    for a in num:
        with np.errstate(over="raise"):
            want = a / b
        sel = (want == 0) | ((want >= F(2.0 ** -40)) & (want <= F(2.0 ** 40)))
        assert np.array_equal(run(tables_ctx.ctx, 11, b, a)[sel], want.astype(np.float64)[sel]), a


def test_root_is_the_nearest_float(tables_ctx):
    x = np.concatenate([F([0.0]), floats(-100, 100, 4096, 4)])
    assert np.array_equal(run(tables_ctx.ctx, 12, x), np.sqrt(x).astype(np.float64))


def test_truncation_is_exact(tables_ctx):
    k = np.arange(1, 1 << 22, 1021).astype(F)
    x = np.concatenate([F([0.0, 2.0 ** 22, 2.0 ** -149]), floats(-126, 22, 512, 5), k, np.nextafter(k, F(0))])
    for which in (13, 14):
        assert np.array_equal(run(tables_ctx.ctx, which, x), np.trunc(x.astype(np.float64)))


def test_faces_are_exact(tables_ctx):
    i = np.arange(0, 2048)
    for up in (0.0, 1.0):
        assert np.array_equal(run(tables_ctx.ctx, 15, i, aux=up), i + up)


def test_hardware_functions_keep_to_their_stated_errors(tables_ctx):
    x = floats(-100, 100, 512, 6)
    d = x.astype(np.float64)
    ref = np.log2(d)
    err = np.abs(run(tables_ctx.ctx, 16, x) - ref)
    near = (d > 0.5) & (d < 2.0)
    assert err[near].max() <= 2.0 ** -22 and (err[~near] / np.abs(ref[~near]).clip(1e-300)).max() <= 2.0 ** -22
    assert (np.abs(run(tables_ctx.ctx, 18, x) * np.sqrt(d) - 1)).max() <= 2.0 ** -22.9
    for e in F([1e-6, 0.3, 1.0, 77.0]):
        # 2 ulp of the quotient are 2^-22 of it or less
        sel = (d > 2.0 ** -60) & (d < 2.0 ** 60)
        assert (np.abs(run(tables_ctx.ctx, 19, x, e)[sel] * d[sel] / np.float64(e) - 1)).max() <= 2.0 ** -22
    t = np.concatenate([-floats(-20, 6, 512, 7), floats(-20, 6, 512, 8)])
    t64 = t.astype(np.float64)
    # the argument of 2^y, x / ln 2, carries a relative error below 2^-23 (a rounded
    # constant and a rounded product)
    assert np.all(np.abs(run(tables_ctx.ctx, 17, t) / np.exp(t64) - 1) <= 2.0 ** -22 + 1.01 * np.abs(t64) * 2.0 ** -23)
