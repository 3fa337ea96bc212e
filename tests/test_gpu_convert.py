"""Layout conversion of lf_fields / lf_fields_set in FP32: the offsets w_i n0
are added as three floats; the results are those of the sum in double, rounded
once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pop(shape, seed):
    rng = np.random.default_rng(seed)
    f = (1.0 / 9.0) * (1 + 0.05 * rng.standard_normal(shape))
    f[0] = 4.0 / 9.0 * (1 + 1e-7 * rng.standard_normal(shape[1:]))     # deviations of a few ulp
    return f.astype(np.float32)


@pytest.mark.parametrize("kw", [dict(nx=64, ny=9), dict(nx=61, ny=7), dict(nx=2, ny=2), dict(nx=1030, ny=3),
                                dict(d=3, nx=36, ny=5, nz=4), dict(d=3, nx=33, ny=5, nz=4)])
@pytest.mark.parametrize("n0", [1.0, 0.7])
def test_fp32_offsets_as_the_double_sum(kw, n0):
    from paper_1102_3094_gb300 import lf

    sim = lf.Lattice(precision="fp32", n0=n0, **kw)
    f = _pop((sim.Q,) + sim.shape, 3)
    _, w = lf.lf_lattice(kw.get("d", 2))
    off = (w * n0).reshape((-1,) + (1,) * len(sim.shape))
    # float in: one rounding of f - w n0, exactly as the double in gives it
    # (both sums are correct to 2^-46 before that rounding, so they may differ
    # by one unit in the last place where they straddle a tie)
    sim.set("pop", f.astype(np.float64))
    want = sim.get("pop") - off
    sim.set("pop", f)
    got = sim.get("pop") - off
    ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
    assert np.all(np.abs(got - want) <= ulp + 2.0 ** -52)     # off is added and taken away in double
    # float out: the double sum rounded to float
    full = sim.get("pop")
    out = sim.get("pop", dtype="fp32")
    assert np.all(np.abs(out.astype(np.float64) - full) <= np.spacing(np.abs(out)).astype(np.float64) * (0.5 + 2.0 ** -20))
    sim.close()


def test_fp32_offsets_special_values():
    from paper_1102_3094_gb300 import lf

    sim = lf.Lattice(precision="fp32", nx=8, ny=4)
    f = _pop((9, 4, 8), 5)
    f[1, 0, 0], f[2, 1, 3], f[3, 3, 7], f[4, 2, 2] = np.nan, np.inf, -np.inf, np.finfo(np.float32).max
    sim.set("pop", f)
    out = sim.get("pop", dtype="fp32")
    bad = ~np.isfinite(f)
    np.testing.assert_array_equal(out[bad], f[bad])
    np.testing.assert_array_equal(np.isfinite(out), ~bad)
    phi = np.zeros((4, 8), np.float32)
    phi[0, 0], phi[1, 1], phi[2, 2] = -0.0, np.inf, 1e-42
    sim.set("phi", phi)
    np.testing.assert_array_equal(sim.get("phi", dtype="fp32"), phi)
    sim.close()
