"""The real transforms behind S(k) and the implicit temperature step, on line
lengths of every radix and parity, against library transforms in FP64.

Tolerances: an FP64 transform is good to about log2(n) eps of the largest
amplitude; a shell's sum of squares of an i.i.d. field is good to 1e-10
relative with room to spare (n <= 4096: 12 x 2.2e-16 x 1e3 terms of both
signs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [dict(nx=1, ny=6), dict(nx=2, ny=3), dict(nx=3, ny=5), dict(nx=4, ny=4), dict(nx=5, ny=7), dict(nx=7, ny=31),
         dict(nx=8, ny=9), dict(nx=30, ny=25), dict(nx=31, ny=62), dict(nx=45, ny=27), dict(nx=128, ny=2),
         dict(nx=256, ny=33), dict(nx=243, ny=50), dict(nx=512, ny=24), dict(nx=1001, ny=6), dict(nx=2048, ny=3),
         dict(nx=4096, ny=2), dict(nx=6, ny=4096), dict(nx=4095, ny=3), dict(d=3, nx=9, ny=8, nz=7),
         dict(d=3, nx=16, ny=5, nz=32), dict(d=3, nx=33, ny=48, nz=10)]


def _shells(phi):
    n = phi.shape[::-1]
    lmin = min(n)
    S = np.abs(np.fft.fftn(phi - phi.mean())) ** 2 / phi.size
    r2 = 0.0
    for ax, m in enumerate(phi.shape):
        k = np.fft.fftfreq(m, 1.0 / m)
        shape = [1] * phi.ndim
        shape[ax] = m
        r2 = r2 + ((k * lmin / m) ** 2).reshape(shape)
    b = np.floor(np.sqrt(r2) + 0.5).astype(int)
    b.flat[0] = 0
    out = np.zeros(lmin // 2 + 1)
    for i in range(1, lmin // 2 + 1):
        out[i] = S[b == i].mean() if (b == i).any() else 0.0
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kw", SIZES, ids=lambda k: "x".join(str(k[a]) for a in ("nx", "ny", "nz") if a in k))
def test_structure_factor_of_every_radix(kw, prec):
    from paper_1102_3094_gb300 import lf

    sim = lf.Lattice(precision=prec, walls=0, **kw)
    phi = np.random.default_rng(7).uniform(-1, 1, size=sim.shape)
    sim.set("phi", phi)
    want = _shells(sim.get("phi"))
    got = sim.structure_factor()
    np.testing.assert_allclose(got, want, rtol=1e-10, atol=1e-12)
    sim.close()


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("kw", [dict(nx=1, ny=5), dict(nx=2, ny=9), dict(nx=31, ny=15), dict(nx=27, ny=4), dict(nx=512, ny=7),
                                dict(d=3, nx=15, ny=14, nz=5), dict(d=3, nx=2, ny=25, nz=6), dict(d=3, nx=64, ny=3, nz=9)],
                         ids=lambda k: "x".join(str(k[a]) for a in ("nx", "ny", "nz") if a in k))
def test_implicit_step_on_odd_lines(kw, walls):
    """FP64, one backward-Euler step: 1e-12, the single-step tolerance of the parity tests."""
    from oracle import t_implicit as TI
    from paper_1102_3094_gb300 import lf

    sim = lf.Lattice(precision="fp64", walls=walls, t_wall_mode=1, xi=7.0, hydro=0, **kw)
    T = np.random.default_rng(8).uniform(0.5, 1.1, size=sim.shape)
    sim.set("T", T)
    sim.set_t_solver("implicit")
    sim.step(1)
    want = TI.implicit_step(T, 7.0, 0.5, walls, 1, 0)
    assert np.abs(sim.get("T") - want).max() / np.abs(want).max() < 1e-12
    sim.close()
