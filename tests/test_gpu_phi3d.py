"""Pass C of the 3D step with four sites per thread (FP32) on rows that end
inside a vector, that fit exactly, and that leave lanes without sites, against
the oracle; and the automatic segment heights of both passes on such lattices.
Tolerance 2e-6: the single-step tolerance of FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import oracle as O  # noqa: E402

from test_gpu_step import make_pair, relerr, to_oracle_f  # noqa: E402

# (nq + LX - 1) / LX at the edges of the 8, 16 and 32 lanes of a row; nx mod 4 = 0 .. 3; odd heights
SHAPES = [(1, 3, 4), (2, 5, 3), (3, 4, 2), (4, 1, 5), (5, 9, 3), (29, 6, 5), (32, 17, 3), (33, 8, 4), (35, 5, 6), (60, 7, 3),
          (64, 33, 2), (66, 4, 9), (127, 5, 4), (128, 6, 3), (129, 5, 3), (131, 3, 30), (256, 4, 3), (258, 3, 4)]


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("opt", [dict(), dict(walls=0), dict(t_wall_mode=1), dict(hydro=0, t_wall_mode=1)],
                         ids=["layers", "periodic", "halfway", "nohydro"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_one_step_on_ragged_rows(shape, opt, stencil):
    case = dict(d=3, nx=shape[0], ny=shape[1], nz=shape[2], xi=0.1, **opt)
    sim, cfg, st = make_pair(case, "fp32", stencil=stencil)
    sim.step(1)
    ref = O.run(st, 1)
    for name, got, want in (("phi", sim.get("phi"), ref.phi), ("T", sim.get("T"), ref.T),
                            ("f", to_oracle_f(sim.get("pop"), 3), ref.f)):
        assert relerr(got, want) < 2e-6, name
    sim.close()


def test_nonfinite_site_is_seen_and_padding_is_not():
    """A NaN in the last site of a partial vector raises the flag; the padding beyond it never does."""
    from paper_1102_3094_gb300 import lf

    sim = lf.Lattice(d=3, nx=37, ny=6, nz=5, precision="fp32", hydro=0)
    sim.step(2)
    sim.step(1)
    assert sim.diag()["rc"] == 0
    phi = sim.get("phi")
    phi[2, 3, 36] = np.nan
    sim.set("phi", phi)
    sim.step(1)
    assert sim.diag()["rc"] == lf.LF_ENONFINITE
    sim.close()


@pytest.mark.parametrize("opt", [dict(), dict(walls=0), dict(t_wall_mode=1), dict(hydro=0)],
                         ids=["layers", "periodic", "halfway", "nohydro"])
@pytest.mark.parametrize("shape", [(32, 20, 17), (29, 13, 40), (61, 25, 33)], ids=lambda s: "x".join(map(str, s)))
def test_packed_and_one_lane_force_passes_give_the_same_bits(shape, opt):
    """The isotropic force pass on two packed lanes (the automatic choice) against one lane: three steps, every bit."""
    from paper_1102_3094_gb300 import lf

    out = []
    for param in (0, 5, (4 << 16) | 7):           # automatic (packed), one lane of 5 planes, packed lanes of 7
        sim = lf.Lattice(d=3, nx=shape[0], ny=shape[1], nz=shape[2], precision="fp32", stencil="isotropic", xi=0.1,
                         tau=3.0, phi_amp=0.4, **opt)
        sim.set_variant("split3", param)
        sim.step(3)
        out.append([sim.get(k) for k in ("phi", "T", "pop")])
        sim.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)
