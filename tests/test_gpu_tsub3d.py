"""Extra temperature sub-steps of 3D FP32 lattices, four sites per thread: rows
that end inside a quad, rows of one to several warps, segments that start at the
last plane, one plane, periodic and walled, against the oracle.  Tolerance 2e-6
(FP32), one step of three to eight sub-steps."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import oracle as O  # noqa: E402

from test_gpu_step import make_pair, relerr  # noqa: E402


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("opt", [dict(), dict(walls=0), dict(t_wall_mode=1)], ids=["layers", "periodic", "halfway"])
@pytest.mark.parametrize("xi", [0.4, 1.0])
@pytest.mark.parametrize("shape", [(5, 3, 4), (33, 6, 7), (130, 5, 9), (32, 17, 33), (61, 40, 13)],
                         ids=lambda s: "x".join(map(str, s)))
def test_substeps_against_oracle(shape, xi, opt, stencil):
    nx, ny, nz = shape
    sim, cfg, st = make_pair(dict(d=3, nx=nx, ny=ny, nz=nz, xi=xi, **opt), "fp32", stencil=stencil)
    sim.step(1)
    ref = O.run(st, 1)
    assert relerr(sim.get("T"), ref.T) < 2e-6
    assert relerr(sim.get("phi"), ref.phi) < 2e-6
    sim.close()
