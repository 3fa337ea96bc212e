"""The CTA width and rows per lane that the FP32 2D step takes by itself: strips
of 56 and 120 columns and their remainders, lanes of one row, odd row counts,
and sizes where each width is chosen, against the oracle.  Tolerance 2e-6 per
step (FP32), one step."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import oracle as O  # noqa: E402

from test_gpu_step import make_pair, relerr, to_oracle_f  # noqa: E402


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("opt", [dict(), dict(walls=0)], ids=["walls", "periodic"])
@pytest.mark.parametrize("width", [0, 1], ids=["auto", "narrow"])
@pytest.mark.parametrize("shape", [(55, 4), (56, 2), (57, 3), (113, 7), (121, 5), (200, 150), (300, 221), (1031, 40), (24, 700)],
                         ids=lambda s: "x".join(map(str, s)))
def test_default_shape_against_oracle(shape, width, opt, stencil):
    sim, cfg, st = make_pair(dict(nx=shape[0], ny=shape[1], xi=0.05, **opt), "fp32", stencil=stencil)
    if width:
        sim.set_variant("march2", width << 16)          # 64 threads, rows chosen
    sim.step(1)
    ref = O.run(st, 1)
    assert relerr(sim.get("T"), ref.T) < 2e-6
    assert relerr(sim.get("phi"), ref.phi) < 2e-6
    assert relerr(to_oracle_f(sim.get("pop"), 2), ref.f) < 2e-6
    sim.close()
