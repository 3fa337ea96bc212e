"""Several temperature sub-steps in one pass (2D, FP32): strips of 30 quads and
their halo, rows that end inside a quad, lattices smaller than the halo, one to
four sub-steps per pass and several passes, against the oracle.  Tolerance
2e-6 per step (FP32), three steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import oracle as O  # noqa: E402

from test_gpu_step import make_pair, relerr  # noqa: E402


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("opt", [dict(), dict(walls=0), dict(t_wall_mode=1)], ids=["layers", "periodic", "halfway"])
# n_sub = ceil(xi / 0.2): 2, 3, 4, 5, 6 (two passes of 3 and 2), 12 (three passes)
@pytest.mark.parametrize("xi", [0.3, 0.5, 0.7, 0.9, 1.1, 2.3])
@pytest.mark.parametrize("shape", [(1, 4), (3, 2), (8, 3), (119, 5), (120, 64), (121, 9), (130, 70), (243, 6)],
                         ids=lambda s: "x".join(map(str, s)))
def test_substeps_against_oracle(shape, xi, opt, stencil):
    sim, cfg, st = make_pair(dict(nx=shape[0], ny=shape[1], xi=xi, **opt), "fp32", stencil=stencil)
    sim.step(1)
    ref = O.run(st, 1)
    assert relerr(sim.get("T"), ref.T) < 2e-6
    assert relerr(sim.get("phi"), ref.phi) < 2e-6
    sim.close()
