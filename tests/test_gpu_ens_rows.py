"""The default height of an ensemble's lanes where another one was measured to
be slower: many small runs (rows of 8 to 11: 600 runs of 64^2 111 us a step, 102
with 16) and large lattices (256 rows at four CTAs per SM: 1 x 4096^2 398, 171 rows
335)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


@pytest.mark.parametrize("runs,side,stencil,hydro,lanes", [
    (2000, 32, "compact", 1, (16,)), (1000, 48, "compact", 1, (12,)), (600, 64, "compact", 1, (16,)),
    (1, 4096, "compact", 1, (171,)), (1, 4096, "compact", 0, (171,)), (4, 1024, "compact", 0, (43,)),
    (200, 256, "isotropic", 1, (26, 32)), (16, 64, "isotropic", 1, (2,))])
def test_rows_per_lane(runs, side, stencil, hydro, lanes):
    ens = lf.Ensemble([dict(nx=side, ny=side, xi=1e-3, seed=i) for i in range(runs)], stencil=stencil, hydro=hydro, T_w=0.9)
    rows = ens.rows(0)
    pairs = min(-(-side // (2 * rows)), side // 2)
    assert -(-side // (2 * pairs)) in lanes            # several heights mean the same lanes
    ens.close()
