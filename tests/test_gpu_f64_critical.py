"""The FP64 2D step on tiles at the critical temperature: a = (T - Tc) / Tc is
zero there, so with b = kappa = c = 0 the chemical potential vanishes and phi
keeps its bits, whatever Tc and Gamma."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("Tc", [0.005, 0.3, 0.7, 1.1])
def test_phi_is_unchanged_at_Tc(Tc, stencil):
    sim = lf.Lattice(nx=24, ny=20, walls=0, hydro=0, precision="fp64", stencil=stencil, Tc=Tc, T0=Tc, T_w=Tc, b=0.0, kappa=0.0,
                     c=0.0, Gamma=1000.0)
    before = sim.get("phi", device=True)
    sim.step(1)
    assert torch.equal(sim.get("phi", device=True), before)
    sim.close()
