"""The finite check of the 3D FP32 phi pass itself: phi, T and mu are finite and
only phi(t+1) overflows, at one site.  With b = kappa = c = 0 and no flow, mu = a
phi with a = -0.99, and phi(t+1) - phi = Gamma lap(mu): at a site with phi = 1 in a
field of zeros 6 (isotropic: 4) Gamma |a|, beyond the largest FP32 number at Gamma
|a| = 1e38, and at its neighbours 1 (1/3) Gamma |a|, within."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("nx,x", [(36, 35), (37, 36), (38, 37), (39, 38), (37, 0), (5, 4), (130, 129)])
def test_only_the_phi_pass_sees_it(nx, x, stencil):
    for scale, want in ((1e38, lf.LF_ENONFINITE), (3e37, lf.LF_OK)):
        sim = lf.Lattice(d=3, nx=nx, ny=6, nz=5, precision="fp32", stencil=stencil, hydro=0, walls=0, b=0.0, kappa=0.0,
                         c=0.0, Tc=1.0, T0=0.01, T_w=0.01, Gamma=scale / 0.99, xi=0.0)
        phi = torch.zeros(sim.shape, device="cuda")
        phi[2, 3, x] = 1.0
        sim.set("phi", phi)
        sim.step(1)
        bad = ~torch.isfinite(sim.get("phi", dtype="fp32", device=True))
        assert int(bad.sum()) == (1 if want else 0)
        assert sim.diag()["rc"] == want
        sim.close()
