"""The one-lane force passes at their automatic planes per segment against the
best of a few named heights (they come within 5 % of the best of all; 1.17 times
it, and 1.09 times in FP32, where the lag of a segment was taken too long)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


@pytest.mark.parametrize("precision,stencil,form,dims", [
    ("fp64", "isotropic", 0, (256, 128, 64)), ("fp64", "compact", 0, (128, 128, 128)), ("fp64", "isotropic", 0, (32, 32, 256)),
    ("fp64", "compact", 0, (48, 48, 48)), ("fp32", "isotropic", 3, (256, 128, 64)), ("fp32", "isotropic", 2, (100, 90, 80)),
    ("fp32", "isotropic", 1, (200, 200, 200)), ("fp32", "compact", 2, (64, 64, 64))])
def test_automatic_height(precision, stencil, form, dims):
    sim = lf.Lattice(d=3, nx=dims[0], ny=dims[1], nz=dims[2], precision=precision, stencil=stencil, T_w=0.9)
    sim.set_pass_timing(True)
    ms = {}
    for h in (0, 3, 9, 11, 16, 22, 29, 32):
        sim.set_variant("split3", form << 16 | h)
        ms[h] = float("inf")
        for _ in range(30):
            sim.step(1)
            ms[h] = min(ms[h], sim.pass_times()[0])
    sim.close()
    assert ms.pop(0) <= 1.08 * min(ms.values())
