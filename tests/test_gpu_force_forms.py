"""Forms of the isotropic FP32 force pass that the variant's param names: the
kernel that runs, with automatic and with given planes per segment."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from torch.profiler import ProfilerActivity, profile  # noqa: E402

from paper_1102_3094_gb300 import lf  # noqa: E402


def kernels(f):
    for _ in range(3):                                 # the first records of a process may be empty
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            f()
            torch.cuda.synchronize()
        names = [e.key for e in p.key_averages() if "k_" in e.key]
        if names:
            return names
    pytest.skip("no kernel records on this machine")


@pytest.mark.parametrize("param,packed", [(0, True), (16, False), (2 << 16, False), (2 << 16 | 16, False), (4 << 16, True),
                                          (4 << 16 | 16, True)])
def test_form_of_the_force_pass(param, packed):
    sim = lf.Lattice(d=3, nx=40, ny=30, nz=33, precision="fp32", stencil="isotropic", T_w=0.9)
    sim.set_variant("split3", param)
    names = kernels(lambda: sim.step(1))
    assert any("k_force3d_iso_x2" in n for n in names) == packed
    assert any("k_force3d_iso<" in n for n in names) != packed
    sim.close()


def test_the_tuner_times_one_lane_at_automatic_heights():
    """One-lane heights differ (automatic, 8 and 16 planes): three grids of that kernel, of which the automatic one is
    the form 2 at param 0."""
    sim = lf.Lattice(d=3, nx=41, ny=30, nz=31, precision="fp32", stencil="isotropic", T_w=0.9)
    calls = {}
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        sim.tune(1)
        torch.cuda.synchronize()
    for e in p.events():
        if "k_force3d_iso" in e.name:
            calls[e.name] = calls.get(e.name, 0) + 1
    if not calls:
        pytest.skip("no kernel records on this machine")
    one = [n for k, n in calls.items() if "k_force3d_iso<float, 28, 12, 2>" in k]
    other = [n for k, n in calls.items() if "k_force3d_iso<float, 28, 28, 1>" in k]
    assert one and one == other                        # as many heights as the 28 x 28 tiles are timed at
    sim.close()
