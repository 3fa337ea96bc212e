"""Overlapped launches of the FP64 3D step: a pass that is let in early may not
run so unevenly spread over the SMs that the step takes longer than its passes
do one by one.  32 x 32 x 256, where the passes have few blocks: the isotropic
step took 660 us when it was, 517 with the same passes in order."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


def step_us(sim, n=20):
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        sim.step(n)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


def lattice(stencil, xi):
    return lf.Lattice(d=3, nx=32, ny=32, nz=256, precision="fp64", stencil=stencil, xi=xi, T_w=0.9)


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
def test_step_is_not_slower_than_its_passes(stencil):
    sim = lattice(stencil, 0.1)
    whole = step_us(sim)
    sim.set_pass_timing(True)
    parts = []
    for _ in range(10):
        sim.step(1)
        parts.append(sim.pass_times())
    sim.close()
    assert whole < 1.12 * 1e3 * sum(min(p) for p in zip(*parts))


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
def test_sub_steps_cost_what_they_take(stencil):
    """Seven more sub-steps beside the passes: compact 1.15 times the step (1.64 when they crowded the next force
    pass)."""
    one, eight = lattice(stencil, 0.1), lattice(stencil, 1.0)
    assert step_us(eight) < 1.35 * step_us(one)
    one.close()
    eight.close()
