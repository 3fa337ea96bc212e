"""Lattices so long in y that their blocks do not fit the grid's y axis (65,535),
periodic with a short period: every period steps as a lattice of that length."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


def one_step(period, times, **kw):
    """phi and T after a step of `times` periods [.., ny, nx], as they are and as one period."""
    torch.manual_seed(5)
    out = []
    for n in (times, 1):
        sim = lf.Lattice(ny=period * n, walls=0, **dict(dict(xi=0.1), **kw))
        shape = (sim.shape[:-2] + (1, period, sim.shape[-1]))
        dt = torch.float64 if kw["precision"] == "fp64" else torch.float32
        if n == times:
            start = {k: 0.1 * torch.rand(shape, device="cuda", dtype=dt) + b for k, b in (("phi", 0.0), ("T", 0.9))}
        for k, v in start.items():
            sim.set(k, v.expand(*shape[:-3], n, *shape[-2:]).reshape(sim.shape))
        sim.step(1)
        out.append([sim.get(k, dtype=kw["precision"], device=True).view(*shape[:-3], n, *shape[-2:]) for k in ("phi", "T")])
        sim.close()
    return out


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("nx", [1, 2])
def test_fp64_2d(nx, stencil):
    # 262,144 rows: 65,536 rows of tiles.  A step is about 200 operations on values below 1.
    long, short = one_step(16, 16384, nx=nx, precision="fp64", stencil=stencil)
    for a, b in zip(long, short):
        assert (a - b).abs().max() <= 200 * 2.0 ** -53


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
def test_fp32_3d_quads(stencil):
    # 262,144 rows of 25 quads, 32 lanes each: 65,536 blocks of four rows; xi = 0.1 is one sub-step, so T
    # takes the phi pass.  Rows do the same operations wherever they lie.
    long, short = one_step(16, 16384, d=3, nx=100, nz=2, precision="fp32", stencil=stencil, hydro=0)
    for a, b in zip(long, short):
        assert (a - b).abs().max() == 0


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
def test_fp32_3d_sub_steps(stencil):
    long, short = one_step(16, 16384, d=3, nx=100, nz=2, precision="fp32", stencil=stencil, hydro=0, xi=0.3)
    for a, b in zip(long, short):
        assert (a - b).abs().max() == 0
