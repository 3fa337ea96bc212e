"""Ensembles at their default shape and with several temperature sub-steps per
pass: one to twelve sub-steps in one batch (passes of one to four), odd sizes,
lattices of one strip and of several, both stencils, one run and more runs than
SMs hold CTAs for.  Every run equals the run stepped alone with the same shape,
bit for bit (the per-site arithmetic is shared code)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402

SHAPES = [(24, 3), (57, 9), (119, 33), (121, 64), (243, 40), (64, 130)]
XIS = [0.1, 0.3, 0.5, 0.7, 0.9, 1.1, 2.3]           # 1, 2, 3, 4, 5, 6 and 12 sub-steps


def _members(n, stencil):
    kinds = [dict(), dict(walls=0), dict(t_wall_mode=1)]
    out = []
    for i in range(n):
        nx, ny = SHAPES[i % len(SHAPES)]
        st = ("compact", "isotropic")[i & 1] if stencil == "both" else stencil
        out.append(dict(nx=nx, ny=ny, xi=XIS[i % len(XIS)], tau=1.0, seed=40 + i, stencil=st, **kinds[i % 3]))
    return out


@pytest.mark.parametrize("stencil", ["compact", "isotropic", "both"])
@pytest.mark.parametrize("n", [1, 7, 42, 400])
def test_default_shape_equals_single_runs(n, stencil):
    members = _members(n, stencil)
    ens = lf.Ensemble(members)
    ens.step(3)
    ens.step(2)
    for r in sorted(set(range(min(n, 42))) | {n - 1}):
        m = members[r]
        assert 1 <= ens.rows(r) <= max(1, m["ny"] // 2)
        ref = lf.Lattice(precision="fp32", **m)
        ref.set_variant("march2", ens.param(r))
        ref.step(5)
        for name in ("phi", "T", "pop"):
            np.testing.assert_array_equal(ens.run(r).get(name, "fp32"), ref.get(name, "fp32"), err_msg=f"run {r} {name}")
        ref.close()
    ens.close()
