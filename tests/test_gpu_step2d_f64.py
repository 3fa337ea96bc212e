"""The FP64 2D step on tiles: lattices that select each tile size, with ragged
edges, every wall rule, both stencils, with and without hydrodynamics, against
the oracle (1e-12, the single-step tolerance of FP64)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import oracle as O  # noqa: E402

from test_gpu_step import make_pair, relerr, to_oracle_f  # noqa: E402


@pytest.mark.parametrize("stencil", ["compact", "isotropic"])
@pytest.mark.parametrize("opt", [dict(), dict(walls=0), dict(t_wall_mode=1), dict(hydro=0)],
                         ids=["layers", "periodic", "halfway", "nohydro"])
@pytest.mark.parametrize("shape", [(1, 2), (2, 3), (3, 5), (7, 4), (8, 9), (64, 64), (61, 47), (128, 128), (131, 77), (200, 150),
                                   (203, 149), (256, 256), (250, 243), (513, 300)], ids=lambda s: "x".join(map(str, s)))
def test_fp64_tiles_against_oracle(shape, opt, stencil):
    sim, cfg, st = make_pair(dict(nx=shape[0], ny=shape[1], xi=0.15, **opt), "fp64", stencil=stencil)
    sim.step(1)
    ref = O.run(st, 1)
    for name, got, want in (("phi", sim.get("phi"), ref.phi), ("T", sim.get("T"), ref.T),
                            ("f", to_oracle_f(sim.get("pop"), 2), ref.f)):
        assert relerr(got, want) < 1e-12, name
    sim.close()
