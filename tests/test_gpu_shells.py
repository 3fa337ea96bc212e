"""S(k) of lattices with few rows, whose shells are summed over parts of rows:
against its definition with numpy's transform (1e-10, as for the other
lattices), and no slower than the same lattice on its side."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


def shells(phi):
    """S_b with |k| / dk from exact ratios: 4096 x 64 has modes on the half, where 2 pi / L would round."""
    n, least = phi.shape, min(phi.shape)
    S = np.abs(np.fft.fft2(phi - phi.mean())) ** 2 / phi.size
    f = [np.where(2 * np.arange(m) <= m, np.arange(m), np.arange(m) - m) * float(least) / m for m in n]
    b = np.floor(np.sqrt(f[0][:, None] ** 2 + f[1][None, :] ** 2) + 0.5).astype(np.int64).ravel()
    B = least // 2
    total, count = (np.bincount(b, weights=w, minlength=B + 1)[:B + 1] for w in (S.ravel(), None))
    out = np.where(count > 0, total / np.maximum(count, 1), 0.0)
    out[0] = 0.0
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", [(4096, 64), (4096, 3), (4096, 2), (1000, 30), (65, 40), (62, 9), (33, 31), (2, 64)],
                         ids=lambda s: "x".join(map(str, s)))
def test_few_rows_against_the_definition(shape, prec):
    sim = lf.Lattice(nx=shape[0], ny=shape[1], walls=0, precision=prec)
    want = shells(sim.get("phi"))
    np.testing.assert_allclose(sim.structure_factor(), want, rtol=1e-10, atol=1e-14)
    sim.close()


def test_a_wide_lattice_takes_no_longer_than_a_tall_one():
    best = []
    for nx, ny in ((4096, 64), (64, 4096)):
        sim = lf.Lattice(nx=nx, ny=ny, precision="fp32")
        t = []
        for _ in range(30):
            start = time.perf_counter()
            sim.structure_factor()
            t.append(time.perf_counter() - start)
        best.append(min(t))
        sim.close()
    assert best[0] < 2 * best[1]
