"""The bias gradients of the surrogate on lattices that leave partial passes of their kernel."""
import pytest

pytestmark = pytest.mark.gpu


def test_bias_gradient_of_ragged_batches():
    """Bias gradients on lattice widths and heights that leave partial passes, against FP64 sums of the
    same network in torch (BF16 activations: 2 % as the parity test of the training step allows)."""
    import numpy as np
    import torch

    from oracle import sur_oracle as SO
    from paper_1102_3094_gb300 import lf

    B, NY, NX = 3, 5, 384
    g = torch.Generator().manual_seed(4)
    x, y = (0.3 * torch.randn(B, 4, NY, NX, generator=g) for _ in range(2))
    sur = lf.Surrogate(NY, NX, B, scale=[1.0] * 4, offset=[0.0] * 4, seed=3)
    _, grads = sur.grads(x.cuda(), y.cuda())
    p = torch.from_numpy(sur.get_params())
    Ws, bs, off = [], [], 0
    for cin, cout in ((16, 64), (64, 64), (64, 64), (64, 64), (64, 64), (64, 16)):
        Ws.append(p[off:off + 9 * cin * cout].view(9, cout, cin).to(torch.bfloat16).double()); off += 9 * cin * cout
        bs.append(p[off:off + cout].double()); off += cout
    xn = x.permute(0, 2, 3, 1)
    x16 = torch.nn.functional.pad(xn, (0, 12)).to(torch.bfloat16).double()
    _, _, gb = SO.loss_and_grads(x16, y.permute(0, 2, 3, 1).double(), Ws, bs, x4=xn.double(), bf16_acts=True)
    off = 0
    for (cin, cout), want in zip(((16, 64), (64, 64), (64, 64), (64, 64), (64, 64), (64, 16)), gb):
        off += 9 * cin * cout
        got = grads[off:off + cout].astype(np.float64)
        off += cout
        want = want.numpy()
        assert np.abs(got - want).max() <= 0.02 * np.abs(want).max()
    sur.close()
