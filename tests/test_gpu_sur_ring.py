"""A residual that is the layer's own input is read from the ring of input rows
in shared memory; a copy of the input as the residual takes the other path.
Both give the same bits, also when the epilogue (here with two outputs) falls
behind the loads that reuse the ring, every time."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zout", [False, True])
def test_ring_residual_is_the_input(zout):
    import torch

    from paper_1102_3094_gb300 import lf

    B, NY, NX = 16, 256, 256
    g = torch.Generator(device="cuda").manual_seed(3)
    h = lf.pad_nhwc(torch.randn(B, NY, NX, 64, generator=g, device="cuda").to(torch.bfloat16))
    w = (0.05 * torch.randn(9, 64, 64, generator=g, device="cuda")).to(torch.bfloat16)
    bias = torch.randn(64, generator=g, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")

    def run(resid):
        out, z = torch.zeros_like(h), torch.zeros_like(h) if zout else None
        lf.lf_sur_conv3x3(B, NY, NX, 64, 64, h, w, bias, 1, resid, None, out, None, z, None, None, err)
        return out

    want = run(h.clone())
    for _ in range(40):
        assert torch.equal(run(h), want)
    assert err.item() == 0
