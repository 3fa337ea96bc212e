"""Convolutions whose BF16 buffers are 16-byte but not 32-byte aligned give the
same bits as on aligned buffers (16-byte accesses in place of 32-byte ones)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1102_3094_gb300 import lf  # noqa: E402


def _at(t, offset):
    """t in a buffer that starts `offset` BF16 elements after a 256-byte boundary."""
    buf = torch.zeros(t.numel() + 128, dtype=t.dtype, device=t.device)
    assert buf.data_ptr() % 256 == 0
    v = buf[offset:offset + t.numel()].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("which", ["resid", "out", "out2", "zout"])
@pytest.mark.parametrize("cin,cout", [(16, 64), (64, 64), (64, 16)])
def test_offset_buffers_give_the_same_bits(cin, cout, which):
    B, NY, NX = 1, 5, 128
    g = torch.Generator().manual_seed(3)

    def rand(*shape):
        return torch.randn(*shape, generator=g).to(torch.bfloat16)

    inp = lf.pad_nhwc(rand(B, NY, NX, cin)).cuda()
    w = rand(9, cout, cin).cuda()
    bias = torch.randn(cout, generator=g).cuda()
    resid, mask = lf.pad_nhwc(rand(B, NY, NX, cout)).cuda(), lf.pad_nhwc(rand(B, NY, NX, cout)).cuda()
    got = []
    for shift in (0, 8):
        bufs = dict(resid=resid, out=torch.zeros_like(resid), out2=torch.zeros_like(resid), zout=torch.zeros_like(resid))
        bufs = {k: _at(v, shift if k == which else 0) for k, v in bufs.items()}
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        lf.lf_sur_conv3x3(B, NY, NX, cin, cout, inp, w, bias, 1, bufs["resid"], mask, bufs["out"], bufs["out2"],
                          bufs["zout"], None, None, err)
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        got.append([bufs[k].clone() for k in ("out", "out2", "zout")])
    for a, b in zip(*got):
        assert torch.equal(a, b)
