"""The surrogate's fused layer calls against the calls they join, bit for bit (each value is one copy or one
chain of FP32 additions in the same order): upsampling and im2col; col2im, the upsampling's pair sums and the
ReLU's mask.  The joined calls remain public entry points."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 8), (3, 2, 16), (5, 3, 10), (128, 4, 64), (2, 5, 2056), (7, 1, 2), (4, 33, 40)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _randn(*shape, seed=0, dtype=torch.float32):
    g = torch.Generator().manual_seed(seed + sum(shape))
    return torch.randn(*shape, generator=g).to(dtype).cuda()


@pytest.mark.parametrize("C,B,T", SIZES)
@pytest.mark.parametrize("kw,pad", [(5, 2), (3, 1)])
def test_upsampled_columns(C, B, T, kw, pad):
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    bf, st = dict(dtype=torch.bfloat16, device="cuda"), _stream()
    x = _randn(C, B, T // 2, dtype=torch.bfloat16)
    up, want, got = torch.zeros(C, B, T, **bf), torch.zeros(C * kw, B, T, **bf), torch.ones(C * kw, B, T, **bf)
    L.sbp_nn_upsample2(x, up, C * B, T // 2, 0, st)
    L.sbp_nn_im2col(up, want, C, B, T, kw, pad, st)
    L.sbp_nn_upsample_im2col(x, got, C, B, T, 2, kw, pad, st)
    assert torch.equal(up, x.repeat_interleave(2, 2)) and torch.equal(got, want)


@pytest.mark.parametrize("C,B,T", SIZES)
@pytest.mark.parametrize("kw,pad", [(5, 2), (3, 1)])
@pytest.mark.parametrize("up", [1, 2])
def test_column_gradient_upsampling_and_relu(C, B, T, kw, pad, up):
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    f32, bf, st = dict(device="cuda"), dict(dtype=torch.bfloat16, device="cuda"), _stream()
    d = _randn(C * kw, B, T)
    a = torch.relu(_randn(C, B, T // up, seed=1, dtype=torch.bfloat16))
    da = du = torch.zeros(C, B, T, **f32)
    L.sbp_nn_col2im(d, du, C, B, T, kw, pad, st)
    if up == 2:
        da = torch.zeros(C, B, T // 2, **f32)
        L.sbp_nn_upsample2(du, da, C * B, T // 2, 1, st)
    want, got = torch.zeros(C, B, T // up, **bf), torch.ones(C, B, T // up, **bf)
    L.sbp_nn_relu_backward(da, a, want, a.numel(), st)
    L.sbp_nn_conv_relu_backward(d, a, got, C, B, T, up, kw, pad, st)
    assert torch.equal(got, want)
