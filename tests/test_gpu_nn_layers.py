"""The surrogate's fused layer kernels against plain torch, at the sizes where their paths change:
sample lengths that eight columns divide and that they do not, one and several samples, one row and
many, the ends of a sample, short and long rows of a bias gradient, several Adam tensors.

Copies, the masked gradients and the moment backward round once in the same order as the reference:
equal.  The moment combination: six products and sums in FP32, fused or not, 4e-7 of the largest
term's sum.  Bias gradients: FP32 sums of N BF16 values, N 2^-24 of the sum of magnitudes at most.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _api():
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    return L, _stream()


def _randn(*shape, seed=0, dtype=torch.float32):
    g = torch.Generator().manual_seed(seed + sum(shape))
    return torch.randn(*shape, generator=g).to(dtype).cuda()


def _columns(x, kw, pad):
    """[C][B][T] -> [C * kw][B][T] with zeros outside each sample."""
    C, B, T = x.shape
    xp = torch.nn.functional.pad(x, (pad, max(0, kw - 1 - pad)))
    return torch.stack([xp[..., k:k + T] for k in range(kw)], 1).reshape(C * kw, B, T)


SIZES = [(1, 1, 8), (3, 2, 16), (5, 3, 10), (128, 4, 64), (2, 5, 2056), (7, 1, 2), (4, 33, 40)]


@pytest.mark.parametrize("C,B,T", SIZES)
@pytest.mark.parametrize("up", [1, 2])
@pytest.mark.parametrize("kw,pad", [(5, 2), (3, 1)])
def test_upsampled_columns(C, B, T, up, kw, pad):
    L, st = _api()
    x = _randn(C, B, T // up, dtype=torch.bfloat16)
    out = torch.full((C * kw, B, T), 7.0, dtype=torch.bfloat16, device="cuda")
    L.sbp_nn_upsample_im2col(x, out, C, B, T, up, kw, pad, st)
    assert torch.equal(out, _columns(x.repeat_interleave(up, 2), kw, pad))


@pytest.mark.parametrize("C,B,T", SIZES)
@pytest.mark.parametrize("up", [1, 2])
@pytest.mark.parametrize("kw,pad", [(5, 2), (3, 1)])
def test_column_gradient_through_upsampling_and_relu(C, B, T, up, kw, pad):
    L, st = _api()
    d = _randn(C, kw, B, T)
    a = torch.relu(_randn(C, B, T // up, seed=1, dtype=torch.bfloat16))
    dz = torch.full((C, B, T // up), 7.0, dtype=torch.bfloat16, device="cuda")
    L.sbp_nn_conv_relu_backward(d, a, dz, C, B, T, up, kw, pad, st)
    du = torch.zeros(C, B, T, device="cuda")
    for k in range(kw):   # the column of tap k holds x[t + k - pad]
        lo, hi = max(0, k - pad), min(T, T + k - pad)
        du[..., lo:hi] += d[:, k, :, lo - k + pad:hi - k + pad]
    da = du if up == 1 else du[..., 0::2] + du[..., 1::2]
    assert torch.equal(dz, torch.where(a > 0, da, torch.zeros_like(da)).to(torch.bfloat16))


@pytest.mark.parametrize("n_out,B,T", [(1, 1, 8), (3, 2, 16), (12, 3, 10), (192, 2, 256), (5, 7, 264)])
def test_moment_combination(n_out, B, T):
    L, st = _api()
    G, m = _randn(6, n_out, B, T, dtype=torch.bfloat16), _randn(6, B, seed=1)
    y = torch.full((n_out, B, T), 7.0, device="cuda")
    L.sbp_nn_moment_combine(G, m, y, None, None, n_out, B, T, 0, st)
    terms = m[:, None, :, None].double() * G.double()
    assert ((y - terms.sum(0)).abs() <= 4e-7 * terms.abs().sum(0)).all()
    dy, dG = _randn(n_out, B, T, seed=2, dtype=torch.bfloat16), torch.empty_like(G)
    L.sbp_nn_moment_combine(None, m, None, dy, dG, n_out, B, T, 1, st)
    assert torch.equal(dG, (m[:, None, :, None] * dy.float()).to(torch.bfloat16))


@pytest.mark.parametrize("M,N", [(1, 1), (9, 32), (4097, 33), (3, 2048), (5, 2049), (130, 4104), (2, 32768)])
def test_bias_gradient(M, N):
    L, st = _api()
    dz, db = _randn(M, N, dtype=torch.bfloat16), torch.full((M,), 7.0, device="cuda")
    L.sbp_nn_bias_grad(dz, db, M, N, st)
    assert ((db - dz.double().sum(1)).abs() <= N * 2.0 ** -24 * dz.double().abs().sum(1)).all()


@pytest.mark.parametrize("sizes", [(1,), (2048, 2049, 5), tuple(range(1, 40))])
def test_adam_of_several_tensors(sizes):
    L, st = _api()
    one = [[_randn(n, seed=s).abs() if s == 3 else _randn(n, seed=s) for s in range(4)] +
           [torch.zeros(n, dtype=torch.bfloat16, device="cuda") if n % 2 else None] for n in sizes]
    many = [[None if t is None else t.clone() for t in row] for row in one]
    for w, g, m, v, wb in one:
        L.sbp_nn_adam(w, g, m, v, wb, w.numel(), 1e-3, 0.9, 0.999, 1e-8, 3, st)
    L.sbp_nn_adam_multi(many, 1e-3, 0.9, 0.999, 1e-8, 3, st)
    for a, b in zip(one, many):
        assert all(x is None or torch.equal(x, y) for x, y in zip(a, b))
