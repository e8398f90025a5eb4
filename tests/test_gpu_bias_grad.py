"""The rounding of the bias gradients' column sums: a value passes through at most ceil(N / 256) + 8 FP32
additions, so that db differs from the exact sum by that many 2^-24 of the sum of magnitudes at most.  The
first 256 values are 1 and the others 2^-21: eight ones in one chain of additions would swallow them."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("N", [256, 600, 1024, 2041, 2048, 2049, 4096, 32768, 40001])
@pytest.mark.parametrize("M", [1, 9])
def test_additions_per_value(M, N):
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    row = torch.full((N,), 2.0 ** -21, dtype=torch.bfloat16)
    row[:256] = 1.0
    dz, db = row.repeat(M, 1).cuda(), torch.zeros(M, device="cuda")
    L.sbp_nn_bias_grad(dz, db, M, N, _stream())
    exact = float(row.double().sum())
    assert ((db.double() - exact).abs() <= (-(-N // 256) + 8) * 2.0 ** -24 * exact).all()
