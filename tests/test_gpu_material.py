"""The stored coefficients 1/(rho J), lambda/J, mu/J: one rounding per operation in FP64, then one to
the grid's precision, bit for bit as torch's IEEE divisions give them.  One node is infinitely dense
(it keeps its velocity): its moduli stay finite."""
import numpy as np
import pytest
import torch

from workloads.geometry import make_map, node_coordinates

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("name,nodes", [("curvy", (37, 21, 18)), ("gaussian_hill", (16, 17, 33))])
def test_coefficients(precision, name, nodes):
    from paper_2011_02600_gb300 import ElasticSolver
    X = torch.from_numpy(np.stack(node_coordinates(make_map(name, (20000.0, 19000.0, 15000.0)), nodes)))
    g = torch.Generator().manual_seed(sum(nodes))
    rho, lam, mu = (lo + w * torch.rand(*reversed(nodes), generator=g, dtype=torch.float64)
                    for lo, w in ((1500.0, 1800.0), (-1.0e9, 5.0e10), (1.0e9, 4.0e10)))
    rho[3, 4, 5] = float("inf")
    s = ElasticSolver(nodes, 6, precision, [("free",)] * 6)
    s.setup(X, torch.stack([rho, lam, mu]), keep_metrics=True)
    J = s.metrics()[0]
    rho, lam, mu = (f.to(J.device) for f in (rho, lam, mu))
    want = torch.stack([1.0 / (rho * J), lam / J, mu / J]).to(s.dtype)
    assert torch.isfinite(want).all()
    assert torch.equal(s.view(s.mat, 3), want)


def test_padding_is_not_read():
    """Only the nodes of the coordinates, metrics and moduli count: NaN between the rows changes nothing."""
    from paper_2011_02600_gb300 import ElasticSolver
    from paper_2011_02600_gb300 import _lib as L
    from workloads.media import make_medium
    nodes = (37, 21, 18)
    X = np.stack(node_coordinates(make_map("gaussian_hill", (20000.0, 19000.0, 15000.0)), nodes))
    mat = np.stack(make_medium("smooth_gradient", Lz=15000.0)(*X))
    a, b = (ElasticSolver(nodes, 4, 32, [("free",)] * 6) for _ in range(2))
    a.setup(torch.from_numpy(X), torch.from_numpy(mat), keep_metrics=True)
    xyz, jmet, rlm = (torch.full((n * b.fs,), float("nan"), dtype=torch.float64, device="cuda") for n in (3, 10, 3))
    b.view(xyz, 3).copy_(torch.from_numpy(X))
    b.view(rlm, 3).copy_(torch.from_numpy(mat))
    st = torch.cuda.current_stream().cuda_stream
    L.sbp_metrics(b.h, xyz, jmet, st)
    L.sbp_set_material(b.h, jmet, rlm, st)
    assert b.status() == 0 and b.map_path() == a.map_path() == "topography"
    assert torch.equal(b.view(jmet, 10), a.view(a.jmet, 10))
    assert torch.equal(b.view(b.met, 9), a.view(a.met, 9)) and torch.equal(b.view(b.mat, 3), a.view(a.mat, 3))
