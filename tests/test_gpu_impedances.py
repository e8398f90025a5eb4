"""The impedances and normals of face nodes on the device.

An interface trace holds v, T = sigma n, Z_p and Z_s of a face: with u the precision's unit roundoff,
Z_s = sqrt(mu / r) carries at most 1.5 u (quotient, halved by the root, and the root) and Z_p 2 u (the sum
lambda + 2 mu besides); the traction of a unit pressure is n, at most 4.5 u off (three squares and two sums,
halved by the root, the root, the reciprocal and the product).  1.001 for the terms of second order."""
import numpy as np
import pytest
import torch

from workloads.geometry import make_map, node_coordinates

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _block(precision, faces, operator="upwind", order=4, nodes=(19, 24, 21)):
    from paper_2011_02600_gb300 import ElasticSolver
    bc = [("interface",) if f in faces else ("free",) for f in range(6)]
    s = ElasticSolver(nodes, order, precision, bc, operator=operator)
    X = torch.from_numpy(np.stack(node_coordinates(make_map("curvy", (1000.0, 1100.0, 900.0)), nodes)))
    g = torch.Generator().manual_seed(11)
    rho, lam, mu = (lo + w * torch.rand(*reversed(nodes), generator=g, dtype=torch.float64)
                    for lo, w in ((1500.0, 1800.0), (-1.0e9, 5.0e10), (1.0e9, 4.0e10)))
    s.setup(X, torch.stack([rho, lam, mu]))
    return s


def _face(field, f):
    """[c][w][u] of face f from (c, ns, nr, nq)."""
    i = -1 if f % 2 else 0
    return (field[..., i], field[..., i, :], field[:, i])[f // 2]


def _trace(s, f, q):
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    n = _face(s.view(s.mat, 3), f)[0].numel()
    out = torch.zeros(8 * n, dtype=s.dtype, device="cuda")
    L.sbp_interface_trace(s.h, f, q, out, _stream())
    return out


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("face", range(6))
def test_trace_impedances_and_normals(precision, face):
    s = _block(precision, (face,))
    q = s.new_fields(9)
    s.view(q, 9)[3:6] = 1.0
    got = _trace(s, face, q).cpu().numpy().reshape(8, -1).astype(np.longdouble)
    r, lam, mu = _face(s.view(s.mat, 3), face).reshape(3, -1).cpu().numpy().astype(np.longdouble)
    a = _face(s.view(s.met, 9)[3 * (face // 2):3 * (face // 2) + 3], face).reshape(3, -1).cpu().numpy().astype(np.longdouble)
    u = np.longdouble(2.0) ** (-53 if precision == 64 else -24)
    n = a / np.sqrt((a ** 2).sum(0))
    for value, want, bound in ((got[6], np.sqrt((lam + 2 * mu) / r), 2.0), (got[7], np.sqrt(mu / r), 1.5),
                               (got[3:6], n, 4.5)):
        assert (np.abs(value - want) <= 1.001 * bound * u * np.abs(want)).all()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("face", [0, 1])
def test_equal_media_have_equal_impedances_at_an_interface(precision, face):
    """Equal media on both sides, this one moving along the normal with a power of two, the other at rest:
    the interface takes half of it, exactly (a quotient of Z v and 2 Z; the tangential part multiplies by a
    rounded reciprocal).  Traditional order 2 (its rows sum to zero exactly), unit metrics, lambda = 0: the
    stress rate at the face is the penalty's alone, a whole number times mu."""
    from paper_2011_02600_gb300 import _lib as L
    s = _block(precision, (face,), operator="traditional", order=2)
    s.set_map_path("general")
    s.view(s.met, 9).copy_(torch.eye(3, dtype=s.dtype).reshape(9, 1, 1, 1))
    s.view(s.mat, 3)[1].zero_()
    other = _trace(s, face, s.new_fields(9))
    assert (other.view(8, -1)[6:] > 0).all()
    L.sbp_set_interface(s.h, face, other)
    mu = _face(s.view(s.mat, 3), face)[2]
    inner = (slice(1, -1),) * 2
    Q = torch.zeros(9, *reversed(s.nodes), dtype=s.dtype)
    Q[0] = 0.5
    rate = _face(s.rhs(Q), face)[3]
    jump = 0.25 * 2 * (s.nodes[0] - 1)                      # half the velocity over H0 = h / 2
    assert torch.equal(rate.abs()[inner], (2.0 * mu * jump)[inner])
