"""The tiled kernel's march along s.  A small grid's blocks take one or two planes each by the chunk
rule, so that its loop hardly runs: here the length is set (sbp_set_chunk).  A node's arithmetic does not
depend on where its block began (each running sum and queue takes the same planes in the same order), so that
chunks of one plane, three, a ragged part and the whole column agree bit for bit; and with the general
kernel, which does not march, to 1e-12 (FP64) and 1e-5 (FP32) of each field's largest value."""
import dataclasses

import numpy as np
import pytest
import torch

from workloads.configs import config_by_name
from workloads.fields import random_state
from workloads.geometry import make_map, node_coordinates
from workloads.media import make_medium

pytestmark = pytest.mark.gpu

BC = [("char", 0.0), ("char", 0.2), ("char", -0.3), ("char", 0.0), ("char", 0.0), ("free",)]
OPERATORS = [(2, "upwind"), (3, "upwind"), (4, "upwind"), (5, "upwind"), (6, "upwind"), (7, "upwind"),
             (2, "traditional"), (4, "traditional"), (6, "traditional")]
NODES = (37, 19, 45)          # a narrow last tile; the column holds 2 (r + q) + 3 planes of every operator
LENGTHS = (1, 3, 19, 45)


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _grid(name, nodes=NODES):
    X = np.stack(node_coordinates(make_map(name, (1000.0, 1100.0, 900.0)), nodes))
    return X, np.stack(make_medium("smooth_gradient", Lz=900.0)(*X))


def _solver(name, order, prec, operator="upwind"):
    from paper_2011_02600_gb300 import ElasticSolver
    X, mat = _grid(name)
    s = ElasticSolver(NODES, order, prec, BC, operator=operator)
    s.setup(torch.from_numpy(X), torch.from_numpy(mat), keep_metrics=True)
    topo = name == "gaussian_hill" and operator == "upwind" and order % 2 == 0
    assert s.map_path() == ("topography" if topo else "general")
    return s


def _close(a, b, prec):
    scale = b.abs().amax(dim=(1, 2, 3))
    assert scale.min() > 0
    return ((a - b).abs().amax(dim=(1, 2, 3)) / scale).max() < (1e-12 if prec == 64 else 1e-5)


@pytest.mark.parametrize("order,operator", OPERATORS)
@pytest.mark.parametrize("name", ["curvy", "gaussian_hill"])
@pytest.mark.parametrize("prec", [64, 32])
def test_stages_do_not_depend_on_the_chunk(name, order, operator, prec):
    from paper_2011_02600_gb300 import _lib as L
    s = _solver(name, order, prec, operator)
    Q = torch.from_numpy(random_state(NODES, 5, 1.0, 1.0e6))
    s.set_kernel_path(1)
    want = s.rhs(Q).double()
    s.set_kernel_path(0)
    first = None
    for n in LENGTHS:
        L.sbp_set_chunk(s.h, n)
        rate = s.rhs(Q).clone()
        s.set_state(Q)
        s.step(2, 2.0e-4)
        got = rate, s.state().clone(), s.view(s.dq, 9).clone()
        assert s.status() == 0
        if first is None:
            first = got
            assert _close(rate.double(), want, prec)
        assert all(torch.equal(a, b) for a, b in zip(got, first)), n


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("name", ["curvy", "gaussian_hill"])
@pytest.mark.parametrize("prec", [64, 32])
def test_adjoint_step_does_not_depend_on_the_chunk(name, order, prec):
    """L^T w, and a whole adjoint step with its material gradient (one state: one writer per node)."""
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    s, st = _solver(name, order, prec), _stream()
    rlmj = s.new_fields(4, torch.float64)
    J, mat, r = s.view(s.jmet, 10)[0], s.view(s.mat, 3).double(), s.view(rlmj, 4)
    for f, x in enumerate((1.0 / (mat[0] * J), mat[1] * J, mat[2] * J, J)):
        r[f].copy_(x)
    fields = lambda seed, v, t: s.to_layout(torch.from_numpy(random_state(NODES, seed, v, t)), s.dtype)  # noqa: E731
    w, ub0, wb0 = (fields(seed, 1.0e-6, 1.0) for seed in (71, 73, 74))
    u = torch.cat([fields(80 + k, 1.0, 1.0e6) for k in range(5)])

    def run():
        lt, scratch = s.new_fields(9), s.new_fields(18)
        L.sbp_rhs_adjoint(s.h, w, lt, scratch, st)
        ub, wb, grad = ub0.clone(), wb0.clone(), s.new_fields(3, torch.float64)
        L.sbp_adjoint_step(s.h, 2.0e-4, u, ub, wb, scratch, rlmj, grad, st)
        return [s.view(x, n).clone() for x, n in ((lt, 9), (ub, 9), (wb, 9), (grad, 3))]

    s.set_kernel_path(1)
    want = run()
    s.set_kernel_path(0)
    first = None
    for n in LENGTHS:
        L.sbp_set_chunk(s.h, n)
        got = run()
        assert s.status() == 0
        if first is None:
            first = got
            assert _close(got[0].double(), want[0].double(), prec)
        assert all(torch.equal(a, b) for a, b in zip(got, first)), n


@pytest.mark.parametrize("name,prec,order,operator", [("gaussian_hill", 32, 6, "upwind"), ("gaussian_hill", 32, 4, "upwind"),
                                                      ("curvy", 32, 6, "upwind"), ("curvy", 64, 5, "upwind"),
                                                      ("curvy", 32, 4, "traditional")])
@pytest.mark.parametrize("length", [1, 9, 24])
def test_slabs_march_from_their_ghost_planes(name, prec, order, operator, length):
    """Slabs of a block, bit for bit the undivided block, with marches that start in ghost planes."""
    from paper_2011_02600_gb300 import ElasticSolver
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300 import slab as S
    nodes = (37, 19, 70)
    X, mat = _grid(name, nodes)
    Q0 = torch.from_numpy(random_state(nodes, 5, 1.0, 1.0e6))
    whole = ElasticSolver(nodes, order, prec, BC, operator=operator)
    whole.setup(torch.from_numpy(X), torch.from_numpy(mat))
    whole.set_state(Q0)
    L.sbp_set_chunk(whole.h, 70)
    sol = [S.SlabSolver(nodes, order, prec, BC, sl, lambda a, b: X[:, a:b], lambda a, b: mat[:, a:b],
                        operator=operator) for sl in S.partition(nodes[2], 3, order, operator)]
    for s in sol:
        assert s.s.map_path() == whole.map_path() == ("topography" if name == "gaussian_hill" else "general")
        s.state().copy_(Q0[:, s.slab.lo:s.slab.hi])
        L.sbp_set_chunk(s.s.h, length)
    whole.step(3, 2.0e-4)
    S.step_local(sol, 3, 2.0e-4)
    for s in sol:
        assert torch.equal(s.owned(), whole.state()[:, s.slab.k0:s.slab.k1]), s.slab


@pytest.mark.parametrize("prec", [64, 32])
def test_batches_and_the_longest_chunks(prec):
    """A batch with more planes set than the grid holds, against single states by the rule; a negative
    count is refused."""
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.workload_setup import build_solver
    cfg = dataclasses.replace(config_by_name("hill129_o6"), nodes=NODES)
    many, info = build_solver(cfg, precision=prec, batch=3)
    L.sbp_set_chunk(many.h, 1000)
    Q = [torch.from_numpy(random_state(NODES, 5 + b, 1.0, 1.0e6)) for b in range(3)]
    for b in range(3):
        many.state(b).copy_(Q[b])
    many.step(2, info["dt"])
    for b in range(3):
        one, _ = build_solver(cfg, precision=prec)
        one.set_state(Q[b])
        one.step(2, info["dt"])
        assert torch.equal(many.state(b), one.state())
    with pytest.raises(L.SbpError) as e:
        L.sbp_set_chunk(many.h, -1)
    assert e.value.code == 1
