"""The energy of rows around the length from which a lane takes two neighbouring nodes (FP32), against the
same state one element off its alignment, which is read node by node: the densities are the same FP32 values
and all are positive, so that only the order of the FP64 additions differs (1e-13 of the sum)."""
import numpy as np
import pytest
import torch

from workloads.fields import random_state
from workloads.geometry import make_map, node_coordinates
from workloads.media import make_medium

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nq", [16, 223, 224, 225, 256, 257, 391])
@pytest.mark.parametrize("order", [2, 4, 6])
def test_pairs_match_single_nodes(nq, order):
    from paper_2011_02600_gb300 import ElasticSolver
    from paper_2011_02600_gb300 import _lib as L
    from paper_2011_02600_gb300.solver import _stream
    nodes = (nq, 17, 19)
    X = node_coordinates(make_map("curvy", (1000.0, 1100.0, 900.0)), nodes)
    s = ElasticSolver(nodes, order, 32, [("free",)] * 6)
    s.setup(torch.from_numpy(np.stack(X)), torch.from_numpy(np.stack(make_medium("smooth_gradient", Lz=900.0)(*X))))
    s.set_state(torch.from_numpy(random_state(nodes, 21, 1.0, 1.0e6)))
    s.qbuf[s.current].view(9, s.fs)[:, 17 * 19 * s.ldq:] = float("nan")     # the padding is not summed
    off = torch.empty(9 * s.fs + 1, dtype=torch.float32, device="cuda")[1:]
    off.copy_(s.qbuf[s.current])
    assert off.data_ptr() % 8 == 4
    want = L.sbp_energy_noalloc(off, s.mat, nodes, s.ldq, s.fs, order, 32, 0, _stream())
    assert want > 0 and abs(s.energy() - want) <= 1e-13 * want
