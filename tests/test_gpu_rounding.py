"""How often the stage kernel rounds, where one product more would bias every step alike."""
import dataclasses

import pytest
import torch

from workloads.configs import config_by_name

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nodes", [(33, 18, 17), (36, 21, 40)])
@pytest.mark.parametrize("path", ["auto", "general"])
def test_register_of_the_first_stage_is_dt_times_the_rate(precision, nodes, path):
    """One product in the grid's precision: the same kernel's rates, times dt, bit for bit."""
    from paper_2011_02600_gb300.workload_setup import build_solver
    from workloads.fields import random_state
    cfg = dataclasses.replace(config_by_name("hill129_o6"), nodes=nodes)
    s, info = build_solver(cfg, precision=precision)
    s.set_map_path(path)
    s.set_state(torch.from_numpy(random_state(nodes, 5, 1.0e-2, 1.0e5)))
    rate = s.rhs()
    dt = 0.0123456789   # not a power of two
    s.rk_stage(0, dt)
    want = torch.tensor(dt, dtype=s.dtype, device=rate.device) * rate
    assert torch.equal(s.view(s.dq, 9), want)


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nodes,extent", [((36, 22, 40), (20000.0, 13000.0, 15000.0)),
                                          ((47, 31, 20), (7000.0, 9500.0, 5000.0))])
def test_strain_rates_on_topography_maps_round_once_per_product(precision, nodes, extent):
    """Order 2 with velocities linear in the node index and lambda = 0: the derivative times N - 1 is a
    whole number, so that sigma_xx and sigma_yy away from the faces are mu/J a (N - 1) dv with one rounding
    per product of the kernel's (and one for a_r = c a_q,x), bit for bit."""
    from paper_2011_02600_gb300.workload_setup import build_solver
    cfg = dataclasses.replace(config_by_name("hill129_o6"), nodes=nodes, extent=extent, order=2)
    s, _ = build_solver(cfg, precision=precision, keep_metrics=True)
    assert s.map_path() == "topography"
    s.view(s.mat, 3)[1].zero_()                              # lambda / J
    jq, mu2 = s.view(s.met, 9)[0], 2 * s.view(s.mat, 3)[2]
    jm = s.view(s.jmet, 10)
    c = (jm[5, 0, 0, 0] / jm[1, 0, 0, 0]).to(s.dtype)
    inner = (slice(2, -2),) * 3
    for f in (1, 3, 5, 7, 11, 25):
        Q = torch.zeros(9, *reversed(nodes), dtype=s.dtype)
        Q[0] = f * torch.arange(nodes[0], dtype=s.dtype)
        Q[1] = f * torch.arange(nodes[1], dtype=s.dtype)[:, None]
        rate = s.rhs(Q)
        for row, a, n in ((3, jq, nodes[0]), (4, c * jq, nodes[1])):
            assert torch.equal(rate[row][inner], (mu2 * (a * (f * (n - 1.0))))[inner]), (f, row)
