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
