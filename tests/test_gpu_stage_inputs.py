"""sbp_stage_inputs against the same stages run one by one through the bound buffers.

The two run the same kernels on the same values, from other addresses: they agree bit for bit,
with the last row of tiles and chunks ragged, with a source, for a batch and on both kernel paths."""
import numpy as np
import pytest
import torch

from test_gpu_adjoint import _batched_problem, _misfit_case, _set, _three_sources

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,nodes", [(2, (21, 18, 16)), (4, (33, 19, 30)), (6, (64, 30, 27))])
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("batch", [1, 3])
def test_stage_inputs_match_the_stages(order, nodes, prec, path, batch):
    from paper_2011_02600_gb300 import _lib as L
    c = _misfit_case(nsteps=4, order=order, nodes=nodes)
    p, _ = _batched_problem(c, _three_sources()[:batch], prec, path)
    _set(p, c["mat"])
    s, st = p.s, torch.cuda.current_stream().cuda_stream
    p.forward()                                            # a state that is not zero
    n = 9 * batch * s.fs
    u0 = s.qbuf[s.current].clone()
    assert float(u0.abs().max()) > 0
    stages = s.new_fields(5 * 9 * batch)
    stages[:n].copy_(u0)
    s.set_time(3 * c["dt"], 3)
    L.sbp_stage_inputs(s.h, c["dt"], stages, st)
    assert torch.equal(s.qbuf[s.current], u0)              # the bound state is not touched
    for k in range(5):
        assert torch.equal(stages[k * n:(k + 1) * n], s.qbuf[s.current]), k
        L.sbp_rk_stage(s.h, k, c["dt"], st)
    assert s.status() == 0


def test_stage_inputs_refuse_bad_buffers():
    from paper_2011_02600_gb300 import _lib as L
    c = _misfit_case(nsteps=1)
    p, _ = _batched_problem(c, _three_sources()[:1])
    _set(p, c["mat"])
    buf = p.s.new_fields(46)
    for bad in (None, buf[2:], p.s.qbuf[0], p.s.dq):
        with pytest.raises(L.SbpError):
            L.sbp_stage_inputs(p.s.h, c["dt"], bad, None)
    for dt in (0.0, float("nan")):
        with pytest.raises(L.SbpError):
            L.sbp_stage_inputs(p.s.h, dt, buf, None)


def test_gradient_leaves_the_solver_after_the_first_step():
    """What the solver holds after gradient() is the state after step 1, at time 0, as before."""
    c = _misfit_case(nsteps=9)
    p, _ = _batched_problem(c, _three_sources()[:2])
    _set(p, c["mat"])
    p.forward()
    p.gradient()
    left = p.s.qbuf[p.s.current].clone()
    assert p.s.time == 0.0
    p._reset()
    p.s.step(1, c["dt"])
    assert np.array_equal(left.cpu().numpy(), p.s.qbuf[p.s.current].cpu().numpy())


@pytest.mark.parametrize("batch", [1, 2])
def test_stage_inputs_refuse_a_buffer_that_overlaps_a_bound_one(batch):
    """Refused before any launch: a buffer that starts inside a bound one, at its first and its last
    aligned address, or that runs into one.  The bytes behind the addresses are not touched."""
    from paper_2011_02600_gb300 import _lib as L
    c = _misfit_case(nsteps=1)
    p, _ = _batched_problem(c, _three_sources()[:batch])
    _set(p, c["mat"])
    s = p.s
    field = s.fs * s.met.element_size()
    state = 9 * batch * field
    for buf, size in ((s.qbuf[0], state), (s.qbuf[1], state), (s.dq, state), (s.met, 9 * field), (s.mat, 3 * field)):
        base = buf.data_ptr()
        for at in (base, base + 256, base + size - 256, base - 5 * state + 256):
            with pytest.raises(L.SbpError) as e:
                L.sbp_stage_inputs(s.h, c["dt"], at, None)
            assert e.value.code == 1 and "overlap" in str(e.value)
