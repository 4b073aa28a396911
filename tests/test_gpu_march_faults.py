"""Failure reporting of the multi-step launches (lines of more than 128
positions), with the fault made on the host: the call reports TIMEOUT, does
no work, and the next one on the same context is right."""
import pytest
import torch

from rte_inputs import workload_custom

pytestmark = pytest.mark.gpu

TF32X3, TIMEOUT = 1, 5


def _wl(nx, ny, groups, steps=6, M=32):
    return workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=80.0, n_groups=groups, t_s=0.1, sigma_t=0.1)


def _solver(wl, **kw):
    from paper_2202_09421_gb300.solver import FCDOMSolver
    dev = torch.device("cuda:0")
    return FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                       torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=TF32X3, **kw)


def _timeout(fn, *args):
    from paper_2202_09421_gb300.binding import RTEError
    with pytest.raises(RTEError) as e:
        fn(*args)
    assert e.value.status == TIMEOUT


def _results(s, wl):
    s.forward(wl.groups, wl.n_steps)
    return [s.readout(wl.detectors)] + [s.state(g) for g in range(len(wl.groups))]


@pytest.mark.parametrize("groups,balance", [(1, False), (3, True)])
def test_timeout_word_stops_a_multi_step_launch(groups, balance):
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(136, 40, groups)
    flags = B.RTE_FLAG_PHOTON_BALANCE if balance else 0
    s, clean = _solver(wl, flags=flags), _solver(wl, flags=flags)
    B.rte_inject_fault(s.ctx, B.RTE_FAULT_TIMEOUT_WORD)
    _timeout(s.forward, wl.groups, wl.n_steps)
    state = torch.empty((wl.grid.ny, wl.grid.nx, wl.grid.M), dtype=torch.float32, device="cuda:0")
    B.rte_get_state(s.ctx, 0, state)
    assert float(state.abs().max()) == 0.0
    assert all(torch.equal(x, y) for x, y in zip(_results(s, wl), _results(clean, wl)))
    if balance:
        assert torch.equal(s.photon_balance(), clean.photon_balance())
    s.close()
    clean.close()


@pytest.mark.parametrize("groups", [1, 24])              # two marches in one launch, and in turn
def test_timeout_word_stops_the_marched_adjoint(groups):
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(200, 136, groups, steps=9, M=16)
    s = _solver(wl, ckpt_interval=4)
    s.forward(wl.groups, wl.n_steps)
    meas = 0.5 * s.readout(wl.detectors)
    good = s.adjoint_gradient(wl.detectors, meas)
    s.forward(wl.groups, wl.n_steps)
    B.rte_inject_fault(s.ctx, B.RTE_FAULT_TIMEOUT_WORD)
    _timeout(s.adjoint_gradient, wl.detectors, meas)
    s.forward(wl.groups, wl.n_steps)
    again = s.adjoint_gradient(wl.detectors, meas)
    assert good[0] == again[0] > 0
    assert torch.equal(good[1], again[1]) and torch.equal(good[2], again[2])
    s.close()


def test_timeout_word_of_one_medium_of_a_batch():
    """The word of one medium: the batch reports TIMEOUT, that medium's state
    stays at its zero start, and the others' curves are their own."""
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import forward_batch
    wls = [_wl(136, 40, 1, steps=5), _wl(48, 64, 2, steps=5), _wl(150, 140, 1, steps=5)]
    for k in range(3):
        ss = [_solver(w) for w in wls]
        B.rte_inject_fault(ss[k].ctx, B.RTE_FAULT_TIMEOUT_WORD)
        _timeout(forward_batch, ss, [w.groups for w in wls], 5)
        for i, (s, w) in enumerate(zip(ss, wls)):
            s.n_groups, s.n_steps = len(w.groups), 5
            curves, u = s.readout(w.detectors), s.state(0)
            if i == k:
                assert float(u.abs().max()) == 0.0
            fresh = _results(s, w)
            if i != k:
                assert torch.equal(curves, fresh[0]) and torch.equal(u, fresh[1])
            assert float(fresh[1].abs().max()) > 0
            s.close()


@pytest.mark.parametrize("groups,balance", [(1, False), (2, True), (12, False)])
def test_expiring_wait_of_a_multi_step_launch(groups, balance):
    """One CTA's wait runs out (about 2 s) while the others copy, multiply and
    wait for its item: every role gives up, what is in flight is drained, the
    call reports TIMEOUT after one launch's work, and the next is right."""
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(150, 140, groups, steps=12)
    flags = B.RTE_FLAG_PHOTON_BALANCE if balance else 0
    s, clean = _solver(wl, flags=flags), _solver(wl, flags=flags)
    B.rte_set_pass_variant(s.ctx, 1)
    B.rte_inject_fault(s.ctx, B.RTE_FAULT_EXPIRE_WAIT)
    before = B.rte_kernel_launches(s.ctx)
    _timeout(s.forward, wl.groups, wl.n_steps)
    assert B.rte_kernel_launches(s.ctx) - before < (3 if balance else 2) * wl.n_steps      # not the single passes
    assert all(torch.equal(x, y) for x, y in zip(_results(s, wl), _results(clean, wl)))
    s.close()
    clean.close()


def test_expiring_wait_of_the_marched_adjoint():
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(160, 136, 2, steps=9)
    s = _solver(wl, ckpt_interval=4)
    B.rte_set_pass_variant(s.ctx, 1)
    s.forward(wl.groups, wl.n_steps)
    meas = 0.5 * s.readout(wl.detectors)
    good = s.adjoint_gradient(wl.detectors, meas)
    s.forward(wl.groups, wl.n_steps)
    B.rte_inject_fault(s.ctx, B.RTE_FAULT_EXPIRE_WAIT)
    _timeout(s.adjoint_gradient, wl.detectors, meas)
    s.forward(wl.groups, wl.n_steps)
    again = s.adjoint_gradient(wl.detectors, meas)
    assert good[0] == again[0] > 0
    assert torch.equal(good[1], again[1]) and torch.equal(good[2], again[2])
    s.close()


def _taken(fn):
    """Device memory that a call leaves allocated."""
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    fn()
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("balance,ckpt", [(False, 20), (True, 0)])
def test_multi_step_launches_take_no_states_of_their_own(balance, ckpt):
    """A forward keeps the state, its scratch, three histories and four states
    per checkpoint; a gradient two segments, the adjoint state, its scratch
    and three histories.  The multi-step launches add none (a few MB of tables
    and the allocator's granules aside)."""
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(256, 256, 3, steps=41)
    s = _solver(wl, ckpt_interval=ckpt, flags=B.RTE_FLAG_PHOTON_BALANCE if balance else 0)
    state = 3 * 256 * 256 * 32 * 4
    n_ckpt = 3 if ckpt else 0
    assert _taken(lambda: s.forward(wl.groups, wl.n_steps)) <= (5 + 4 * n_ckpt) * state + state
    if ckpt:
        meas = torch.zeros_like(s.readout(wl.detectors))
        assert _taken(lambda: s.adjoint_gradient(wl.detectors, meas)) <= (2 * ckpt + 5) * state + state
    s.close()
