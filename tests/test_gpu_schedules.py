"""Every kernel schedule rounds alike: the same splits, products and sums in
the same order, exitance included, so states and detector curves do not
depend on the schedule."""
import pytest
import torch

from rte_inputs import workload_custom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,M,groups,prec", [(64, 64, 16, 2, 1), (100, 90, 32, 3, 1), (128, 72, 32, 2, 3),
                                                 (200, 131, 32, 1, 2), (40, 64, 64, 1, 3)])
def test_schedules_agree_bit_for_bit(nx, ny, M, groups, prec):
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import FCDOMSolver
    wl = workload_custom(nx, ny, M, 60, 0.02, L=(nx - 1) / 66, mus=40.0, n_groups=groups, t_s=0.3, sigma_t=0.1)
    dev = torch.device("cuda:0")
    out = {}
    for variant in (1, 0, 2, 4, 5):
        s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                        torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=prec)
        B.rte_set_pass_variant(s.ctx, variant)
        s.forward(wl.groups, wl.n_steps)
        out[variant] = [s.readout(wl.detectors)] + [s.state(g) for g in range(groups)]
        s.close()
    assert float(out[1][0].abs().max()) > 0
    for variant, arrays in out.items():
        assert all(torch.equal(x, y) for x, y in zip(arrays, out[1])), variant


@pytest.mark.parametrize("nx,ny,M,groups,prec,marched", [
    (256, 256, 32, 1, 1, True), (512, 40, 64, 1, 1, True), (200, 131, 32, 3, 2, True), (170, 300, 32, 2, 3, True),
    (24, 256, 16, 40, 1, False), (260, 24, 32, 16, 2, False), (130, 130, 16, 16, 2, False), (206, 21, 32, 22, 4, False)])
def test_multi_step_launches_by_size(nx, ny, M, groups, prec, marched):
    """A context whose schedule nobody set takes the multi-step launches where
    they are faster; set to schedule 1, wherever they are supported.  The
    results are the same bits."""
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import FCDOMSolver
    wl = workload_custom(nx, ny, M, 9, 0.02, L=(nx - 1) / 66, mus=40.0, n_groups=groups, t_s=0.1, sigma_t=0.05)
    dev = torch.device("cuda:0")
    out = []
    for explicit in (False, True):
        s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                        torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=prec)
        if explicit:
            B.rte_set_pass_variant(s.ctx, 1)
        before = B.rte_kernel_launches(s.ctx)
        s.forward(wl.groups, wl.n_steps)
        launches = B.rte_kernel_launches(s.ctx) - before
        assert (launches < 2 * wl.n_steps) == (explicit or marched)
        out.append([s.readout(wl.detectors)] + [s.state(g) for g in range(groups)])
        s.close()
    assert float(out[0][1].abs().max()) > 0
    assert all(torch.equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("groups,snaps", [(1, [0, 1, 2, 5]), (3, [0, 1, 4, 5, 8]), (3, [2, 3])])
def test_runs_too_short_for_a_multi_step_launch(groups, snaps):
    """Runs cut short by snapshots and checkpoints take the passes, between
    longer ones that do not: states alternate between the buffers and end in
    the right one, whatever the mixture."""
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import FCDOMSolver
    wl = workload_custom(256, 160, 32, 12, 0.02, L=255 / 66, mus=40.0, n_groups=groups, t_s=0.1, sigma_t=0.05)
    dev = torch.device("cuda:0")
    out = []
    for timed in (False, True):                       # kernel timing takes two passes every step
        s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                        torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=1, ckpt_interval=5)
        if timed:
            B.rte_set_kernel_timing(s.ctx, True)
        fl = s.forward(wl.groups, wl.n_steps, snaps)
        curves = s.readout(wl.detectors)
        states = [s.state(g) for g in range(groups)]
        out.append([fl, curves] + states + list(s.adjoint_gradient(wl.detectors, 0.5 * curves)[1:]))
        s.close()
    assert float(out[0][2].abs().max()) > 0
    assert all(torch.equal(x, y) for x, y in zip(out[0][:-2], out[1][:-2]))
    for x, y in zip(out[0][-2:], out[1][-2:]):
        assert torch.linalg.norm(x - y) <= 1e-6 * torch.linalg.norm(y)
