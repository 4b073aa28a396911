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
