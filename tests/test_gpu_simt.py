"""The FP32 passes at the edges of their tiles: thread tiles of 4 x 4 and
8 x 8 outputs, lines that end inside a chunk or a thread tile, the last line
tile partly filled or one line wide, ordinate counts that do not divide a
tile, one tile per pass, the longest line."""
import numpy as np
import pytest
import torch

from gpu_helpers import gpu_forward, oracle_forward, rel_l2
from rte_inputs import workload_custom

pytestmark = pytest.mark.gpu
TOL = 1e-5                    # of the other FP32 tests: rounding through the march stays below 1e-6


# 64 * 256 * 152 outputs and more take the 8 x 8 form; so do lines too long
# for 512 threads of 4 x 4 outputs (512 positions of M > 16, 256 of M > 32).
# Two beams in the first case's first group (only the first one's source is
# staged ahead).
@pytest.mark.parametrize("nx,ny,M,groups,steps", [
    (17, 33, 8, 2, 40), (16, 130, 40, 1, 30), (31, 16, 64, 5, 30), (129, 65, 56, 6, 10),
    (100, 101, 24, 11, 12), (260, 24, 48, 1, 12), (512, 17, 16, 1, 8), (33, 512, 64, 3, 6)])
def test_fp32_tiles_match_oracle(nx, ny, M, groups, steps):
    wl = workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=40.0, n_groups=groups, t_s=0.2, sigma_t=0.1)
    if M == 8:
        wl.groups = [[b for g in wl.groups for b in g]] + list(wl.groups[1:])
    s, _, curves = gpu_forward(wl)
    c_ref, _, u_ref = oracle_forward(wl)
    umax = max(np.abs(u).max() for u in u_ref)
    assert umax > 0 and np.abs(c_ref).max() > 0
    # so few steps after the pulse the curves are far below the state: their
    # rounding is that of the boundary values (1e-6 of the largest) times the
    # ordinate weights (at most 2 in sum) and the window (2 sigma_d)
    assert np.abs(curves - c_ref).max() <= 4 * wl.detectors[0].sigma_d * 1e-6 * umax
    for g in range(len(wl.groups)):
        assert rel_l2(s.state(g).cpu().numpy(), np.moveaxis(u_ref[g], 0, -1)) <= TOL
    s.close()


@pytest.mark.parametrize("nx,ny,M,groups", [(100, 101, 24, 11), (72, 90, 56, 7)])
def test_fp32_tile_forms_agree(nx, ny, M, groups):
    """Forward, continuous and discrete gradient of all groups at once (8 x 8
    outputs a thread) against the sum over the groups alone (4 x 4)."""
    from paper_2202_09421_gb300.solver import FCDOMSolver
    wl = workload_custom(nx, ny, M, 90, 0.02, mus=20.0, n_groups=groups, t_s=0.5, sigma_t=0.2)
    dev = torch.device("cuda:0")
    s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                    torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, ckpt_interval=40)
    s.forward(wl.groups, wl.n_steps)
    curves = s.readout(wl.detectors)
    meas = 0.5 * curves
    both = [s.discrete_adjoint_gradient(wl.detectors, meas)]
    s.forward(wl.groups, wl.n_steps)
    both.append(s.adjoint_gradient(wl.detectors, meas))
    parts = [[0.0, 0.0, 0.0], [0.0, 0.0, 0.0]]
    for g in range(groups):
        for k, fn in enumerate((s.discrete_adjoint_gradient, s.adjoint_gradient)):
            s.forward(wl.groups[g:g + 1], wl.n_steps)
            assert rel_l2(s.readout(wl.detectors).cpu(), curves[g:g + 1].cpu()) <= TOL
            out = fn(wl.detectors, meas[g:g + 1].contiguous())
            parts[k] = [p + (o.double().cpu() if torch.is_tensor(o) else o) for p, o in zip(parts[k], out)]
    for (J, ga, gb), (J1, ga1, gb1) in zip(both, parts):
        assert J > 0 and abs(J - J1) <= TOL * J
        assert rel_l2(ga.cpu(), ga1) <= TOL and rel_l2(gb.cpu(), gb1) <= TOL
    s.close()


# The exitance partial sums of each form, at detectors on the beams themselves:
# there the back-scattered light of every group is 1e-5 to 1e-4 of its state
# within a few steps, far above the absolute rounding of the boundary values,
# and its sums are of products of one sign, so that the relative bound of the
# other FP32 tests holds group by group.
@pytest.mark.parametrize("nx,ny,M,groups,steps", [(33, 512, 64, 3, 24), (129, 65, 56, 6, 12), (100, 101, 24, 11, 12),
                                                  (16, 130, 40, 2, 24)])
def test_fp32_exitance_of_every_group(nx, ny, M, groups, steps):
    from rte_inputs import Detector
    wl = workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=40.0, n_groups=groups, t_s=0.1, sigma_t=0.1)
    wl.detectors = [Detector(g[0].x, g[0].y, 0.1) for g in wl.groups]
    s, _, curves = gpu_forward(wl)
    c_ref, _, u_ref = oracle_forward(wl)
    s.close()
    for g in range(groups):
        assert np.abs(c_ref[g]).max() > 1e-5 * np.abs(u_ref[g]).max()
        assert rel_l2(curves[g], c_ref[g]) <= TOL
