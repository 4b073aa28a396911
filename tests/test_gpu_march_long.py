"""Marches of more steps than one multi-step launch takes: buffers, history
rotation and counters from one launch to the next, in the forward direction,
in both forms of the adjoint and in a replayed graph; and the benchmark's
workload at full size."""
import numpy as np
import pytest
import torch

from gpu_helpers import oracle_forward, rel_l2
from rte_inputs import workload_custom, workload_tomo256

pytestmark = pytest.mark.gpu

TF32X3, TF32, BF16X3 = 1, 2, 3
TOL = 1e-5                    # curves and fluence against the oracle, as test_gpu_forward


def _solver(wl, precision=TF32X3, **kw):
    from paper_2202_09421_gb300.solver import FCDOMSolver
    dev = torch.device("cuda:0")
    return FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                       torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=precision, **kw)


def _wl(nx, ny, M, groups, steps):
    return workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=80.0, n_groups=groups, t_s=0.3, sigma_t=0.15)


@pytest.mark.parametrize("nx,ny,M,groups,prec,steps", [(136, 24, 16, 1, TF32X3, 301), (150, 140, 32, 2, TF32, 300),
                                                       (24, 136, 64, 1, BF16X3, 257)])
def test_many_launches_equal_two_passes_a_step(nx, ny, M, groups, prec, steps):
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(nx, ny, M, groups, steps)
    out, launches = [], []
    for timed in (False, True):
        s = _solver(wl, prec)
        B.rte_set_pass_variant(s.ctx, 1)
        B.rte_set_kernel_timing(s.ctx, timed)
        before = s.kernel_launches()
        s.forward(wl.groups, steps)
        launches.append(s.kernel_launches() - before)
        out.append([s.readout(wl.detectors)] + [s.state(g) for g in range(groups)])
        s.close()
    assert 4 <= launches[0] <= steps // 16 and launches[1] == 2 * steps
    assert float(out[0][1].abs().max()) > 0
    assert all(torch.equal(x, y) for x, y in zip(*out))


# two marches in one launch and, with more groups, in turn; segments of more
# levels than a launch takes, the last one shorter
@pytest.mark.parametrize("nx,ny,M,groups,steps,ckpt", [(256, 150, 32, 1, 170, 100), (160, 136, 16, 24, 120, 70)])
def test_long_segments_of_the_marched_adjoint(nx, ny, M, groups, steps, ckpt):
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(nx, ny, M, groups, steps)
    out, launches = [], []
    for timed in (False, True):
        s = _solver(wl, ckpt_interval=ckpt)
        B.rte_set_pass_variant(s.ctx, 1)
        B.rte_set_kernel_timing(s.ctx, timed)
        s.forward(wl.groups, steps)
        meas = 0.5 * s.readout(wl.detectors)
        before = s.kernel_launches()
        out.append(s.adjoint_gradient(wl.detectors, meas))
        launches.append(s.kernel_launches() - before)
        s.close()
    assert launches[0] < steps < launches[1]
    (J, ga, gb), (J1, ga1, gb1) = out
    assert J == J1 > 0
    # FP64 sums over bitwise equal states (their order may differ)
    for x, y in ((ga, ga1), (gb, gb1)):
        assert torch.linalg.norm(x - y) <= 1e-6 * torch.linalg.norm(y)


def test_graph_replay_of_a_march_in_many_launches():
    from paper_2202_09421_gb300 import binding as B
    wl = _wl(256, 150, 32, 2, 75)
    out = []
    for flags in (0, B.RTE_FLAG_CUDA_GRAPH):
        s = _solver(wl, flags=flags, ckpt_interval=40)
        for _ in range(3):
            s.forward(wl.groups, wl.n_steps)
            curves = s.readout(wl.detectors)
            out.append([curves] + [s.state(g) for g in range(2)] + list(s.adjoint_gradient(wl.detectors, 0.5 * curves)[1:]))
        assert s.graph_captures() == (1 if flags else 0)
        s.close()
    assert float(out[0][1].abs().max()) > 0
    for o in out[1:]:
        assert all(torch.equal(x, y) for x, y in zip(o, out[0]))


def test_tomo256_in_the_schedule_of_the_benchmark():
    """256 x 256, M = 32, 16 sources, 3xTF32 in the schedule that the autotuner
    picks there (multi-step launches of the one-tile schedule).  (1) The first
    and the last source over 60 steps (the oracle's bounded sample) against
    the oracle.  (2) Over all 2000 steps a source's curves equal those of a
    march of that source alone, whose items are cut otherwise, bit for bit."""
    from paper_2202_09421_gb300 import binding as B

    def solver(wl):
        s = _solver(wl)
        B.rte_set_pass_variant(s.ctx, 1)
        return s

    short = workload_tomo256(n_steps=60)
    s = solver(short)
    before = s.kernel_launches()
    fl = s.forward(short.groups, short.n_steps, [59]).cpu().numpy()
    assert s.kernel_launches() - before < short.n_steps
    curves = s.readout(short.detectors).cpu().numpy()
    s.close()
    c_ref, f_ref, _ = oracle_forward(short, groups=[short.groups[0], short.groups[-1]], snaps=[59])
    for k, gi in enumerate((0, len(short.groups) - 1)):
        assert rel_l2(curves[gi], c_ref[k]) <= TOL and rel_l2(fl[gi], f_ref[k]) <= TOL

    full = workload_tomo256()
    s = solver(full)
    s.forward(full.groups, full.n_steps)
    together = s.readout(full.detectors).cpu().numpy()
    s.close()
    assert np.isfinite(together).all() and together.max() > 0
    for gi in (0, 7, 15):
        s = solver(full)
        s.forward([full.groups[gi]], full.n_steps)
        assert np.array_equal(s.readout(full.detectors).cpu().numpy()[0], together[gi]), gi
        s.close()
