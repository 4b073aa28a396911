"""The multi-step launch of the tensor-core passes against the two launches
per step of the same schedule (which kernel timing selects): the same splits,
MMAs and epilogue arithmetic in the same order, so states, curves and
fluence are bit for bit the same."""
import numpy as np
import pytest
import torch

from rte_inputs import workload_custom

pytestmark = pytest.mark.gpu

TF32X3, TF32, BF16X3, BF16 = 1, 2, 3, 4


# sizes: one and two row tiles, ragged ends, a short other axis (items of a
# single unit), two lines per tile (M = 64), more items than SMs; odd and even
# step counts; snapshots and checkpoints that cut the march into runs; segments
# longer than one launch of the reverse sweep
@pytest.mark.parametrize("nx,ny,M,groups,steps,prec", [
    (129, 129, 32, 1, 7, TF32X3), (256, 256, 32, 7, 9, TF32X3), (203, 131, 16, 2, 12, TF32),
    (256, 24, 32, 3, 11, BF16X3), (24, 256, 16, 40, 6, TF32X3), (140, 300, 64, 2, 5, BF16X3),
    (300, 40, 64, 1, 8, BF16), (136, 24, 16, 1, 90, TF32X3)])
def test_multi_step_launch_matches_two_launches_per_step(nx, ny, M, groups, steps, prec):
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import FCDOMSolver
    wl = workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=80.0, n_groups=groups, t_s=0.1, sigma_t=0.1)
    snaps = [3, steps - 1]
    dev = torch.device("cuda:0")
    out = []
    for two_launches in (False, True):
        s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                        torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=prec,
                        ckpt_interval=4 if steps < 40 else 40)
        B.rte_set_pass_variant(s.ctx, 1)
        if two_launches:
            B.rte_set_kernel_timing(s.ctx, True)
        before = B.rte_kernel_launches(s.ctx)
        fl = s.forward(wl.groups, wl.n_steps, snaps).cpu().numpy()
        launches = B.rte_kernel_launches(s.ctx) - before
        curves = s.readout(wl.detectors)
        states = [s.state(g).cpu().numpy() for g in range(groups)]
        J, ga, gb = s.adjoint_gradient(wl.detectors, torch.zeros_like(curves))
        out.append((curves.cpu().numpy(), fl, states, ga.cpu().numpy(), gb.cpu().numpy(), launches))
        s.close()
    a, b = out
    assert a[5] < b[5]                                   # the two sides took different paths
    assert np.abs(a[0]).max() > 0 and all(np.abs(u).max() > 0 for u in a[2])
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert all(np.array_equal(x, y) for x, y in zip(a[2], b[2]))
    # FP64 sums over bitwise equal recomputed states (their order may differ)
    for k in (3, 4):
        assert np.linalg.norm(a[k] - b[k]) <= 1e-7 * np.linalg.norm(b[k])


@pytest.mark.parametrize("steps,ckpt", [(13, 0), (9, 1), (10, 3)])
def test_photon_balance_of_a_multi_step_launch(steps, ckpt):
    """The balance of every step, from states in slots, against single passes;
    runs of one step (a checkpoint at each) and of four."""
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import FCDOMSolver
    wl = workload_custom(150, 40, 32, steps, 0.02, L=149 / 66, mus=80.0, n_groups=2, t_s=0.1, sigma_t=0.1)
    dev = torch.device("cuda:0")
    out = []
    for two_launches in (False, True):
        s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                        torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=TF32X3,
                        ckpt_interval=ckpt, flags=B.RTE_FLAG_PHOTON_BALANCE)
        B.rte_set_pass_variant(s.ctx, 1)
        if two_launches:
            B.rte_set_kernel_timing(s.ctx, True)
        before = B.rte_kernel_launches(s.ctx)
        s.forward(wl.groups, steps)
        launches = B.rte_kernel_launches(s.ctx) - before
        out.append((s.photon_balance().cpu().numpy(), s.state(1).cpu().numpy(), s.readout(wl.detectors).cpu().numpy(),
                    launches))
        s.close()
    a, b = out
    assert a[3] < b[3] and np.abs(a[0]).max() > 0
    assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3]))


@pytest.mark.parametrize("M,prec,steps,sizes", [
    (32, TF32X3, 7, [(200, 140, 2), (48, 64, 1), (129, 40, 3), (300, 260, 1)]),
    (16, BF16X3, 6, [(24, 260, 1), (257, 129, 2)]), (64, TF32, 5, [(140, 36, 1), (40, 300, 2)])])
def test_batched_persistent_passes_match_each_medium_alone(M, prec, steps, sizes):
    """Media with lines of more than 128 positions in one batch: the items of
    all of them in one persistent launch per pass, states alternating between
    two buffers (odd and even step counts, checkpoints from either)."""
    from paper_2202_09421_gb300 import binding as B
    from paper_2202_09421_gb300.solver import FCDOMSolver, adjoint_gradient_batch, forward_batch
    dev = torch.device("cuda:0")
    wls = [workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=80.0 - 10 * k, n_groups=g, t_s=0.1,
                           sigma_t=0.1, g=0.9 - 0.1 * k) for k, (nx, ny, g) in enumerate(sizes)]
    ss = [FCDOMSolver(w.grid, w.optics, torch.tensor(w.mua, dtype=torch.float32, device=dev),
                      torch.tensor(w.mus, dtype=torch.float32, device=dev), w.c, w.dt, precision=prec,
                      ckpt_interval=3) for w in wls]
    before = B.rte_kernel_launches(ss[0].ctx)
    forward_batch(ss, [w.groups for w in wls], steps)
    assert B.rte_kernel_launches(ss[0].ctx) - before == 2 * steps
    curves = [s.readout(w.detectors) for s, w in zip(ss, wls)]
    states = [[s.state(g).cpu().numpy() for g in range(len(w.groups))] for s, w in zip(ss, wls)]
    grads = adjoint_gradient_batch(ss, [w.detectors for w in wls], [0.5 * c for c in curves])
    for s, w, c, us, (J, ga, gb) in zip(ss, wls, curves, states, grads):
        s.forward(w.groups, steps)
        assert torch.equal(s.readout(w.detectors), c)
        for g, u in enumerate(us):
            assert np.abs(u).max() > 0 and np.array_equal(s.state(g).cpu().numpy(), u)
        J1, ga1, gb1 = s.adjoint_gradient(w.detectors, 0.5 * c)
        assert J == J1
        assert torch.allclose(ga, ga1, rtol=1e-5, atol=0) and torch.allclose(gb, gb1, rtol=1e-5, atol=0)
        s.close()
