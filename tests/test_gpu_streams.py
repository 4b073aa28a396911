"""Solves side by side on streams of their own.  A multi-step launch keeps
every SM, so a march beside others takes the passes (which overlap), and the
results do not depend on what runs beside it."""
import threading
import time

import pytest
import torch

from rte_inputs import workload_custom

pytestmark = pytest.mark.gpu

FP32, TF32X3 = 0, 1
LATELY = 0.1                  # seconds after which a march beside another is forgotten


@pytest.fixture(autouse=True)
def forgotten():
    yield
    time.sleep(LATELY)                                   # other tests count the launches of a march alone


def _wl(nx, ny, M, groups, steps):
    return workload_custom(nx, ny, M, steps, 0.02, L=(nx - 1) / 66, mus=80.0, n_groups=groups, t_s=0.1, sigma_t=0.1)


def _solver(wl, precision, **kw):
    from paper_2202_09421_gb300.solver import FCDOMSolver
    dev = torch.device("cuda:0")
    s = FCDOMSolver(wl.grid, wl.optics, torch.tensor(wl.mua, dtype=torch.float32, device=dev),
                    torch.tensor(wl.mus, dtype=torch.float32, device=dev), wl.c, wl.dt, precision=precision, **kw)
    s.stream = kw["stream"]
    torch.cuda.synchronize()
    return s


def _load_kernels(s, wl):
    """Both forms once: the first launch of a kernel loads it, which waits for
    the GPU to be idle."""
    from paper_2202_09421_gb300 import binding as B
    for timed in (True, False):
        B.rte_set_kernel_timing(s.ctx, timed)
        s.forward(wl.groups, wl.n_steps)
        s.adjoint_gradient(wl.detectors, torch.zeros_like(s.readout(wl.detectors)))


def _solve(s, wl, launches=None, snaps=()):
    before = s.kernel_launches()
    fl = s.forward(wl.groups, wl.n_steps, snaps)
    if launches is not None:
        launches.append(s.kernel_launches() - before)
    out = [s.readout(wl.detectors)] + [s.state(g) for g in range(len(wl.groups))]
    s.stream.synchronize()                               # the copies, before another stream reads them
    return out + [fl] if snaps else out


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("busy_steps,steps,graph", [(150, 20, False), (8, 4000, False), (150, 20, True)])
def test_a_march_beside_another_takes_the_passes(busy_steps, steps, graph):
    """An FP32 forward (which returns before its work is done) under way on
    another stream for all, or for a part, of the march."""
    from paper_2202_09421_gb300 import binding as B
    busy_wl, wl = _wl(512, 512, 64, 1, busy_steps), _wl(256, 150, 32, 1, steps)
    busy = _solver(busy_wl, FP32, stream=torch.cuda.Stream())
    s = _solver(wl, TF32X3, stream=torch.cuda.Stream(), ckpt_interval=70,
                flags=B.RTE_FLAG_CUDA_GRAPH if graph else 0)
    snaps = [] if graph else [3, steps - 1]
    alone, beside = [], []
    _load_kernels(s, wl)
    _solve(s, wl, alone, snaps)
    busy.forward(busy_wl.groups, busy_wl.n_steps)
    torch.cuda.synchronize()
    alone.clear()
    time.sleep(LATELY)
    ref = _solve(s, wl, alone, snaps)
    torch.cuda.synchronize()
    busy.forward(busy_wl.groups, busy_wl.n_steps)
    out = _solve(s, wl, beside, snaps)
    torch.cuda.synchronize()
    assert float(ref[1].abs().max()) > 0 and _same(out, ref)
    assert alone[0] < steps                              # multi-step launches
    if busy_steps == 150:
        assert beside[0] >= 2 * steps                    # the passes throughout
    else:
        assert alone[0] < beside[0] < 2 * steps          # first the passes, then launches
    again = []
    time.sleep(LATELY)
    assert _same(_solve(s, wl, again, snaps), ref) and again == alone
    s.close()
    busy.close()


@pytest.mark.parametrize("groups,busy_steps", [(1, 300), (1, 25), (3, 40)])
def test_a_gradient_beside_another_march(groups, busy_steps):
    busy_wl, wl = _wl(512, 512, 64, 1, busy_steps), _wl(256, 150, 32, groups, 721)
    busy = _solver(busy_wl, FP32, stream=torch.cuda.Stream())
    s = _solver(wl, TF32X3, stream=torch.cuda.Stream(), ckpt_interval=24)
    _load_kernels(s, wl)
    busy.forward(busy_wl.groups, busy_wl.n_steps)
    torch.cuda.synchronize()
    s.forward(wl.groups, wl.n_steps)
    meas = 0.5 * s.readout(wl.detectors)
    torch.cuda.synchronize()
    results = []
    for beside in (False, True, False):
        s.forward(wl.groups, wl.n_steps)
        torch.cuda.synchronize()
        time.sleep(LATELY)
        if beside:
            busy.forward(busy_wl.groups, busy_wl.n_steps)
        results.append(s.adjoint_gradient(wl.detectors, meas))
        torch.cuda.synchronize()
    for J, ga, gb in results[1:]:
        assert J == results[0][0] > 0
        for x, y in ((ga, results[0][1]), (gb, results[0][2])):
            assert torch.linalg.norm(x - y) <= 1e-6 * torch.linalg.norm(y)
    assert torch.equal(results[0][1], results[2][1])
    s.close()
    busy.close()


def test_threads_with_solvers_of_their_own():
    """Five threads, each with its stream and solver, forward and gradient
    again and again, against the same calls one after another."""
    wls = [_wl(256, 150, 32, 1, 80), _wl(200, 131, 32, 2, 50), _wl(300, 64, 64, 1, 60), _wl(64, 64, 16, 2, 90),
           _wl(256, 256, 32, 1, 70)]
    streams = [torch.cuda.Stream() for _ in wls]
    solvers = [_solver(w, TF32X3, stream=st, ckpt_interval=16) for w, st in zip(wls, streams)]

    def call(k):
        with torch.cuda.stream(streams[k]):
            out = _solve(solvers[k], wls[k])
            J, ga, gb = solvers[k].adjoint_gradient(wls[k].detectors, 0.5 * out[0])
            streams[k].synchronize()
        return out, J, ga, gb

    ref = [call(k) for k in range(len(wls))]
    got = [[] for _ in wls]

    def work(k):
        for _ in range(4):
            got[k].append(call(k))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(wls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k, (out, J, ga, gb) in enumerate(ref):
        assert len(got[k]) == 4 and J > 0
        for o, j, a, b in got[k]:
            assert _same(o, out) and j == J
            assert torch.linalg.norm(a - ga) <= 1e-6 * torch.linalg.norm(ga)
            assert torch.linalg.norm(b - gb) <= 1e-6 * torch.linalg.norm(gb)
    for s in solvers:
        s.close()
