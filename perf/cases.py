"""Performance cases: what a program that uses this library has it do, through its public entry points.

The cases stand for forward solves (the library's default FP32 form and the tensor-core forms users pick for speed),
the two adjoint gradients, the batched solve of many media, and the decomposed operator's fused step, each at sizes
that the repository's workloads, tests and benchmark use: from a 64 x 64 grid with one source, where the latency of a
step counts, to the 256 x 256 tomography with 16 sources and the 512 x 512, 64-ordinate medium, with ragged grids in
between.  The pulse widths are scaled to the simulated time, so that light is moving through the medium.

`exact` is a plain FP64 torch restatement of the method (dense FC derivative, AB4, Fresnel boundary, readout, adjoint),
sharing no code with the package; the media are rounded to FP32 first, as the library receives them."""
import dataclasses
import math

import numpy as np
import torch

from paper_2202_09421_gb300 import binding as B
from paper_2202_09421_gb300.solver import FCDOMSolver, RTEObjective, forward_batch
from rte_inputs import (Beam, Grid, Optics, Workload, face_point, perimeter_detectors, workload_custom, workload_inverse,
                        workload_mss256, workload_precision512, workload_small, workload_tomo256)
from rte_inputs.workloads import C0_CM_PER_PS, neck_medium

FP32, TF32X3, TF32, BF16X3 = B.RTE_PREC_FP32, B.RTE_PREC_TF32X3, B.RTE_PREC_TF32, B.RTE_PREC_BF16X3
MAX_UPDATES = 1.2e9          # of a drawn case; the largest listed one has 1.6e9


def _case(kind, medium, precision, nx, ny, M, groups, steps, name=None, **more):
    c = {"kind": kind, "medium": medium, "precision": precision, "nx": nx, "ny": ny, "M": M, "groups": groups,
         "steps": steps, "ckpt": 0, "parts": 1, "graph": False, "autotune": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest solve, in the library's default precision: launch and per-step latency
        _case("forward", "small", FP32, 64, 64, 16, 1, 200, "small64_fp32"),
        # the same grid at 3xTF32, captured as a CUDA graph and replayed (a fitting loop that solves again and again)
        _case("forward", "small", TF32X3, 64, 64, 16, 1, 200, "small64_tf32x3_graph", graph=True),
        # one source on the tomography grid: the latency of one solve at full resolution
        _case("forward", "tomo", TF32X3, 256, 256, 32, 1, 100, "tomo256_1src_tf32x3"),
        # the benchmark's workload: 16 sources at once, in the schedule that the autotuner picks
        _case("forward", "tomo", TF32X3, 256, 256, 32, 16, 48, "tomo256_16src_tf32x3", autotune=True),
        # default precision at the tomography size, four sources
        _case("forward", "tomo", FP32, 256, 256, 32, 4, 40, "tomo256_4src_fp32"),
        # a ragged grid and an ordinate count that only the FP32 kernels take
        _case("forward", "custom", FP32, 203, 131, 24, 3, 60, "ragged203x131_m24_fp32"),
        # a ragged grid in the reduced-precision single-product form
        _case("forward", "custom", TF32, 200, 131, 32, 3, 80, "ragged200x131_tf32"),
        # the 512 x 512, 64-ordinate medium with split BF16 operands
        _case("forward", "precision", BF16X3, 512, 512, 64, 1, 40, "precision512_bf16x3"),
        # the gradient of the tomography problem: forward, checkpoint recompute, continuous adjoint; 4 staggered groups
        _case("gradient", "mss", TF32X3, 256, 256, 32, 4, 60, "mss256_gradient_tf32x3", ckpt=20, autotune=True),
        # one evaluation of the inverse loop through autograd: 16 sources on 64 x 64, exact discrete gradient
        _case("autograd", "inverse", TF32X3, 64, 64, 32, 16, 100, "inverse64_autograd_exact", ckpt=50),
        # independent media of mixed sizes marched together, captured as a CUDA graph
        _case("batch", "neck", TF32X3, 0, 0, 32, 12, 30, "neck_batch12_tf32x3", graph=True),
        # the decomposed operator's tile-local fused step, 16 sources
        _case("forward", "tomo", FP32, 256, 256, 32, 16, 48, "fused256_16src_parts16", parts=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "forward", "gradient", "autograd", "batch", "fused"])
    if kind == "batch":
        return _case("batch", "neck", TF32X3, 0, 0, 32, rng.randint(2, 12), rng.randint(12, 30), graph=rng.random() < 0.5)
    if kind == "fused":
        # parts of 14 to 16 points per axis
        parts = rng.randint(3, 16)
        own = [rng.choice([14, 15, 16, 16]) for _ in range(2)]
        nx, ny, M = parts * own[0], parts * own[1], rng.choice([16, 32])
        c = _case("forward", "custom", FP32, nx, ny, M, rng.randint(1, 16), rng.randint(20, 60), parts=parts)
    elif kind == "forward":
        precision = rng.choice([FP32, TF32X3, TF32X3, BF16X3])
        M = rng.choice([8, 16, 24, 32, 64]) if precision == FP32 else rng.choice([16, 32, 32, 64])
        c = _case("forward", "custom", precision, _log_int(rng, 24, 512), _log_int(rng, 24, 512), M,
                  _log_int(rng, 1, 16), _log_int(rng, 30, 200), graph=rng.random() < 0.2)
    else:
        precision = rng.choice([FP32, TF32X3, TF32X3])
        steps = rng.randint(24, 60)
        c = _case(kind, "custom", precision, _log_int(rng, 32, 256), _log_int(rng, 32, 256), rng.choice([16, 32]),
                  _log_int(rng, 1, 8), steps, ckpt=rng.randint(7, steps))
    cost = 4 if c["kind"] != "forward" else 1
    if c["precision"] == FP32 and c["parts"] == 1:
        cost *= 4
    while c["nx"] * c["ny"] * c["M"] * c["groups"] * c["steps"] * cost > MAX_UPDATES:
        if c["groups"] > 1:
            c["groups"] = max(1, c["groups"] // 2)
        else:
            c["steps"] = max(12, c["steps"] // 2)
            c["ckpt"] = min(c["ckpt"], c["steps"])
            if c["steps"] == 12:
                break
    return c


# ------------------------------------------------------------------ inputs
def _workloads(case, seed):
    """The workloads of the case (one per medium), with pulses inside the simulated time."""
    kind, G, steps = case["medium"], case["groups"], case["steps"]
    rng = np.random.default_rng(seed)
    if kind == "small":
        wl = workload_small(n_steps=steps, dt=0.05)
        wl.groups = [[dataclasses.replace(wl.groups[0][0], x=float(rng.uniform(0.5, 1.5)))]]
        wls = [wl]
    elif kind == "tomo":
        wls = [workload_tomo256(n_steps=steps, n_sources=G, seed=seed)]
    elif kind == "precision":
        wls = [workload_precision512(n_steps=steps, seed=seed)]
    elif kind == "mss":
        wls = [workload_mss256(n_steps=steps, target=True, seed=seed)]
    elif kind == "inverse":
        wls = [workload_inverse("ts", n=case["nx"], n_steps=steps, target=True, seed=seed)]
    elif kind == "neck":
        # the sizes of the 48-media workload in turn; the seed draws the media and the beams
        wls = []
        for k in range(G):
            n = (128, 192, 256, 384)[k % 4]
            L = 4.0 / 255 * (n - 1)
            grid = Grid(n, n, 0.0, L, 0.0, L, case["M"])
            x, y, th = face_point(("bottom", "right", "top", "left")[k % 4], float(rng.uniform(0.3, 0.7)), L)
            a, b = neck_medium(grid, rng)
            wls.append(Workload("neck", grid, Optics(g=0.9), a, b, C0_CM_PER_PS / 1.4, 0.04, steps, [[Beam(x, y, th)]],
                                perimeter_detectors(L, 8)))
    else:
        # equal spacing 1/66 cm whatever the size: dt = 0.04 ps is stable
        wls = [workload_custom(case["nx"], case["ny"], case["M"], steps, 0.04, L=(case["nx"] - 1) / 66.0, mus=80.0,
                               n_groups=G, seed=seed, n_det_per_face=4)]
    for wl in wls:
        T = wl.n_steps * wl.dt
        wl.groups = [[dataclasses.replace(b, t_s=0.3 * T, sigma_t=0.12 * T, tau=min(b.tau, 0.4 * T),
                                          amplitude=float(rng.uniform(0.5, 1.5))) for b in grp] for grp in wl.groups]
    return wls


def _f32(a):
    return torch.tensor(np.asarray(a), dtype=torch.float32)


def _measured(wl, seed):
    """Detector data [group][det][step]: smooth positive pulses with 10 % noise, as a fit would be given."""
    g = torch.Generator().manual_seed(seed + 1)
    t = torch.linspace(0, 1, wl.n_steps)
    shape = (len(wl.groups), len(wl.detectors))
    centre, height = 0.4 + 0.3 * torch.rand(shape, generator=g), 1e-3 * torch.rand(shape, generator=g)
    pulse = height[..., None] * torch.exp(-((t - centre[..., None]) / 0.15) ** 2)
    return (pulse * (1 + 0.1 * torch.randn(pulse.shape, generator=g))).contiguous()


def prepare(case, seed):
    dev = torch.device("cuda")
    wls = _workloads(case, seed)
    flags = B.RTE_FLAG_CUDA_GRAPH if case["graph"] else 0
    parts = (case["parts"], case["parts"])
    state = {"case": case, "wls": wls, "solvers": [], "measured": None}
    for wl in wls:
        mua, mus = _f32(wl.mua).to(dev), _f32(wl.mus).to(dev)
        s = FCDOMSolver(wl.grid, wl.optics, mua, mus, wl.c, wl.dt, ckpt_interval=case["ckpt"],
                        precision=case["precision"], flags=flags, fc_parts=parts)
        if case["parts"] > 1:
            B.rte_set_pass_variant(s.ctx, 3)
        elif case["autotune"]:
            s.autotune(wl.groups, 20)
        state["solvers"].append(s)
        state["mua"], state["mus"] = mua, mus
    if case["kind"] in ("gradient", "autograd"):
        state["measured"] = _measured(wls[0], seed).to(dev)
    return state


def run(state):
    case, wls, solvers = state["case"], state["wls"], state["solvers"]
    wl, s = wls[0], solvers[0]
    if case["kind"] == "batch":
        forward_batch(solvers, [w.groups for w in wls], case["steps"])
        return {"curves": [v.readout(w.detectors) for v, w in zip(solvers, wls)],
                "u": [v.state(0) for v in solvers]}
    if case["kind"] == "gradient":
        s.forward(wl.groups, case["steps"])
        J, ga, gb = s.adjoint_gradient(wl.detectors, state["measured"])
        return {"J": J, "dmua": ga, "dmus": gb}
    if case["kind"] == "autograd":
        mua, mus = state["mua"].clone().requires_grad_(), state["mus"].clone().requires_grad_()
        J = RTEObjective.apply(mua, mus, state["measured"], s, wl.groups, case["steps"], wl.detectors, True)
        J.backward()
        return {"J": J.detach().float(), "dmua": mua.grad, "dmus": mus.grad}
    if case["graph"]:
        # no snapshots: the replayed graph is tied to the buffers it was captured with
        s.forward(wl.groups, case["steps"])
        return {"curves": s.readout(wl.detectors), "u": [s.state(g) for g in range(len(wl.groups))]}
    fluence = s.forward(wl.groups, case["steps"], [case["steps"] // 2, case["steps"] - 1])
    return {"fluence": fluence, "curves": s.readout(wl.detectors), "u": [s.state(g) for g in range(len(wl.groups))]}


def work(case):
    """One AB4 step moves 24 bytes per value of the intensity at least (read u and the three stored right-hand sides,
    write u and the new one) and does the two FC derivatives (2 n each), the scattering sum (2 M) and the update.  A
    gradient is three marches (forward, recompute, adjoint) and one read of both fields."""
    if case["kind"] == "batch":
        shapes = [(w.grid.nx, w.grid.ny, w.grid.M, 1) for w in _workloads(case, 1)]
    else:
        shapes = [(case["nx"], case["ny"], case["M"], case["groups"])]
    n_bytes = flops = 0.0
    for nx, ny, M, G in shapes:
        updates = float(nx) * ny * M * G * case["steps"]
        lines = 2 * (nx + ny) if case["parts"] == 1 else 80
        step_b, step_f = 24.0 * updates, updates * (lines + 2 * M + 12)
        marches = 3 if case["kind"] in ("gradient", "autograd") else 1
        n_bytes += marches * step_b + (8.0 * updates if marches == 3 else 0.0)
        flops += marches * step_f + (2.0 * (M + 2) * updates if marches == 3 else 0.0)
    return {"bytes": n_bytes, "flops": flops}


# ------------------------------------------------------------------ FP64 restatement
# FC-Gram data for 5 matching points and 25 continuation points: Gram polynomials on the matching points, and their
# continuations to zero (rows: distance 1..25 past the end of the line).
_GRAM = [[0.4472135954999579, -0.6324555320336759, 0.5345224838248488, -0.31622776601683794, 0.11952286093343936],
         [0.4472135954999579, -0.31622776601683794, -0.2672612419124244, 0.6324555320336759, -0.47809144373375745],
         [0.4472135954999579, 0.0, -0.5345224838248488, 0.0, 0.7171371656006362],
         [0.4472135954999579, 0.31622776601683794, -0.2672612419124244, -0.6324555320336759, -0.47809144373375745],
         [0.4472135954999579, 0.6324555320336759, 0.5345224838248488, 0.31622776601683794, 0.11952286093343936]]
_CONT = [
    [0.44721359549700146, 0.9486832980418872, 1.8708286929997828, 4.427188722633765, 15.059880377297775],
    [0.4472135941112565, 1.2649110583714287, 3.741657203960408, 13.281565112104625, 65.25943439425541],
    [0.4472135000401771, 1.581138335305175, 6.1469959125477605, 28.460406478507604, 179.9981012884362],
    [0.44721123363482274, 1.8973519805103611, 9.086566575028936, 51.54238164761199, 396.8515341811631],
    [0.44718354632289165, 2.213380415711073, 12.557221559041894, 84.07617208660285, 760.9859243984441],
    [0.44697725544547345, 2.527937032378835, 16.537901252911382, 127.39718481384972, 1320.9877052253105],
    [0.44593195599629704, 2.834830179285124, 20.935971772462995, 181.8879328023658, 2113.4736738766783],
    [0.4420709184474723, 3.113670112052883, 25.466483324467802, 245.10346528092322, 3126.461441262817],
    [0.43118162059961596, 3.317079173837191, 29.497433152732004, 308.9746360195997, 4246.142823249775],
    [0.4069761282808865, 3.367856850379299, 32.01990515890013, 358.46902516936024, 5227.3690857412275],
    [0.3636330007653888, 3.184980313269154, 31.946121798203034, 375.4436601252522, 5749.362257148216],
    [0.30019306130034995, 2.7376292601601575, 28.71932639713539, 348.2982881458781, 5570.6856851484345],
    [0.22360679774997896, 2.0895645125232, 22.838228278648444, 281.2789293220838, 4693.288442572432],
    [0.14702053419960798, 1.3865230120973009, 15.792504396342498, 194.59626939104615, 3394.849800856164],
    [0.08358059473456915, 0.7839477010537111, 9.338341831040843, 113.50222002102316, 2080.2837401143906],
    [0.04023746721907148, 0.3700240035221314, 4.6382494978080135, 54.844339624702435, 1063.3287867614797],
    [0.016031974900342003, 0.1424705584788014, 1.8951626488063722, 21.498199749791567, 444.77245798513246],
    [0.005142677052485623, 0.043500039497337675, 0.6205790314406459, 6.655389960949903, 148.49147453409944],
    [0.0012816395036608814, 0.010149994931723597, 0.15731683119383275, 1.5697754756056725, 38.25519456886343],
    [0.00023634005448450404, 0.0017198875976318314, 0.0294243251525772, 0.26826064362755214, 7.252466859692846],
    [3.0049177066299665e-05, 0.00019650272970298338, 0.0037855784725752957, 0.03085551562282558, 0.9436480045225863],
    [2.361865135203807e-06, 1.3494485903290914e-05, 0.00030047203186116256, 0.0021301556633287044, 0.07560397667767091],
    [9.545978080184925e-08, 4.586978205140662e-07, 1.2241696969336232e-05, 7.270643156051929e-05, 0.0031038666127178676],
    [1.3887014175158539e-09, 5.2971455652284715e-09, 1.7922544665435412e-07, 8.422982443084186e-07, 4.5720284642184114e-05],
    [2.9565025747437146e-12, 8.041429084218171e-12, 3.8343771142267104e-10, 1.2817157956554484e-09, 9.827316255303149e-08]
]
_AB4 = (55.0 / 24.0, -59.0 / 24.0, 37.0 / 24.0, -9.0 / 24.0)


def _window(v):
    v = np.abs(np.asarray(v, dtype=np.float64))
    out = np.where(v == 0, 1.0, 0.0)
    inner = (v > 0) & (v < 1)
    out[inner] = np.exp(2.0 * np.exp(-1.0 / v[inner]) / (v[inner] - 1.0))
    return out


def _derivative(n, h):
    """The dense FC derivative of a line of n points at spacing h."""
    Q, A = np.array(_GRAM), np.array(_CONT)
    C = A.shape[0]
    Np = n + C
    while True:
        r = Np
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if r == 1:
            break
        Np += 1
    E = np.eye(n)
    right, left = E[:, n - 5:] @ Q @ A.T, E[:, :5][:, ::-1] @ Q @ A.T
    pad = np.zeros((n, Np - n - C))
    ext = np.concatenate([E, np.concatenate([right, pad], 1) + np.concatenate([pad, left[:, ::-1]], 1)], 1)
    k = np.fft.fftfreq(Np, d=1.0 / Np)
    mult = 2j * np.pi * k / (Np * h) * np.exp(-2.0 * np.abs(2.0 * k / Np) ** 110.0)
    if Np % 2 == 0:
        mult[Np // 2] = 0.0
    return np.fft.ifft(np.fft.fft(ext, axis=1) * mult, axis=1).real[:, :n].T


def _derivative_parts(n, h, parts):
    if parts <= 1:
        return _derivative(n, h)
    D = np.zeros((n, n))
    for k in range(parts):
        lo, hi = k * n // parts, (k + 1) * n // parts
        a, b = (lo - 2 if k else lo), (hi + 2 if k < parts - 1 else hi)
        D[lo:hi, a:b] = _derivative(b - a, h)[lo - a:hi - a]
    return D


class _Exact:
    def __init__(self, wl, parts, dev):
        g, o = wl.grid, wl.optics
        self.wl, self.dev, self.M, self.G = wl, dev, g.M, len(wl.groups)
        t = lambda v: torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)  # noqa: E731
        M = g.M
        theta = 2 * np.pi * np.arange(M) / M
        xi, eta = np.cos(theta), np.sin(theta)
        self.w = 2 * np.pi / M
        p = (1 - o.g ** 2) / (1 + o.g ** 2 - 2 * o.g * np.cos(theta[:, None] - theta[None])) ** o.hg_exponent
        self.P = t(p / p.sum(1, keepdims=True))
        self.Dx, self.Dy = t(_derivative_parts(g.nx, g.dx, parts)), t(_derivative_parts(g.ny, g.dy, parts))
        self.xi, self.eta = t(xi), t(eta)
        self.a, self.b = _f32(wl.mua).double().to(dev), _f32(wl.mus).double().to(dev)
        self.cdt = wl.c * wl.dt
        # boundary: governing face, reflected ordinate and Fresnel coefficient of every incoming (node, ordinate)
        cosf = np.array([-xi, xi, -eta, eta])
        refl = np.array([(M // 2 - np.arange(M)) % M] * 2 + [(-np.arange(M)) % M] * 2)
        ci = np.abs(cosf)
        st = o.n_in / o.n_out * np.sqrt(np.maximum(0.0, 1 - ci ** 2))
        ct = np.sqrt(np.maximum(0.0, 1 - st ** 2))
        with np.errstate(invalid="ignore", divide="ignore"):
            rs = (o.n_in * ci - o.n_out * ct) / (o.n_in * ci + o.n_out * ct)
            rp = (o.n_out * ci - o.n_in * ct) / (o.n_out * ci + o.n_in * ct)
        fres = np.where(st < 1.0, 0.5 * (rs ** 2 + rp ** 2), 1.0)
        jj, ii = np.meshgrid(np.arange(g.ny), np.arange(g.nx), indexing="ij")
        on = np.stack([ii == 0, ii == g.nx - 1, jj == 0, jj == g.ny - 1], -1).reshape(-1, 4)
        self.nodes = np.flatnonzero(on.any(1))
        inc = on[self.nodes][:, :, None] & (cosf < -1e-12)[None]                 # [node, face, m]
        x_face = np.where(inc[:, 0] | inc[:, 1], np.where(inc[:, 0], 0, 1), -1)
        y_face = np.where(inc[:, 2] | inc[:, 3], np.where(inc[:, 2], 2, 3), -1)
        m = np.arange(M)[None]
        x_wins = (x_face >= 0) & ((y_face < 0) | (ci[x_face, m] > ci[y_face, m] + 1e-12))
        face = np.where(x_wins, x_face, y_face)
        self.act = torch.tensor(face >= 0, device=dev)
        self.refl = torch.tensor(np.where(face >= 0, refl[face, m], 0), device=dev)
        self.f = t(np.where(face >= 0, fres[face, m], 0.0))
        self.idx = torch.tensor(self.nodes, device=dev)
        self.x = g.xmin + g.dx * (self.nodes % g.nx)
        self.y = g.ymin + g.dy * (self.nodes // g.nx)
        # detectors: readout[det, node, m] = sum over the node's faces of trapezoid x window x exitance weight
        wex = np.where(cosf > 1e-12, self.w * (1 - fres) * cosf, 0.0)
        dist = np.stack([np.hypot(self.x - d.x, self.y - d.y) / d.sigma_d for d in wl.detectors])
        self.Wn = t(_window(dist))                                               # [det, node]
        R = np.zeros((len(self.nodes), M))
        jn, i_n = self.nodes // g.nx, self.nodes % g.nx
        for F in range(4):
            h, ends = (g.dy, (jn == 0) | (jn == g.ny - 1)) if F < 2 else (g.dx, (i_n == 0) | (i_n == g.nx - 1))
            R += (on[self.nodes, F] * np.where(ends, 0.5 * h, h))[:, None] * wex[F][None]
        self.R = t(R)
        self.beams = []
        kmax = max([len(b) for b in wl.groups] + [1])
        S, A = np.zeros((self.G, kmax, len(self.nodes))), np.zeros((self.G, kmax, M))
        T = np.zeros((wl.n_steps, self.G, kmax))
        for gi, grp in enumerate(wl.groups):
            for k, b in enumerate(grp):
                S[gi, k] = np.exp(-((self.x - b.x) ** 2 + (self.y - b.y) ** 2) / (2 * b.sigma_x ** 2))
                d = np.mod(np.abs(theta - b.theta), 2 * np.pi)
                A[gi, k] = b.amplitude * _window(np.minimum(d, 2 * np.pi - d) / b.sigma_theta)
                tt = (np.arange(wl.n_steps) + 4) * wl.dt - b.tau - b.t_s
                T[:, gi, k] = np.exp(-tt ** 2 / (2 * b.sigma_t ** 2)) if b.profile == 0 else _window(tt / b.sigma_t)
        self.S, self.A, self.T = t(S), t(A), t(T)
        wx, wy = np.full(g.nx, g.dx), np.full(g.ny, g.dy)
        wx[[0, -1]] *= 0.5
        wy[[0, -1]] *= 0.5
        self.area = t(wy[:, None] * wx[None])

    def zeros(self):
        g = self.wl.grid
        return torch.zeros((self.G, g.ny, g.nx, self.M), dtype=torch.float64, device=self.dev)

    def L(self, u, a, b):
        dy = (self.Dy @ u.reshape(self.G, u.shape[1], -1)).reshape(u.shape)
        return b[..., None] * (u @ self.P) - (a + b)[..., None] * u - self.xi * (self.Dx @ u) - self.eta * dy

    def step(self, u, hist, q, a, b):
        """u^{k+1} with the boundary inflow q [group, node, m], and the new history."""
        Lk = self.L(u, a, b)
        un = u + self.cdt * (_AB4[0] * Lk + _AB4[1] * hist[0] + _AB4[2] * hist[1] + _AB4[3] * hist[2])
        flat = un.reshape(self.G, -1, self.M)
        pre = flat[:, self.idx]
        val = torch.where(self.act, self.f * pre.gather(2, self.refl.expand(self.G, -1, -1)) + q, pre)
        return flat.index_copy(1, self.idx, val).reshape(un.shape), [Lk, hist[0], hist[1]]

    def inflow(self, s):
        return torch.einsum("gkn,gkm,gk->gnm", self.S, self.A, self.T[s])

    def read(self, u):
        return (u.reshape(self.G, -1, self.M)[:, self.idx] * self.R).sum(2) @ self.Wn.T

    def march(self, steps, a, b, snaps=(), keep=False):
        u, hist = self.zeros(), [self.zeros() for _ in range(3)]
        curves, fluence, states = [], [], []
        for s in range(steps):
            u, hist = self.step(u, hist, self.inflow(s), a, b)
            curves.append(self.read(u))
            if s in snaps:
                fluence.append(self.w * u.sum(3))
            if keep:
                states.append(u)
        return u, torch.stack(curves, 2), fluence, states

    def gradient(self, steps, measured):
        """The continuous adjoint: the flipped field marches forward in reversed time, driven by the residual."""
        dt = self.wl.dt
        _, curves, _, states = self.march(steps, self.a, self.b, keep=True)
        r = curves - measured
        mu, hist, ga, gb = self.zeros(), [self.zeros() for _ in range(3)], 0.0, 0.0
        for lvl in range(steps - 2, -1, -1):
            q = (1 - self.f) * (r[:, :, lvl] @ self.Wn)[..., None]
            mu, hist = self.step(mu, hist, q, self.a, self.b)
            lam, u = torch.roll(mu, self.M // 2, 3), states[lvl]
            ga = ga - (lam * u).sum((0, 3))
            gb = gb - (lam * (u - u @ self.P)).sum((0, 3))
        scale = self.area * self.w * dt
        return 0.5 * (r * r).sum() * dt, scale * ga, scale * gb

    def autograd(self, steps, measured):
        """The derivative of the discrete objective itself."""
        a, b = self.a.clone().requires_grad_(), self.b.clone().requires_grad_()
        r = self.march(steps, a, b)[1] - measured
        J = 0.5 * (r * r).sum() * self.wl.dt
        J.backward()
        return J.detach(), a.grad, b.grad


def exact(case, seed):
    dev = torch.device("cuda")
    wls, steps = _workloads(case, seed), case["steps"]
    if case["kind"] == "batch":
        out = {"curves": [], "u": []}
        for wl in wls:
            e = _Exact(wl, 1, dev)
            u, curves, _, _ = e.march(steps, e.a, e.b)
            out["curves"].append(curves)
            out["u"].append(u[0])
        return out
    e = _Exact(wls[0], case["parts"], dev)
    if case["kind"] in ("gradient", "autograd"):
        fn = e.gradient if case["kind"] == "gradient" else e.autograd
        J, ga, gb = fn(steps, _measured(wls[0], seed).double().to(dev))
        return {"J": J, "dmua": ga, "dmus": gb}
    u, curves, fluence, _ = e.march(steps, e.a, e.b, snaps=(steps // 2, steps - 1))
    out = {} if case["graph"] else {"fluence": torch.stack(fluence, 1)}
    return {**out, "curves": curves, "u": list(u)}
