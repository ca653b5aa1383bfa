"""The workloads that a user of this framework runs, as measured cases.

Each case is one call (or one loop body) of a seismic-inversion program through
the package's public entry points: modelling a survey, evaluating a misfit and
its gradient (directly, through autograd, or as a recorded graph), and the
start-model network's training gradient and prediction. Sizes are those of the
repository's own workloads (synth.py, learned.py, the benchmark), with fewer
time steps where more would only repeat the same work.
"""

import math

import numpy as np
import torch

from paper_2003_06027_gb300 import autograd, fwi, learned, synth


def listed():
    return [
        # one shot on the 100 x 100 two-layer grid: the smallest modelling call, bound by latency
        dict(name="small_forward", kind="forward", nz=100, nx=100, shots=1, nt=500, order=4, npml=20, dt=1e-3, op=0, ckpt=0),
        # earthquake location: one Gaussian source, gradient in its position and time function and in the model
        dict(name="small_location", kind="misfit", nz=121, nx=173, shots=1, nt=600, order=4, npml=20, dt=1e-3, op=0, ckpt=100),
        # a training survey of the start-model network: 16 shots on 128 x 256
        dict(name="survey_forward", kind="forward", nz=128, nx=256, shots=16, nt=1000, order=8, npml=32, dt=1e-3, op=0, ckpt=0),
        # one evaluation of that survey's inversion loop (recorded graph, replayed for every model)
        dict(name="survey_gradient", kind="graph", nz=128, nx=256, shots=16, nt=1000, order=8, npml=32, dt=1e-3, op=0, ckpt=100),
        # the FWI benchmark problem (201 x 601, 16 shots), one evaluation of its loop
        dict(name="fwi_gradient", kind="graph", nz=201, nx=601, shots=16, nt=1000, order=8, npml=32, dt=0.8e-3, op=0, ckpt=100),
        # the c^2 Laplacian operator on a grid of odd sizes, any torch loss of the seismograms
        dict(name="laplacian_odd", kind="seismograms", nz=187, nx=333, shots=6, nt=500, order=8, npml=32, dt=0.8e-3, op=1, ckpt=100),
        # many shots: one step's fields are far larger than the L2 cache
        dict(name="xl_gradient", kind="direct", nz=201, nx=601, shots=128, nt=100, order=8, npml=32, dt=0.8e-3, op=0, ckpt=50),
        # elastic modelling of 32 moment-tensor sources on 300 x 800
        dict(name="elastic_forward", kind="e_forward", nz=300, nx=800, shots=32, nt=250, order=4, npml=32, dt=0.5e-3, ckpt=0),
        # elastic inversion: misfit and its gradient in vp, vs, rho and the sources
        dict(name="elastic_gradient", kind="e_misfit", nz=300, nx=800, shots=8, nt=250, order=4, npml=32, dt=0.5e-3, ckpt=100),
        # a small elastic problem of odd sizes at 8th order, any torch loss of the seismograms
        dict(name="elastic_small", kind="e_seismograms", nz=97, nx=131, shots=2, nt=300, order=8, npml=20, dt=0.5e-3, ckpt=100),
        # the start-model network: parameter gradients of one training batch
        dict(name="network_gradient", kind="net_gradient", batch=32),
        # the start-model network applied to one survey
        dict(name="network_predict", kind="net_predict", batch=1),
    ]


# Grid points x shots x steps that a drawn case of each kind may have: no more than the largest listed one.
_MOST = {"forward": 2.4e9, "misfit": 1.2e9, "seismograms": 1.2e9, "graph": 2.4e9, "direct": 2.0e9, "e_forward": 1.2e9,
         "e_misfit": 5.0e8, "e_seismograms": 4.0e8}


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("forward", "forward", "misfit", "seismograms", "graph", "graph", "direct", "e_forward", "e_misfit",
                       "e_seismograms", "net_gradient", "net_predict"))
    if kind == "net_gradient":
        return dict(kind=kind, batch=log(1, 32))
    if kind == "net_predict":
        return dict(kind=kind, batch=log(1, 32))
    elastic = kind.startswith("e_")
    c = dict(kind=kind, nz=log(48, 512), nx=log(48, 1024), shots=log(1, 32 if elastic else 128), nt=log(200, 1000),
             order=rng.choice((4, 8)), npml=rng.choice((16, 20, 32)), dt=0.5e-3 if elastic else 0.8e-3)
    if not elastic:
        c["op"] = rng.choice((0, 0, 0, 1))
    while _points(c) * c["shots"] * c["nt"] > _MOST[kind]:
        k = rng.choice(("shots", "nt"))
        c[k] = max(1 if k == "shots" else 200, int(c[k] * 0.7))
    c["ckpt"] = 0 if kind.endswith("forward") else min(c["nt"], rng.choice((20, 50, 100)))
    return c


def _points(case):
    return (case["nz"] + 2 * case["npml"]) * (case["nx"] + 2 * case["npml"])


# ---------------------------------------------------------------- inputs
def _survey(case, seed):
    """The arrays of a case (numpy, FP32): models, sources, receivers, recorded data."""
    rng = np.random.default_rng([seed, 17])
    nz, nx, S, nt, dt = case["nz"], case["nx"], case["shots"], case["nt"], case["dt"]
    elastic = case["kind"].startswith("e_")
    dx = 5.0 if elastic else 10.0
    f0 = 10.0 if elastic else 8.0
    true = synth.layered_model(int(rng.integers(1 << 30)), nz, nx, dx, vmin=1800.0 if elastic else 1500.0, n_faults=1)
    vp = true if case["kind"].endswith("forward") else synth.smooth(true, 8.0)
    # wavelets that end within a third of the record, and (below) sources whose waves reach the receivers in the next
    freq = max(f0, 3.0 / (nt * dt)) * rng.uniform(0.9, 1.3, S)
    stf = np.stack([synth.ricker(float(f), dt, nt, t0=1.0 / float(f)) for f in freq]).astype(np.float32)
    gauss = elastic or case["kind"] == "misfit"
    if gauss:
        # off-grid positions, at least 5 cells inside the physical grid
        deepest = min(nz - 6.0, max(6.0, 0.33 * nt * dt * 2000.0 / dx))
        x0 = np.stack([rng.uniform(5, nx - 6, S) * dx, rng.uniform(5, deepest, S) * dx], 1)
    else:
        x0 = np.stack([np.linspace(0, nx - 1, S) * dx if S > 1 else np.array([0.5 * (nx - 1) * dx]), np.full(S, 2 * dx)], 1)
    d = dict(dx=dx, dz=dx, dt=dt, order=case["order"], npml=case["npml"], pml_R=1e-5 if case["npml"] >= 32 else 1e-3,
             pml_vmax=4500.0, pml_f0=f0, src_kind=1 if gauss else 0, stf=stf, x0=x0.astype(np.float32))
    step = 4 if elastic else 2
    d["rec_ix"] = np.arange(0, nx, step, dtype=np.int32)
    d["rec_iz"] = np.full(d["rec_ix"].shape, 2, np.int32)
    nrec = d["rec_ix"].size
    if elastic:
        d["vp"], d["vs"], d["rho"] = vp, (vp / 1.73).astype(np.float32), synth.gardner_density(vp)
        d["mt"] = (synth.double_couple(rng.uniform(0, np.pi, S)) * synth.MOMENT_SCALE).astype(np.float32)
    else:
        d["c"] = vp
        d["op"] = case["op"]
    if not case["kind"].endswith("forward"):
        # recorded data (or, for a loss of the seismograms, its weights): three arrivals with hyperbolic moveout and
        # noise, at the amplitude of the modelled data
        t = torch.arange(nt, dtype=torch.float32) * dt
        off = torch.as_tensor(d["rec_ix"] * dx - d["x0"][:, :1], dtype=torch.float32)
        g = torch.Generator().manual_seed(seed)
        comp = 2 if elastic else 1
        obs = 0.02 * torch.randn((S, comp, nrec, nt), generator=g)
        for k in range(3):
            t0, v, amp = rng.uniform(0.1, 0.7) * nt * dt, rng.uniform(1600, 4000), rng.uniform(0.3, 1.0, comp)
            arr = (torch.sqrt(t0**2 + (off / v) ** 2)[:, :, None] - t) * (math.pi * float(freq.mean()))
            w = (1 - 2 * arr**2) * torch.exp(-(arr**2))
            obs += w[:, None] * torch.as_tensor(amp, dtype=torch.float32)[None, :, None, None]
        d["obs"] = (obs * (0.05 if elastic else 1e-7)).reshape((S, 2, nrec, nt) if elastic else (S, nrec, nt)).numpy()
    return d


def _net_inputs(case, seed):
    """Gathers of random events, peak-normalised as gathers_to_input does, and normalised target models."""
    B = case["batch"]
    g = torch.Generator().manual_seed(seed)
    t = torch.arange(learned.NT, dtype=torch.float32)[None, None, :, None] / learned.NT
    x = torch.zeros((learned.NSHOT, B, learned.NT, learned.NREC))
    src = torch.linspace(0, 1, learned.NSHOT)[:, None, None, None]
    rec = torch.linspace(0, 1, learned.NREC)
    for _ in range(4):
        t0, p = 0.7 * torch.rand((1, B, 1, 1), generator=g), 0.2 + 0.6 * torch.rand((1, B, 1, 1), generator=g)
        a = torch.randn((1, B, 1, 1), generator=g)
        arr = (torch.sqrt(t0**2 + (p * (rec - src)) ** 2) - t) * 25.0
        x += a * (1 - 2 * arr**2) * torch.exp(-(arr**2))
    x = x * t
    x = (x / x.abs().amax(dim=(0, 2, 3), keepdim=True)).contiguous()
    z = torch.linspace(-1, 1, learned.NZ)[:, None]
    y = (z + 0.2 * torch.randn((B, 1, learned.NX), generator=g)).clamp(-1, 1)[None].contiguous()
    return x, y


def _net_weights(net, seed):
    """Weights of the seed in a network handle: He-scaled weights and small biases."""
    g = torch.Generator().manual_seed(seed + 1)
    theta = torch.empty(net.nparams)
    for L in net.layers:
        nw = L["O"] * L["C"] * 9
        theta[L["off"]:L["off"] + nw] = torch.randn(nw, generator=g) * math.sqrt(2.0 / (9 * L["C"]))
        theta[L["off"] + nw:L["off"] + nw + L["O"]] = 0.05 * torch.randn(L["O"], generator=g)
    return theta


def prepare(case, seed):
    kind = case["kind"]
    if kind.startswith("net_"):
        net = learned.Net(0, seed=0)
        net.theta.copy_(_net_weights(net, seed))
        net.theta_bf16 = learned.to_bf16(net.theta)
        x, y = _net_inputs(case, seed)
        return dict(kind=kind, net=net, x=x.cuda(), y=y.cuda())
    d = _survey(case, seed)
    cu = {k: torch.as_tensor(np.ascontiguousarray(v)).cuda() for k, v in d.items() if isinstance(v, np.ndarray)}
    kw = {k: v for k, v in d.items() if not isinstance(v, np.ndarray)}
    s = dict(kind=kind, kw=kw, **cu)
    if kind not in ("forward", "e_forward"):
        s["kw"] = kw = dict(kw, ckpt_every=case["ckpt"])
    if kind == "graph":
        s["graph"] = fwi.GradGraph(s["c"], s["stf"], s["x0"], s["rec_iz"], s["rec_ix"], s["obs"], **kw)
    if kind in ("misfit", "seismograms", "e_misfit", "e_seismograms"):
        names = ("vp", "vs", "rho", "stf", "x0") if kind.startswith("e_") else ("c", "stf", "x0")
        if kind == "seismograms":  # point sources: no position gradient is asked for
            names = ("c", "stf")
        s["params"] = [s[n].requires_grad_(True) for n in names]
    return s


def run(s):
    kind = s["kind"]
    if kind == "net_gradient":
        net = s["net"]
        out = net.forward(s["x"])
        _, dout = learned.mse(net.h, out, s["y"])
        net.backward(dout)
        return {"out": out, "grad": net.grad}
    if kind == "net_predict":
        return {"out": s["net"].forward(s["x"])}
    kw = s["kw"]
    rec = (s["rec_iz"], s["rec_ix"])
    if kind == "forward":
        return fwi.forward(s["c"], s["stf"], s["x0"], *rec, **kw)
    if kind == "graph":
        g = s["graph"]
        g.launch()
        return {"misfit": g.misfit, "grad": g.grad}
    if kind == "direct":
        J, grad, gstf, _, _ = fwi.misfit_grad(s["c"], s["stf"], s["x0"], *rec, s["obs"], **kw)
        return {"misfit": J, "grad": grad, "grad_stf": gstf}
    if kind == "e_forward":
        return fwi.forward_elastic(s["vp"], s["vs"], s["rho"], s["stf"], s["x0"], s["mt"], *rec, **kw)
    if kind == "misfit":
        J = autograd.acoustic_misfit(s["c"], s["stf"], s["x0"], s["obs"], *rec, **kw)
        return {"misfit": J.detach(), "grads": torch.autograd.grad(J, s["params"])}
    if kind == "e_misfit":
        J = autograd.elastic_misfit(s["vp"], s["vs"], s["rho"], s["stf"], s["x0"], s["mt"], s["obs"], *rec, **kw)
        return {"misfit": J.detach(), "grads": torch.autograd.grad(J, s["params"])}
    if kind == "seismograms":
        d = autograd.acoustic_seismograms(s["c"], s["stf"], s["x0"], *rec, **kw)
    else:
        d = autograd.elastic_seismograms(s["vp"], s["vs"], s["rho"], s["stf"], s["x0"], s["mt"], *rec, **kw)
    # the gradient of any loss of the seismograms: here its derivative with respect to them is given
    return {"seismograms": d.detach(), "grads": torch.autograd.grad(d, s["params"], s["obs"])}


def work(case):
    kind = case["kind"]
    if kind.startswith("net_"):
        B = case["batch"]
        n = learned.network_flops_per_sample() * B
        par = sum(o * c * 9 + o for c, o, *_ in list(learned.ENCODER) + list(learned.DECODER) + [(32, 1)])
        io = 4.0 * B * (learned.NSHOT * learned.NT * learned.NREC + learned.NZ * learned.NX)
        if kind == "net_predict":
            return {"bytes": io + 2.0 * par, "flops": n}
        return {"bytes": io + 10.0 * par, "flops": 3.0 * n}
    # per grid point and step (FP32): acoustic forward reads u^n, u^{n-1}, m and writes u^{n+1}; the reverse sweep
    # reads two adjoint fields, m and the stored fields and updates the gradient. Elastic likewise.
    p = _points(case) * case["shots"] * case["nt"]
    N = case["order"] // 2
    if kind == "forward":
        return {"bytes": 16.0 * p, "flops": (8 * N + 7) * p}
    if kind == "e_forward":
        return {"bytes": 60.0 * p, "flops": (16 * N + 22) * p}
    if kind.startswith("e_"):
        return {"bytes": 168.0 * p, "flops": 3 * (16 * N + 22) * p}
    return {"bytes": 48.0 * p, "flops": 3 * (8 * N + 7) * p}


# ---------------------------------------------------------------- the same in 64 bits
_FD = {4: (9 / 8, -1 / 24), 8: (1225 / 1024, -245 / 3072, 49 / 5120, -5 / 7168)}


def _cpml(n, npml, h, dt, R, vmax, f0, half):
    """CPML coefficients (a, b) at the grid points (or half points) of one padded axis."""
    N = n + 2 * npml
    x = np.arange(N - 1 if half else N) + (0.5 if half else 0.0)
    dist = np.maximum(np.maximum(npml - x, x - (npml + n - 1)), 0.0) * h
    L = npml * h
    damp = -3.0 * vmax * math.log(R) / (2.0 * L) * (dist / L) ** 2
    b = np.exp(-(damp + math.pi * f0 * (1 - dist / L)) * dt)
    a = np.where(dist > 0, damp * (b - 1) / np.maximum(damp + math.pi * f0 * (1 - dist / L), 1e-300), 0.0)
    return a, np.where(dist > 0, b, 1.0)


class _Scheme:
    """Staggered differences and CPML of a padded grid [shots][Nz][Nx], FP64."""

    def __init__(self, case, d, dev):
        nz, nx, np_ = case["nz"], case["nx"], case["npml"]
        self.a, self.N, self.np = _FD[case["order"]], case["order"] // 2, np_
        self.dx, self.dt = float(np.float32(d["dx"])), float(np.float32(d["dt"]))
        self.Nz, self.Nx, self.dev = nz + 2 * np_, nx + 2 * np_, dev
        f32 = lambda v: float(np.float32(v))  # noqa: E731
        self.tab = {}
        for axis, n in ((1, nz), (2, nx)):
            for half in (False, True):
                t = _cpml(n, np_, self.dx, self.dt, f32(d["pml_R"]), f32(d["pml_vmax"]), f32(d["pml_f0"]), half)
                shape = (1, -1, 1) if axis == 1 else (1, 1, -1)
                self.tab[axis, half] = [torch.as_tensor(v, dtype=torch.float64, device=dev).reshape(shape) for v in t]

    def plus(self, u, axis):
        """D+ at the half points between the points of `axis` (zero beyond the grid)."""
        n, N = u.shape[axis], self.N
        w = torch.nn.functional.pad(u, (N, N) if axis == 2 else (0, 0, N, N))
        return sum(c * (w.narrow(axis, k + N, n - 1) - w.narrow(axis, N - k + 1, n - 1)) for k, c in enumerate(self.a, 1)) / self.dx

    def minus(self, q, axis):
        """D- at the points from values at the half points between them."""
        n, N = q.shape[axis] + 1, self.N
        w = torch.nn.functional.pad(q, (N, N) if axis == 2 else (0, 0, N, N))
        return sum(c * (w.narrow(axis, k - 1 + N, n) - w.narrow(axis, N - k, n)) for k, c in enumerate(self.a, 1)) / self.dx

    def absorb(self, g, mem, axis, half):
        a, b = self.tab[axis, half]
        mem = b * mem + a * g
        return g + mem, mem

    def pad(self, model):
        return torch.nn.functional.pad(model[None, None], (self.np,) * 4, mode="replicate")[0]

    def source(self, x0, kind, off, n_z, n_x):
        """Weights [shots][n_z][n_x] of the sources on nodes offset by `off` cells."""
        S = x0.shape[0]
        w = []
        for s in range(S):
            jc = math.floor(float(x0[s, 0].detach()) / self.dx - off + 0.5) + self.np
            ic = math.floor(float(x0[s, 1].detach()) / self.dx - off + 0.5) + self.np
            f = torch.zeros((n_z, n_x), dtype=torch.float64, device=self.dev)
            if kind == 0:
                f[ic, jc] = 1.0 / self.dx**2
            else:
                k = torch.arange(-3, 4, dtype=torch.float64, device=self.dev)
                xi = (jc - self.np + off + k) * self.dx - x0[s, 0]
                zi = (ic - self.np + off + k) * self.dx - x0[s, 1]
                sg2 = (0.5 * self.dx) ** 2
                box = torch.exp(-(zi[:, None] ** 2 + xi[None] ** 2) / (2 * sg2)) / (2 * math.pi * sg2)
                f = torch.nn.functional.pad(box, (jc - 3, n_x - jc - 4, ic - 3, n_z - ic - 4))
            w.append(f)
        return torch.stack(w)


def _acoustic_step(sc, op, st, par, stf_n, iz, ix):
    u, up, px, pz, zx, zz = st
    m, mx, mz, w = par
    gx, px = sc.absorb(sc.plus(u, 2), px, 2, True)
    gz, pz = sc.absorb(sc.plus(u, 1), pz, 1, True)
    hx, zx = sc.absorb(sc.minus(gx if op else mx * gx, 2), zx, 2, False)
    hz, zz = sc.absorb(sc.minus(gz if op else mz * gz, 1), zz, 1, False)
    r = hx + hz
    un = 2 * u - up + sc.dt**2 * (m * r if op else r) + (sc.dt**2 * stf_n)[:, None, None] * w
    return (un, u, px, pz, zx, zz), un[:, iz, ix]


def _elastic_step(sc, st, par, stf_n, iz, ix):
    vx, vz, sxx, szz, sxz = st[:5]
    m = list(st[5:])
    bx, bz, lam, lp2m, mxz, sn, ss, mt = par
    dt = sc.dt
    d1, m[0] = sc.absorb(sc.plus(sxx, 2), m[0], 2, True)
    d2, m[1] = sc.absorb(sc.minus(sxz, 1), m[1], 1, False)
    d3, m[2] = sc.absorb(sc.minus(sxz, 2), m[2], 2, False)
    d4, m[3] = sc.absorb(sc.plus(szz, 1), m[3], 1, True)
    vx = vx + dt * bx * (d1 + d2)
    vz = vz + dt * bz * (d3 + d4)
    rec = torch.stack([vx[:, iz, ix], vz[:, iz, ix]], 1)
    ex, m[4] = sc.absorb(sc.minus(vx, 2), m[4], 2, False)
    ez, m[5] = sc.absorb(sc.minus(vz, 1), m[5], 1, False)
    d7, m[6] = sc.absorb(sc.plus(vx, 1), m[6], 1, True)
    d8, m[7] = sc.absorb(sc.plus(vz, 2), m[7], 2, True)
    amp = (dt * stf_n)[:, None, None]
    sxx = sxx + dt * (lp2m * ex + lam * ez) - amp * sn * mt[:, 0, None, None]
    szz = szz + dt * (lam * ex + lp2m * ez) - amp * sn * mt[:, 1, None, None]
    sxz = sxz + dt * mxz * (d7 + d8) - amp * ss * mt[:, 2, None, None]
    return (vx, vz, sxx, szz, sxz, *m), rec


def _model64(case, d, p, dev):
    """Seismograms in 64 bits, differentiable in the tensors of `p`."""
    from torch.utils.checkpoint import checkpoint

    sc = _Scheme(case, d, dev)
    S, nt, Nz, Nx = case["shots"], case["nt"], sc.Nz, sc.Nx
    iz = torch.as_tensor(d["rec_iz"], device=dev).long() + sc.np
    ix = torch.as_tensor(d["rec_ix"], device=dev).long() + sc.np
    zero = lambda a, b: torch.zeros((S, a, b), dtype=torch.float64, device=dev)  # noqa: E731
    if case["kind"].startswith("e_"):
        vp, vs, rho = (sc.pad(p[k]) for k in ("vp", "vs", "rho"))
        mu = rho * vs**2
        lam = rho * (vp**2 - 2 * vs**2)
        inv = 1 / mu
        mxz = 4 / (inv[:, :-1, :-1] + inv[:, :-1, 1:] + inv[:, 1:, :-1] + inv[:, 1:, 1:])
        mt = torch.as_tensor(d["mt"], dtype=torch.float64, device=dev)
        par = (2 / (rho[:, :, :-1] + rho[:, :, 1:]), 2 / (rho[:, :-1] + rho[:, 1:]), lam, lam + 2 * mu, mxz,
               sc.source(p["x0"], d["src_kind"], 0.0, Nz, Nx), sc.source(p["x0"], d["src_kind"], 0.5, Nz - 1, Nx - 1), mt)
        shapes = [(Nz, Nx - 1), (Nz - 1, Nx), (Nz, Nx), (Nz, Nx), (Nz - 1, Nx - 1), (Nz, Nx - 1), (Nz, Nx - 1), (Nz - 1, Nx),
                  (Nz - 1, Nx), (Nz, Nx), (Nz, Nx), (Nz - 1, Nx - 1), (Nz - 1, Nx - 1)]
        step = lambda st, par, g: _elastic_step(sc, st, par, g, iz, ix)  # noqa: E731
    else:
        m = sc.pad(p["c"]) ** 2
        par = (m, 0.5 * (m[:, :, :-1] + m[:, :, 1:]), 0.5 * (m[:, :-1] + m[:, 1:]), sc.source(p["x0"], d["src_kind"], 0.0, Nz, Nx))
        shapes = [(Nz, Nx), (Nz, Nx), (Nz, Nx - 1), (Nz - 1, Nx), (Nz, Nx), (Nz, Nx)]
        step = lambda st, par, g: _acoustic_step(sc, case["op"], st, par, g, iz, ix)  # noqa: E731
    npar = len(par)

    def segment(n0, n1, stf, *args):
        par, st, rec = args[:npar], args[npar:], []
        for n in range(n0, n1):
            st, r = step(st, par, stf[:, n])
            rec.append(r)
        return (*st, torch.stack(rec, -1))

    st, out = tuple(zero(*s) for s in shapes), []
    grad = torch.is_grad_enabled()
    seg = 10 if S * _points(case) > 5e6 else 25
    for n0 in range(0, nt, seg):
        args = (n0, min(nt, n0 + seg), p["stf"], *par, *st)
        *st, rec = checkpoint(segment, *args, use_reentrant=False) if grad else segment(*args)
        st = tuple(st)
        out.append(rec)
    return torch.cat(out, -1)


def _net64(case, seed, dev, grad):
    x, y = (t.to(dev, torch.float64) for t in _net_inputs(case, seed))
    specs = [(c, o, sh, sw, True, False) for c, o, sh, sw in learned.ENCODER]
    specs += [(c, o, 1, 1, True, True) for c, o in learned.DECODER] + [(learned.DECODER[-1][1], 1, 1, 1, False, False)]
    layers, off = [], 0
    for c, o, *_ in specs:
        layers.append(dict(C=c, O=o, off=off))
        off += o * c * 9 + o

    class Shape:
        nparams = off

    Shape.layers = layers
    theta = _net_weights(Shape, seed).to(dev, torch.float64).requires_grad_(grad)
    h = x.transpose(0, 1)
    for (c, o, sh, sw, relu, up), L in zip(specs, layers):
        nw = o * c * 9
        if up:
            h = torch.nn.functional.interpolate(h, scale_factor=2, mode="nearest")
        h = torch.nn.functional.conv2d(h, theta[L["off"]:L["off"] + nw].reshape(o, c, 3, 3),
                                       theta[L["off"] + nw:L["off"] + nw + o], (sh, sw), 1)
        h = torch.relu(h) if relu else h
    out = h.transpose(0, 1)
    if not grad:
        return {"out": out}
    loss = 0.5 * ((out - y) ** 2).mean()
    return {"out": out.detach(), "grad": torch.autograd.grad(loss, theta)[0]}


def exact(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if kind == "net_predict":
        with torch.no_grad():
            return _net64(case, seed, dev, False)
    if kind == "net_gradient":
        return _net64(case, seed, dev, True)
    d = _survey(case, seed)
    names = [n for n in ("c", "vp", "vs", "rho", "stf", "x0") if n in d]
    p = {n: torch.as_tensor(d[n], device=dev).double() for n in names}
    if kind in ("forward", "e_forward"):
        with torch.no_grad():
            return _model64(case, d, p, dev)
    for n in names:
        if n != "x0" or d["src_kind"] == 1:
            p[n].requires_grad_(True)
    with torch.enable_grad():
        s = _model64(case, d, p, dev)
        obs = torch.as_tensor(d["obs"], device=dev).double()
        want = [n for n in names if p[n].requires_grad]
        if kind in ("seismograms", "e_seismograms"):
            return {"seismograms": s.detach(), "grads": torch.autograd.grad(s, [p[n] for n in want], obs)}
        J = 0.5 * ((s - obs) ** 2).sum()
        g = dict(zip(want, torch.autograd.grad(J, [p[n] for n in want])))
    J = J.detach()
    if kind == "graph":
        return {"misfit": J.reshape(1), "grad": g["c"]}
    if kind == "direct":
        return {"misfit": J.reshape(1), "grad": g["c"], "grad_stf": g["stf"]}
    return {"misfit": J, "grads": tuple(g[n] for n in want)}
