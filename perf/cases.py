"""Timed cases of the solver's main paths, through its public entry points.

Every case is a workload that a user of the package runs: explicit 2-D
trajectories (Allen-Cahn, Cahn-Hilliard, coupled), batched ensembles, the
calibration gradient of a Cahn-Hilliard trajectory, implicit steps in 2-D and
3-D, the Eshelby solve, and the learned warm start (inference and a training
step).  `exact` evaluates the same quantities in FP64 with plain torch.
"""
import math
import random

import torch

import paper_2601_06079_gb300 as pf

GL = 0.5 - 0.5 / math.sqrt(3.0)  # weight of the far node at a Gauss point
GH = 1.0 - GL
F64 = torch.float64


def listed():
    return [
        # smallest: a 64 x 64 Allen-Cahn run (the package's smoke check and first configuration)
        dict(name="ac_64", kind="explicit", model="ac", ny=64, nx=64, hx=64 / 63, hy=64 / 63,
             dt=0.01, kappa=1.0, steps=200),
        # the headline mesh: spinodal decomposition, the benchmark's parameters
        dict(name="ch_2048", kind="explicit", model="ch", ny=2048, nx=2048, hx=1.0, hy=1.0,
             dt=1e-3, kappa=0.5, steps=1000),
        # a ragged mesh with unequal spacings, a step count that is no round number
        dict(name="ch_ragged", kind="explicit", model="ch", ny=515, nx=1031, hx=0.8, hy=1.25,
             dt=1e-3, kappa=0.7, steps=333),
        # coupled Allen-Cahn / Cahn-Hilliard precipitates at the headline size
        dict(name="coupled_2048", kind="coupled", ny=2048, nx=2048, hx=1.0, hy=1.0, steps=200),
        # parameter study: 256 uneven instances in the default mode, one persistent launch
        dict(name="ensemble_256", kind="ensemble", count=256, lo=128, hi=512, grid=128,
             mode="persistent", steps=200),
        # calibration: loss and gradients of a 2,000-step trajectory, a mobility per node
        dict(name="misfit_512", kind="misfit", ny=512, nx=512, steps=2000, ckpt=100),
        # small implicit run (100 x 100 domain, 64 x 64 mesh, 6 steps): host round trips count
        dict(name="implicit_ac_64", kind="implicit2d", model="ac", ny=64, nx=64, h=100 / 63,
             dt=0.5, kappa=1.0, steps=6),
        # implicit split Cahn-Hilliard at the headline size, 1,000 times the explicit time step
        dict(name="implicit_ch_2048", kind="implicit2d", model="ch", ny=2048, nx=2048, h=1.0,
             dt=1.0, kappa=0.5, steps=1),
        # grain growth, 8 order parameters: one implicit step
        dict(name="grains_128", kind="grains", n=128, nf=8, dt=0.5),
        # Eshelby inclusion: CG to the default tolerance
        dict(name="eshelby_129", kind="eshelby", n=129),
        # learned warm start: the guess for one step of the 128^3 run
        dict(name="predict_128", kind="predict", d=128, h=128, w=128, history=2),
        # learned warm start: one training step on four 64^3 crops
        dict(name="train_64", kind="train", d=64, h=64, w=64, batch=4, history=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["explicit", "explicit", "coupled", "ensemble", "misfit", "implicit2d",
                       "grains", "eshelby", "predict", "train"])
    if kind == "explicit":
        model = rng.choice(["ac", "ch"])
        ny, nx = _log_int(rng, 16, 2048), _log_int(rng, 16, 2048)
        square = rng.random() < 0.6
        hx = rng.uniform(0.8, 1.25)
        return dict(kind=kind, model=model, ny=ny, nx=nx, hx=hx,
                    hy=hx if square else rng.uniform(0.8, 1.25),
                    dt=0.01 if model == "ac" else 1e-3, kappa=rng.uniform(0.4, 1.0),
                    steps=_log_int(rng, 50, 1000))
    if kind == "coupled":
        return dict(kind=kind, ny=_log_int(rng, 33, 2048), nx=_log_int(rng, 33, 2048),
                    hx=rng.uniform(0.9, 1.2), hy=rng.uniform(0.9, 1.2), steps=_log_int(rng, 20, 200))
    if kind == "ensemble":
        return dict(kind=kind, count=_log_int(rng, 8, 256), lo=rng.randrange(4, 100),
                    hi=rng.randrange(120, 400), grid=rng.choice([1, 8, 32]),
                    mode=rng.choice(["per_step", "persistent"]), steps=_log_int(rng, 20, 200))
    if kind == "misfit":
        return dict(kind=kind, ny=_log_int(rng, 40, 512), nx=_log_int(rng, 40, 512),
                    steps=_log_int(rng, 100, 1000), ckpt=rng.choice([25, 50, 100]))
    if kind == "implicit2d":
        model = rng.choice(["ac", "ch"])
        return dict(kind=kind, model=model, ny=_log_int(rng, 32, 1500), nx=_log_int(rng, 32, 1500),
                    h=rng.uniform(0.8, 1.6), dt=rng.choice([0.25, 0.5]),
                    kappa=rng.uniform(0.5, 1.0), steps=rng.randrange(1, 4))
    if kind == "grains":
        return dict(kind=kind, n=_log_int(rng, 24, 128), nf=rng.choice([1, 3, 5, 8]),
                    dt=rng.choice([0.25, 0.5]))
    if kind == "eshelby":
        return dict(kind=kind, n=_log_int(rng, 24, 129))
    if kind == "predict":
        return dict(kind=kind, d=16 * rng.randrange(1, 9), h=rng.choice([64, 128]),
                    w=rng.choice([64, 128]), history=rng.choice([1, 2]))
    return dict(kind=kind, d=16 * rng.randrange(1, 5), h=64, w=64, batch=rng.randrange(1, 5),
                history=rng.choice([1, 2]))


# --- inputs -----------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _explicit_inputs(case, seed):
    amp = 0.05
    return 0.5 + amp * (2 * _rand(_gen(seed), case["ny"], case["nx"]) - 1)


def _coupled_inputs(case, seed):
    """[c; eta]: tanh disks of eta (radii 5 .. 15 % of the shorter side), noisy c."""
    g, ny, nx = _gen(seed), case["ny"], case["nx"]
    y = torch.arange(ny, device="cuda", dtype=F64)[:, None]
    x = torch.arange(nx, device="cuda", dtype=F64)[None, :]
    eta = torch.zeros(ny, nx, device="cuda", dtype=F64)
    for cx, cy, r in _rand(g, 12, 3).double().tolist():
        d = ((x - cx * (nx - 1)) ** 2 + (y - cy * (ny - 1)) ** 2).sqrt()
        rad = (0.05 + 0.10 * r) * min(nx, ny)
        eta = torch.maximum(eta, 0.5 * (1 - torch.tanh((d - rad) / 2.0)))
    c = 0.6 + 0.02 * (2 * _rand(g, ny, nx) - 1)
    return torch.stack([c, eta.float()])


def _ensemble_shapes(case):
    """Instance sizes, from the case alone: the shapes of a study are the same for every seed."""
    r = random.Random(case["count"] * 1000003 + case["lo"] * 1009 + case["hi"])
    q = case["grid"]
    if q == 128:  # square instances of 128, 256, 384 or 512
        return [(n, n) for n in (q * r.randrange(1, 5) for _ in range(case["count"]))]
    side = lambda: max(4, r.randrange(case["lo"], case["hi"] + 1) // q * q)  # noqa: E731
    return [(side(), side()) for _ in range(case["count"])]


def _ensemble_inputs(case, seed):
    """Parameters log-uniform in [0.5, 2] and start fields from the seed."""
    shapes = _ensemble_shapes(case)
    s = random.Random(seed)
    params = [dict(dt=0.01, **{k: math.exp(s.uniform(math.log(0.5), math.log(2.0)))
                               for k in ("W", "kappa", "L")}) for _ in shapes]
    total = sum(a * b for a, b in shapes)
    return shapes, params, 0.45 + 0.1 * _rand(_gen(seed), total)


def _mobility(g, ny, nx):
    """1 + 8 Gaussian bumps, amplitudes 0.2 .. 0.8, widths 16 .. 64 nodes."""
    y = torch.arange(ny, device="cuda", dtype=F64)[:, None]
    x = torch.arange(nx, device="cuda", dtype=F64)[None, :]
    m = torch.ones(ny, nx, device="cuda", dtype=F64)
    for a, s, cx, cy in _rand(g, 8, 4).double().tolist():
        r2 = (x - cx * (nx - 1)) ** 2 + (y - cy * (ny - 1)) ** 2
        m = m + (0.2 + 0.6 * a) * torch.exp(-r2 / (2 * (16 + 48 * s) ** 2))
    return m.float()


def _misfit_inputs(case, seed):
    g, ny, nx = _gen(seed), case["ny"], case["nx"]
    mob = _mobility(g, ny, nx)
    c0 = 0.5 + 0.05 * (2 * _rand(g, ny, nx) - 1)
    y = torch.arange(ny, device="cuda", dtype=F64)[:, None]
    x = torch.arange(nx, device="cuda", dtype=F64)[None, :]
    k, p = (0.2 + 0.2 * _rand(g, 2).double()).tolist(), (6.28 * _rand(g, 2).double()).tolist()
    target = (0.5 + 0.03 * torch.sin(k[0] * x + p[0]) * torch.sin(k[1] * y + p[1])).float()
    return mob, c0, target


_MISFIT = dict(kappa=0.5, W=1.0, M=1.0, dt=1e-3)


def _implicit2d_inputs(case, seed):
    g = _gen(seed)
    if case["model"] == "ac":
        return 0.2 + 0.6 * _rand(g, case["ny"], case["nx"])
    return 0.5 + 0.05 * (2 * _rand(g, case["ny"], case["nx"]) - 1)


def _grain_fields(g, shape, nf, grains=64, width=2.0):
    """Voronoi grains with tanh interfaces, grain i carried by order parameter i mod nf:
    the profile of a polycrystal some steps into its coarsening."""
    z, y, x = (torch.arange(n, device="cuda", dtype=F64) for n in shape)
    pts = (_rand(g, grains, 3).cpu().double() * (torch.tensor(shape) - 1)).tolist()
    best = torch.full((max(nf, 2),) + shape, math.inf, device="cuda", dtype=F64)
    for i, (pz, py, px) in enumerate(pts):  # distance to each order parameter's nearest seed
        d = ((z[:, None, None] - pz) ** 2 + (y[None, :, None] - py) ** 2
             + (x[None, None, :] - px) ** 2).sqrt()
        k = i % best.shape[0]
        torch.minimum(best[k], d, out=best[k])
    two = torch.topk(best, 2, dim=0, largest=False).values
    other = torch.where(best == two[:1], two[1:2], two[:1])
    return (0.5 * (1 - torch.tanh((best - other) / (2 * width))))[:nf].float().contiguous()


_FC = dict(kappa=1.0, mobility=1.0, alpha=1.0, beta=1.0, gamma=1.5, shift=0.0)


def _eshelby_params(case, seed):
    r = random.Random(seed)
    return dict(E=r.uniform(20.0, 25.0), nu=r.uniform(0.28, 0.32), m=r.uniform(0.008, 0.012),
                l=0.5, a=r.uniform(18.0, 22.0))


def _crops(case, seed, samples):
    """Consecutive states of grain-like fields under slow interface motion, newest first."""
    g, shape = _gen(seed), (case["d"], case["h"], case["w"])
    out = []
    for _ in range(samples):
        u = _grain_fields(g, shape, 8, grains=12)
        rate = 0.02 * (0.5 + _rand(g, 8, 1, 1, 1))
        states = [u]
        for _ in range(3):
            u = u + rate * u * (1 - u) * (u - 0.4)
            states.append(u)
        out.append(torch.stack(states[::-1]))
    return torch.stack(out)  # [sample][4 states, newest first][8][d][h][w]


_LAYERS = [(32, 32)] * 14 + [(32, 16)]
_TRAIN = dict(lr=3e-4, stiff=0.5)


def _net_params(g, history):
    """He-normal weights (unused input and output channels zero), small biases."""
    chunks = []
    for k, (ci, co) in enumerate(_LAYERS):
        used = 8 * (history + 1) if k == 0 else ci
        w = torch.randn(27, co, ci, generator=g, device="cuda") * math.sqrt(2 / (27 * used))
        b = 0.01 * torch.randn(co, generator=g, device="cuda")
        w[:, :, used:] = 0
        if k == len(_LAYERS) - 1:
            w[:, 8:] = 0
            w *= 0.1
            b[8:] = 0
        chunks += [w.reshape(-1), b]
    return torch.cat(chunks)


def _train_inputs(case, seed):
    h = case["history"]
    s = _crops(case, seed, case["batch"])
    x = s[:, 1:h + 2].flatten(1, 2).contiguous()
    g = _gen(seed + 1)
    p = _net_params(g, h)
    m = 1e-3 * torch.randn(p.shape, generator=g, device="cuda")
    v = 1e-6 * (0.5 + _rand(g, *p.shape))
    return x, s[:, 0].contiguous(), p, m, v


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, case=case)
    if kind == "explicit":
        s = pf.Solver((case["ny"], case["nx"]), h=(case["hx"], case["hy"]), model=case["model"])
        s.set_params(W=1.0, kappa=case["kappa"], mobility=1.0, dt=case["dt"])
        st.update(solver=s, u0=_explicit_inputs(case, seed))
    elif kind == "coupled":
        s = pf.Solver((case["ny"], case["nx"]), h=(case["hx"], case["hy"]), model="coupled")
        s.set_params(kappa=0.3, mobility=1.0, mobility2=150.0, dt=1e-3)
        st.update(solver=s, u0=_coupled_inputs(case, seed))
    elif kind == "ensemble":
        shapes, params, u0 = _ensemble_inputs(case, seed)
        e = pf.Ensemble(shapes)
        e.set_params(params)
        e.tune()
        st.update(ens=e, u0=u0)
    elif kind == "misfit":
        mob, c0, target = _misfit_inputs(case, seed)
        scalars = [torch.tensor(_MISFIT[k], dtype=torch.float32, device="cuda", requires_grad=True)
                   for k in ("kappa", "W", "M")]
        st.update(mob=mob.requires_grad_(), scalars=scalars, c0=c0, target=target)
    elif kind == "implicit2d":
        s = pf.Solver((case["ny"], case["nx"]), h=case["h"], model=case["model"])
        s.set_params(W=1.0, kappa=case["kappa"], mobility=1.0, dt=case["dt"])
        st.update(solver=s, u0=_implicit2d_inputs(case, seed))
    elif kind == "grains":
        n = case["n"]
        s = pf.Solver((n, n, n), model="fanchen", n_fields=case["nf"])
        s.set_params(dt=case["dt"], **_FC)
        st.update(solver=s, u0=_grain_fields(_gen(seed), (n, n, n), case["nf"]))
    elif kind == "eshelby":
        n = case["n"]
        st.update(elastic=pf.Elastic((n, n, n), h=100.0 / (n - 1), **_eshelby_params(case, seed)))
    elif kind == "predict":
        surr = pf.Surrogate(history=case["history"])
        surr.params.copy_(_net_params(_gen(seed + 1), case["history"]))
        x = _crops(case, seed, 1)[:, :case["history"] + 1].flatten(1, 2).contiguous()
        st.update(surr=surr, x=x)
    else:
        surr = pf.Surrogate(history=case["history"])
        x, y, p, m, v = _train_inputs(case, seed)
        surr.params.copy_(p)
        surr.m.copy_(m)
        surr.v.copy_(v)
        surr.step = 1000
        st.update(surr=surr, x=x, y=y)
    if "u0" in st:
        st["u"] = st["u0"].clone()
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind in ("explicit", "coupled"):
        st["u"].copy_(st["u0"])
        return st["solver"].step_explicit(st["u"], case["steps"])
    if kind == "ensemble":
        st["u"].copy_(st["u0"])
        return st["ens"].step(st["u"], case["steps"], case["mode"])
    if kind == "misfit":
        k, w, m = st["scalars"]
        leaves = [st["mob"], k, w, m]
        loss = pf.ch_misfit(st["mob"], k, w, m, st["c0"], st["target"], _MISFIT["dt"],
                            case["steps"], ckpt_every=case["ckpt"])
        grads = torch.autograd.grad(loss, leaves)
        return dict(loss=loss.float(), mobility=grads[0], kappa=grads[1], W=grads[2], M=grads[3])
    if kind == "implicit2d":
        st["u"].copy_(st["u0"])
        st["solver"].step_implicit(st["u"], case["steps"])
        return st["u"]
    if kind == "grains":
        st["u"].copy_(st["u0"])
        st["solver"].step_implicit(st["u"], 1)
        return st["u"]
    if kind == "eshelby":
        return st["elastic"].solve()
    if kind == "predict":
        return st["surr"].predict(st["x"])
    surr = st["surr"]
    loss = surr.train_step(st["x"], st["y"], **_TRAIN)
    return dict(params=surr.params, m=surr.m, v=surr.v,
                loss=torch.tensor(loss, dtype=torch.float32))


# --- least work -------------------------------------------------------------

def _net_flops(voxels):
    level = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    return sum(2 * 27 * ci * co * voxels // 8 ** lv for (ci, co), lv in zip(_LAYERS, level))


def work(case):
    """Each input once in, each output once out, and the arithmetic of the method
    (Gauss-point terms, projections and stencils, counted per node and step; 20 GMRES
    iterations per implicit step and 5 n CG iterations as typical solves)."""
    kind = case["kind"]
    nodes = case.get("ny", 0) * case.get("nx", 0)
    if kind == "explicit":
        return dict(bytes=8 * nodes,
                    flops=(60 if case["model"] == "ac" else 73) * nodes * case["steps"])
    if kind == "coupled":
        return dict(bytes=16 * nodes, flops=190 * nodes * case["steps"])
    if kind == "ensemble":
        nodes = sum(a * b for a, b in _ensemble_shapes(case))
        return dict(bytes=8 * nodes, flops=60 * nodes * case["steps"])
    if kind == "misfit":
        return dict(bytes=20 * nodes, flops=(2 * 110 + 330) * nodes * case["steps"])
    if kind == "implicit2d":
        per = (70 if case["model"] == "ac" else 95) + 4 * 2 * 10
        return dict(bytes=8 * nodes, flops=20 * per * nodes * case["steps"])
    if kind == "grains":
        v = case["n"] ** 3 * case["nf"]
        return dict(bytes=8 * v, flops=10 * 400 * v)
    if kind == "eshelby":
        v = case["n"] ** 3
        return dict(bytes=12 * v, flops=5 * case["n"] * (267 + 30) * v)
    v = case["d"] * case["h"] * case["w"] * case.get("batch", 1)
    states = 8 * (case["history"] + 1)
    count = sum(27 * ci * co + co for ci, co in _LAYERS)
    if kind == "predict":
        return dict(bytes=4 * v * (states + 8) + 4 * count, flops=_net_flops(v))
    return dict(bytes=4 * v * (states + 8) + 24 * count, flops=3 * _net_flops(v))


# --- FP64 evaluation --------------------------------------------------------
#
# On a uniform grid with zero-flux boundaries the Q1 operators divided by the
# lumped mass are the interior formulas on the field mirrored about its end
# nodes.  The node axes are the last `dim` ones, x last; h is given x first.

def _pad(u, ax):
    n = u.shape[ax]
    return torch.cat((u.narrow(ax, 1, 1), u, u.narrow(ax, n - 2, 1)), ax)


def _tri(u, ax, side, mid):
    n, p = u.shape[ax], _pad(u, ax)
    return mid * u + side * (p.narrow(ax, 0, n) + p.narrow(ax, 2, n))


def _stiff(u, h):
    """M^-1 K u."""
    dim, out = len(h), 0
    for d in range(dim):
        t = u
        for e in range(dim):
            t = _tri(t, -1 - e, -1 / h[e] ** 2, 2 / h[e] ** 2) if e == d else \
                _tri(t, -1 - e, 1 / 6, 2 / 3)
        out = out + t
    return out


def _interp(p, ax):
    n = p.shape[ax] - 1
    lo, hi = p.narrow(ax, 0, n), p.narrow(ax, 1, n)
    return GH * lo + GL * hi, GL * lo + GH * hi


def _gauss(u, dim):
    """Values at the 2^dim Gauss points of every element of the mirrored mesh."""
    q = [u]
    for e in range(dim):
        q = [v for p in q for v in _interp(_pad(p, -1 - e), -1 - e)]
    return q


def _back(lo, hi, ax):
    n = lo.shape[ax] - 1
    return 0.5 * (GL * lo.narrow(ax, 0, n) + GH * hi.narrow(ax, 0, n)
                  + GH * lo.narrow(ax, 1, n) + GL * hi.narrow(ax, 1, n))


def _project(q, dim):
    """M^-1 sum_e sum_q w N_i(q) v_q."""
    for e in reversed(range(dim)):
        q = [_back(q[2 * i], q[2 * i + 1], -1 - e) for i in range(len(q) // 2)]
    return q[0]


def _well1(u, W=1.0):
    return 2 * W * u * (1 - u) * (1 - 2 * u)


def _well2(u, W=1.0):
    return 2 * W * (1 - 6 * u + 6 * u * u)


def _grad_flow(u, f1, kappa, h):
    return _project([f1(q) for q in _gauss(u, len(h))], len(h)) + kappa * _stiff(u, h)


def _exact_explicit(case, seed):
    u, h = _explicit_inputs(case, seed).double(), (case["hx"], case["hy"])
    for _ in range(case["steps"]):
        r = _grad_flow(u, _well1, case["kappa"], h)
        u = u - case["dt"] * (r if case["model"] == "ac" else _stiff(r, h))
    return u


def _poly(a, x):
    s = torch.full_like(x, a[-1])
    for c in reversed(a[:-1]):
        s = s * x + c
    return s


def _dpoly(a, x):
    return _poly([k * a[k] for k in range(1, len(a))], x)


_FA = [-1.6704, -4.776, 5.1622, -2.7375, 1.3687]  # free energies and interpolation of the
_FB = [-1.5924, -5.9746, 5.0]                     # coupled model, increasing powers
_H = [0.0, 0.0, 0.0, 10.0, -15.0, 6.0]


def _exact_coupled(case, seed):
    c, e = _coupled_inputs(case, seed).double()
    h = (case["hx"], case["hy"])
    for _ in range(case["steps"]):
        qc, qe = _gauss(c, 2), _gauss(e, 2)
        gc, ge = [], []
        for a, b in zip(qc, qe):
            w = _poly(_H, b)
            gc.append(_dpoly(_FA, a) * (1 - w) + _dpoly(_FB, a) * w)
            ge.append((_poly(_FB, a) - _poly(_FA, a)) * _dpoly(_H, b))
        re = _project(ge, 2) + 0.3 * _stiff(e, h)
        c, e = c - 1e-3 * _stiff(_project(gc, 2), h), e - 1e-3 * 150.0 * re
    return torch.stack([c, e])


def _exact_ensemble(case, seed):
    shapes, params, u0 = _ensemble_inputs(case, seed)
    offs = [0]
    for a, b in shapes:
        offs.append(offs[-1] + a * b)
    out = torch.empty(u0.shape, dtype=F64, device="cuda")
    for shape in sorted(set(shapes)):
        which = [i for i, s in enumerate(shapes) if s == shape]
        u = torch.stack([u0[offs[i]:offs[i + 1]].view(shape) for i in which]).double()
        par = lambda k: torch.tensor([params[i][k] for i in which], dtype=F64,  # noqa: E731
                                     device="cuda")[:, None, None]
        W, kappa, L = par("W"), par("kappa"), par("L")
        for _ in range(case["steps"]):
            u = u - 0.01 * L * _grad_flow(u, lambda q: _well1(q, W), kappa, (1.0, 1.0))
        for j, i in enumerate(which):
            out[offs[i]:offs[i + 1]] = u[j].reshape(-1)
    return out


def _mob_stiff(u, m, M):
    """M^-1 K_M u on unit cells, M_q = M times the interpolated node multipliers."""
    mq = _gauss(m, 2)  # x first: index 2 * (x point) + (y point)
    px, py = _pad(u, -1), _pad(u, -2)
    gx = _interp(_pad(px[..., 1:] - px[..., :-1], -2), -2)  # du/dx at the two y points
    gy = _interp(_pad(py[..., 1:, :] - py[..., :-1, :], -1), -1)
    fx = [gx[j] * M * 0.5 * (mq[j] + mq[2 + j]) for j in (0, 1)]
    fy = [gy[j] * M * 0.5 * (mq[2 * j] + mq[2 * j + 1]) for j in (0, 1)]
    fx, fy = _back(fx[0], fx[1], -2), _back(fy[0], fy[1], -1)
    return fx[..., :-1] - fx[..., 1:] + fy[..., :-1, :] - fy[..., 1:, :]


def _exact_misfit(case, seed):
    from torch.utils.checkpoint import checkpoint
    mob, c0, target = _misfit_inputs(case, seed)
    mob, c, target = mob.double().requires_grad_(), c0.double(), target.double()
    kappa, W, M = (torch.tensor(_MISFIT[k], dtype=F64, device="cuda", requires_grad=True)
                   for k in ("kappa", "W", "M"))

    def segment(c, n, *_):
        for _ in range(n):
            mu = _grad_flow(c, lambda q: _well1(q, W), kappa, (1.0, 1.0))
            c = c - _MISFIT["dt"] * _mob_stiff(mu, mob, M)
        return c

    left = case["steps"]
    while left > 0:
        n = min(50, left)
        c = checkpoint(segment, c, n, mob, kappa, W, M, use_reentrant=False)
        left -= n
    m = torch.ones_like(target)
    for ax in (0, 1):
        m.narrow(ax, 0, 1).mul_(0.5)
        m.narrow(ax, m.shape[ax] - 1, 1).mul_(0.5)
    loss = 0.5 * (m * (c - target) ** 2).sum()
    g = torch.autograd.grad(loss, [mob, kappa, W, M])
    return dict(loss=loss.detach(), mobility=g[0], kappa=g[1], W=g[2], M=g[3])


def _gmres(A, b, rtol, restart=60, cycles=20):
    x, b0 = torch.zeros_like(b), b.norm().item()
    for _ in range(cycles):
        r = b - A(x)
        beta = r.norm().item()
        if beta <= rtol * b0:
            break
        V = torch.empty((restart + 1, b.numel()), dtype=F64, device=b.device)
        H = torch.zeros((restart + 1, restart), dtype=F64)
        V[0] = r.reshape(-1) / beta
        e1 = torch.zeros(restart + 1, dtype=F64)
        e1[0] = beta
        k = 0
        while k < restart:
            w = A(V[k].view_as(b)).reshape(-1)
            for _ in range(2):
                hk = V[:k + 1] @ w
                w = w - hk @ V[:k + 1]
                H[:k + 1, k] += hk.cpu()
            H[k + 1, k] = w.norm().item()
            V[k + 1] = w / H[k + 1, k].item()
            k += 1
            y = torch.linalg.lstsq(H[:k + 1, :k], e1[:k + 1, None]).solution
            if (H[:k + 1, :k] @ y - e1[:k + 1, None]).norm().item() <= rtol * b0:
                break
        x = x + (y[:, 0].to(b.device) @ V[:k]).view_as(b)
    return x


def _newton(u0, G, J):
    """Root of the mass-scaled residual G from u0, to rounding in FP64."""
    u, first = u0.clone(), None
    for _ in range(30):
        g = G(u)
        size = g.norm().item()
        first = first or size or 1.0
        if size <= 1e-10 * first:
            break
        u = u - _gmres(lambda v: J(u, v), g, 1e-4)
    return u


def _exact_implicit2d(case, seed):
    u = _implicit2d_inputs(case, seed).double()
    h, kappa, dt = (case["h"],) * 2, case["kappa"], case["dt"]
    # Cahn-Hilliard with mu eliminated: (c - c^n)/dt + M^-1 K (M^-1 r(c)) = 0
    K = (lambda t: _stiff(t, h)) if case["model"] == "ch" else (lambda t: t)

    def hess(u, v):
        q = [_well2(a) * b for a, b in zip(_gauss(u, 2), _gauss(v, 2))]
        return _project(q, 2) + kappa * _stiff(v, h)

    for _ in range(case["steps"]):
        un = u
        u = _newton(un, lambda u: (u - un) / dt + K(_grad_flow(u, _well1, kappa, h)),
                    lambda u, v: v / dt + K(hess(u, v)))
    return u


def _exact_grains(case, seed):
    un = _grain_fields(_gen(seed), (case["n"],) * 3, case["nf"]).double()
    h, dt, two_g = (1.0,) * 3, case["dt"], 2 * _FC["gamma"]

    def f1(q):
        return -q + q ** 3 + two_g * q * ((q * q).sum(0) - q * q)

    def hess(u, v):
        out = []
        for a, b in zip(_gauss(u, 3), _gauss(v, 3)):
            s2, t = (a * a).sum(0), (a * b).sum(0)
            out.append((-1 + 3 * a * a + two_g * (s2 - a * a)) * b + 2 * two_g * a * (t - a * b))
        return _project(out, 3) + _stiff(v, h)

    return _newton(un, lambda u: (u - un) / dt + _grad_flow(u, f1, 1.0, h),
                   lambda u, v: v / dt + hess(u, v))


def _line(u, ax, left, mid, right, end0, end1):
    """A tridiagonal 1-D operator along an axis, the diagonal's end values given."""
    n = u.shape[ax]
    out = mid * u
    out.narrow(ax, 0, 1).add_((end0 - mid) * u.narrow(ax, 0, 1))
    out.narrow(ax, n - 1, 1).add_((end1 - mid) * u.narrow(ax, n - 1, 1))
    out.narrow(ax, 0, n - 1).add_(right * u.narrow(ax, 1, n - 1))
    out.narrow(ax, 1, n - 1).add_(left * u.narrow(ax, 0, n - 1))
    return out


def _exact_eshelby(case, seed):
    n, p = case["n"], _eshelby_params(case, seed)
    h = 100.0 / (n - 1)
    lam = p["E"] * p["nu"] / ((1 + p["nu"]) * (1 - 2 * p["nu"]))
    mu = p["E"] / (2 * (1 + p["nu"]))
    ax = {0: -1, 1: -2, 2: -3}  # x fastest
    mass = lambda u, d: _line(u, ax[d], h / 6, 2 * h / 3, h / 6, h / 3, h / 3)  # noqa: E731
    stiff = lambda u, d: _line(u, ax[d], -1 / h, 2 / h, -1 / h, 1 / h, 1 / h)  # noqa: E731
    grad = lambda u, d: _line(u, ax[d], -0.5, 0.0, 0.5, -0.5, 0.5)  # int N_a N_b'  # noqa: E731
    gradt = lambda u, d: _line(u, ax[d], 0.5, 0.0, -0.5, -0.5, 0.5)  # int N_a' N_b  # noqa: E731

    def clamp(v):
        for d in range(3):
            v[d].narrow(ax[d], 0, 1).zero_()
        return v

    def K(u):
        out = torch.zeros_like(u)
        for j in range(3):
            k, l = (j + 1) % 3, (j + 2) % 3
            mk, ml = mass(u[j], k), mass(u[j], l)
            lap = [None] * 3
            lap[j] = stiff(mass(mk, l), j)
            lap[k] = stiff(mass(ml, j), k)
            lap[l] = stiff(mass(mk, j), l)
            out[j] += (lam + mu) * lap[j] + mu * (lap[0] + lap[1] + lap[2])
            for i, m in ((k, ml), (l, mk)):  # coupling to component i, mass along the third axis
                out[i] += lam * gradt(grad(m, j), i) + mu * grad(gradt(m, j), i)
        return clamp(out)

    x = torch.arange(n - 1, device="cuda", dtype=F64)
    b = torch.zeros((3, n, n, n), dtype=F64, device="cuda")
    for q in range(8):
        g = [(q >> d) & 1 for d in range(3)]
        pos = [(x + (GH if s else GL)) * h for s in g]
        r = (pos[0][None, None, :] ** 2 + pos[1][None, :, None] ** 2
             + pos[2][:, None, None] ** 2).sqrt()
        s = (3 * lam + 2 * mu) * p["m"] * h * h / 8 * 0.5 * (1 - torch.tanh(p["l"] * (r - p["a"])))
        for a in range(8):
            c = [(a >> d) & 1 for d in range(3)]
            N = [GH if c[d] == g[d] else GL for d in range(3)]
            node = tuple(slice(c[d], c[d] + n - 1) for d in (2, 1, 0))
            for d in range(3):
                w = (1 if c[d] else -1) * N[(d + 1) % 3] * N[(d + 2) % 3]
                b[d][node] += w * s
    clamp(b)
    u, r = torch.zeros_like(b), b.clone()
    d, rr = r.clone(), (r * r).sum()
    stop = 1e-20 * rr.item()
    for it in range(4000):
        Ad = K(d)
        alpha = rr / (d * Ad).sum()
        u += alpha * d
        r -= alpha * Ad
        new = (r * r).sum()
        if it % 20 == 0 and new.item() <= stop:
            break
        d = r + (new / rr) * d
        rr = new
    return u


def _net(params, x):
    F = torch.nn.functional
    W, o = [], 0
    for ci, co in _LAYERS:
        n = 27 * ci * co
        W.append((params[o:o + n].view(3, 3, 3, co, ci).permute(3, 4, 0, 1, 2),
                  params[o + n:o + n + co]))
        o += n + co

    def conv(k, t):
        p = F.pad(t, (1,) * 6)
        d, e, f = t.shape[-3:]
        w, b = W[k]
        y = b.view(1, -1, 1, 1, 1)
        for tap in range(27):
            z, v, u = tap // 9, tap // 3 % 3, tap % 3
            y = y + torch.einsum("oc,bczyx->bozyx", w[:, :, z, v, u],
                                 p[..., z:z + d, v:v + e, u:u + f])
        return torch.relu(y) if k < 14 else y

    up = lambda t: F.interpolate(t, scale_factor=2, mode="nearest")  # noqa: E731
    pool = lambda t: F.avg_pool3d(t, 2)  # noqa: E731
    a = conv(1, conv(0, F.pad(x, (0,) * 6 + (0, 32 - x.shape[1])))); s0 = a  # noqa: E702
    a = conv(3, conv(2, pool(a))); s1 = a  # noqa: E702
    a = conv(5, conv(4, pool(a))); s2 = a  # noqa: E702
    a = conv(7, conv(6, pool(a)))
    a = conv(9, conv(8, up(a) + s2))
    a = conv(11, conv(10, up(a) + s1))
    return conv(14, conv(13, conv(12, up(a) + s0)))[:, :8]


def _history(x):
    """(network input, extrapolation, output unit) of states [U^n; U^{n-1}; ...]."""
    s = [x[:, 8 * k:8 * k + 8] for k in range(x.shape[1] // 8)]
    rms = lambda t: t.pow(2).mean(dim=(1, 2, 3, 4), keepdim=True).sqrt()  # noqa: E731
    unit = rms(s[0] - s[1])
    inp = torch.cat([s[0]] + [(s[k] - s[k + 1]) / unit for k in range(len(s) - 1)], 1)
    if len(s) == 2:
        return inp, 2 * s[0] - s[1], unit
    curve = torch.maximum(rms(s[0] - 2 * s[1] + s[2]), 1e-3 * unit)
    return inp, 3 * s[0] - 3 * s[1] + s[2], curve


def _exact_predict(case, seed):
    x = _crops(case, seed, 1)[:, :case["history"] + 1].flatten(1, 2).double()
    inp, base, unit = _history(x)
    return base + unit * _net(_net_params(_gen(seed + 1), case["history"]).double(), inp)


def _exact_train(case, seed):
    x, y, p, m, v = (t.double() for t in _train_inputs(case, seed))
    inp, base, unit = _history(x)
    p.requires_grad_()
    e = _net(p, inp) - (y - base) / unit
    w = torch.ones(e.shape[-3:], dtype=F64, device="cuda")
    for ax in range(3):
        w.narrow(ax, 0, 1).mul_(0.5)
        w.narrow(ax, w.shape[ax] - 1, 1).mul_(0.5)
    loss = ((e + _TRAIN["stiff"] * w * _stiff(e, (1.0,) * 3)) ** 2).mean()
    g, = torch.autograd.grad(loss, p)
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    step = 1001
    p = p.detach() - _TRAIN["lr"] * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return dict(params=p, m=m, v=v, loss=loss.detach())


def exact(case, seed):
    return {"explicit": _exact_explicit, "coupled": _exact_coupled, "ensemble": _exact_ensemble,
            "misfit": _exact_misfit, "implicit2d": _exact_implicit2d, "grains": _exact_grains,
            "eshelby": _exact_eshelby, "predict": _exact_predict,
            "train": _exact_train}[case["kind"]](case, seed)
