"""The performance cases of this repository: what a user's program has the time step do.

A program plans the operator of its fault once (``fdph.Plan``) and then marches: in chunks of
prescribed slip rates (``run``, from host buffers ``run_host``), as a dynamic rupture
(``rupture_run``; a serving loop steps several scenarios side by side, each on its plan's stream), or
step by step with its own local law (``predict`` / ``commit``) or its own coupling (``step``).  A case is one of these with a
fault, a size and the plan's options; a pass is the next chunk of ``steps`` steps of a march that is
already under way (``warm`` steps taken, so that the windows of the near field are full), and a
march that has come to its planned end starts again from rest.

Plans with FP32 or FP16 storage multiply in FP32, so their tractions hold single precision and are
kept so (``float32``); FP64 plans return ``float64``.
"""
import math

import numpy as np
import torch

from paper_1903_02118_gb300 import fdph, inputs

PRECISION = {"fp64": fdph.FP64, "fp32": fdph.FP32, "fp16": fdph.FP16}

# options that a case leaves out
DEFAULTS = dict(kind="run", fault="curved", n=1024, M=1024, cfl=0.5, eps=1e-4, eta=0.5, eps_st=1e-4, soe=16,
                precision="fp32", nrhs=1, leaf=32, lmin=0.0, scheme=0, extra=-1, aca=4096, warm=256, steps=64,
                plans=1)


def _case(name, **kw):
    return dict({"name": name}, **kw)


def listed():
    return [
        # the plain step of Eq. 4 from buffers the caller owns (no allocation): the smallest call
        _case("plain-step-256", kind="noalloc", n=256, M=256, precision="fp64"),
        # the plain space-time BIEM march (no approximation) of the smallest configuration, whole
        _case("plain-march-256", kind="march", fault="straight", n=256, M=256, eps=0.0, eta=0.0, eps_st=0.0, soe=0,
              precision="fp64", aca=0, warm=0, steps=256),
        # a program with its own local law takes the step in two halves, one step a pass; a kinked fault of
        # ragged size in the library's default precision and Domain-S threshold
        _case("own-law-1100-fp64", kind="law", fault="kinked", n=1100, M=1 << 17, eps_st=1e-6, soe=0,
              precision="fp64", steps=1),
        # slip rates and tractions in host memory, copied every step
        _case("host-1024-fp32", kind="run_host", n=1024, M=1024),
        # the same march in double precision
        _case("curved-1500-fp64", n=1500, M=1500, precision="fp64", warm=320, steps=32),
        # the benchmark's workload: curved fault, FP32 storage, 16 exponential tail terms
        _case("curved-4096-fp32", n=4096, M=4096, warm=384),
        # the more accurate admissibility (constant eta^2 dist): small leaves, a far field that weighs more
        _case("eta2dist-1500-fp32", n=1500, M=1500, eta=0.25, scheme=1, lmin=8.0, leaf=8, extra=2, warm=320, steps=32),
        # a planar fault with a small eta and half-precision windows: the most accurate setting of a size
        _case("planar-1601-fp16", fault="straight", n=1601, M=2048, eta=0.125, precision="fp16", warm=640, steps=32),
        # four slip-rate histories on one operator of ragged leaves, half-precision windows
        _case("four-rhs-2500-fp16", fault="kinked", n=2500, M=1 << 17, eps_st=1e-5, soe=0, precision="fp16", nrhs=4,
              warm=320, steps=32),
        # the large fault of eight histories, the paper's Domain-S cut, planned by cross approximation
        _case("eight-rhs-6000-fp16", n=6000, M=1 << 17, soe=0, precision="fp16", nrhs=8, steps=16),
        # dynamic rupture of a planar fault with linear slip weakening
        _case("rupture-8192-fp32", kind="rupture", fault="straight", n=8192, M=1 << 17, soe=0),
        # a serving loop's chunk: rupture scenarios of mixed sizes side by side
        _case("serving-three-fp32", kind="serving", n=1300, M=1 << 17, soe=0, plans=3),
    ]


def draw(rng):
    """A case of the same ranges: sizes over their logarithm (odd ones among them), every entry
    point, precision and number of right-hand sides."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["noalloc", "march", "law", "step", "run", "run", "run", "run_host", "rupture", "serving"])
    if kind == "noalloc":
        n = size(32, 400)
        return dict(kind=kind, n=n, M=size(16, 300), precision="fp64")
    if kind == "march":
        return dict(kind=kind, fault=rng.choice(["straight", "kinked"]), n=size(64, 400), M=size(64, 300), eps=0.0,
                    eta=0.0, eps_st=0.0, soe=0, precision=rng.choice(["fp64", "fp32"]), aca=0, warm=0, steps=0)
    fault = rng.choice(["straight", "curved", "kinked"])
    prec = rng.choice(["fp64", "fp32", "fp16"])
    if kind in ("law", "step"):
        return dict(kind=kind, fault=fault, n=size(300, 2500), M=1 << 17, eps_st=1e-5, soe=0, precision=prec,
                    steps=1)
    if kind == "rupture":
        return dict(kind=kind, fault=fault, n=size(500, 4000), M=1 << 17, soe=0, cfl=rng.choice([0.25, 0.5]),
                    precision=rng.choice(["fp64", "fp32"]))
    if kind == "serving":
        return dict(kind=kind, n=size(300, 1000), M=1 << 17, soe=0, plans=rng.randint(2, 4),
                    precision=rng.choice(["fp64", "fp32"]))
    n = size(300, 2500)
    if kind == "run_host":
        return dict(kind=kind, fault=fault, n=n, M=1 << 17, eps_st=1e-5, soe=0, precision=prec,
                    steps=rng.choice([7, 24, 64]))
    soe = rng.choice([0, 16])
    nrhs = rng.choice([1, 1, 2, 4, 8])
    return dict(kind=kind, fault=fault, n=n, M=max(n, 1024) if soe else 1 << 17, eps_st=1e-4 if soe else 1e-5, soe=soe,
                precision=prec, nrhs=nrhs, leaf=rng.choice([13, 32]), eta=rng.choice([0.25, 0.5]) if nrhs == 1 else 0.5,
                steps=rng.choice([5, 16, 50, 64]) if n < 2000 else 32)


def _full(case):
    return dict(DEFAULTS, **case)


def _fault(c, n):
    # the traces are those of the repository's workloads (the seed of a case draws its histories)
    if c["fault"] == "straight":
        return inputs.straight_fault(n)
    if c["fault"] == "kinked":
        return inputs.kinked_fault(n)
    return inputs.curved_fault(n, inputs.seed_for(1, inputs.GEOMETRY))


def _pulses(steps, nrhs, n, seed, device="cuda"):
    """Slip rates [steps, nrhs, n]: Gaussian pulses in space (16 elements) and time (8 steps), as the
    benchmark's, one for every 128 elements, at random places, times and strengths."""
    rng = np.random.default_rng(inputs.seed_for(seed, inputs.SLIP))
    count = max(4, n // 128)
    out = torch.empty((steps, nrhs, n), dtype=torch.float64, device=device)
    s = torch.arange(n, dtype=torch.float64, device=device)
    t = torch.arange(steps, dtype=torch.float64, device=device) + 0.5
    for r in range(nrhs):
        s0 = torch.from_numpy(rng.uniform(0.0, n, count)).to(device)
        t0 = torch.from_numpy(rng.uniform(0.0, steps + 16.0, count)).to(device)
        a = torch.from_numpy(rng.uniform(0.25, 1.0, count)).to(device)
        space = torch.exp(-((s[None, :] - s0[:, None]) ** 2) / (2.0 * 16.0 ** 2))
        time = a[None, :] * torch.exp(-((t[:, None] - t0[None, :]) ** 2) / (2.0 * 8.0 ** 2))
        out[:, r] = time @ space
    return out


def _prestress(n, seed):
    """Background traction of a rupture: 0.45 with 5 % heterogeneity, an overstressed patch in the middle."""
    rng = np.random.default_rng(inputs.seed_for(seed, inputs.FRICTION))
    tau = 0.45 * (1.0 + 0.05 * rng.standard_normal(n))
    w = min(32, n // 8)
    tau[n // 2 - w:n // 2 + w] = 0.61
    return tau


def _plan(c, n, **kw):
    return fdph.Plan(_fault(c, n), c["cfl"], c["M"], c["eps"], eta=c["eta"], eps_st=c["eps_st"], soe_terms=c["soe"],
                     precision=PRECISION[c["precision"]], nrhs=c["nrhs"], leaf_size=c["leaf"], lmin=c["lmin"],
                     eta_scheme=c["scheme"], extra_steps=c["extra"], aca_min=c["aca"],
                     amp_window=0 if c["eta"] == 0.0 else 1, **kw)


def _noalloc_inputs(c, seed):
    """A kernel tensor [k][j][i] that decays with the lag and a ring of slip-rate rows."""
    n, W = c["n"], c["M"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    K = torch.randn((W, n, n), dtype=torch.float64, device="cuda", generator=gen)
    K /= (1.0 + torch.arange(W, dtype=torch.float64, device="cuda"))[:, None, None]
    return K, torch.randn((W, n), dtype=torch.float64, device="cuda", generator=gen)


def _sizes(c):
    """Sizes of a serving loop's scenarios: from the largest down to a third of it, odd ones among them."""
    k = c["plans"]
    return [max(64, int(c["n"] * 3.0 ** (-i / max(k - 1, 1)))) for i in range(k)]


class _Keep:
    """Single-precision copies of a plan's double buffers, ordered with the plan's stream."""

    def __init__(self, plan, single, *buffers):
        self.single = single
        self.buffers = buffers
        self.stream = torch.cuda.ExternalStream(plan.stream)
        self.copies = [torch.empty(b.shape, dtype=torch.float32, device=b.device) for b in buffers] if single else []

    def __call__(self):
        if not self.single:
            return list(self.buffers)
        with torch.cuda.stream(self.stream):
            for c, b in zip(self.copies, self.buffers):
                c.copy_(b)
        return list(self.copies)


def prepare(case, seed):
    c = _full(case)
    kind, n, single = c["kind"], c["n"], c["precision"] != "fp64"
    if kind == "noalloc":
        K, hist = _noalloc_inputs(c, seed)
        return dict(c=c, K=K, hist=hist, T=torch.empty(n, dtype=torch.float64, device="cuda"))
    if kind == "march":
        steps = c["M"]
        D = _pulses(steps, 1, n, seed)
        T = torch.empty_like(D)
        torch.cuda.synchronize()
        plan = _plan(c, n)
        return dict(c=c, plan=plan, steps=steps, D=D, T=T, keep=_Keep(plan, single, T))
    if kind in ("rupture", "serving"):
        plans, Ds, Ts, slips = [], [], [], []
        for i, m in enumerate(_sizes(c) if kind == "serving" else [n]):
            tau0 = torch.from_numpy(_prestress(m, seed + 100 * i)).cuda()
            D = torch.zeros((c["steps"], m), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            plan = _plan(c, m)
            plan.rupture_init(tau0, 1.0, 0.6, 0.3, 6.4)
            plans.append(plan)
            Ds.append(D)
            Ts.append(torch.zeros_like(D))
            slips.append(torch.zeros(m, dtype=torch.float64, device="cuda"))
        torch.cuda.synchronize()
        for plan, D, T in zip(plans, Ds, Ts):
            for _ in range(c["warm"] // c["steps"]):
                plan.rupture_run(c["steps"], D, T)
            plan.synchronize()
        keeps = [_Keep(p, single, D, T, s) for p, D, T, s in zip(plans, Ds, Ts, slips)]
        return dict(c=c, plans=plans, D=Ds, T=Ts, slip=slips, keeps=keeps)
    history = _pulses(c["warm"] + c["steps"], c["nrhs"], n, seed)
    torch.cuda.synchronize()
    plan = _plan(c, n)
    before = torch.empty((c["warm"], c["nrhs"], n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    plan.run(c["warm"], history, before)
    plan.synchronize()
    D = history[c["warm"]:].clone()
    if kind == "run_host":
        D = D.cpu().pin_memory()
        return dict(c=c, plan=plan, D=D, T=torch.empty(D.shape, dtype=torch.float64).pin_memory())
    T = torch.empty_like(D)
    s = dict(c=c, plan=plan, D=D, T=T)
    if kind == "law":
        # the caller's law: the traction stays at the strength wherever it would exceed it
        k0 = torch.from_numpy(plan.self_coefficients()).cuda()
        s["excess"] = torch.from_numpy(_prestress(n, seed)).cuda() - 0.3
        s["inverse"] = -1.0 / k0
        s["stream"] = torch.cuda.ExternalStream(plan.stream)
        s["D"] = torch.empty_like(T)
    s["keep"] = _Keep(plan, single, *((s["D"], T) if kind == "law" else (T,)))
    torch.cuda.synchronize()
    return s


def _again(plans, steps, M):
    """Marches that have come to their planned end start again from rest."""
    if plans[0].current_step() + steps > M:
        for p in plans:
            p.reset()


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "noalloc":
        fdph.plain_step_noalloc(s["K"], c["n"], c["M"], s["hist"], c["M"], c["M"] - 1, s["T"])
        return s["T"]
    if kind == "march":
        s["plan"].reset()
        s["plan"].run(s["steps"], s["D"], s["T"])
        return s["keep"]()
    if kind in ("rupture", "serving"):
        _again(s["plans"], c["steps"], c["M"])
        for plan, D, T, slip in zip(s["plans"], s["D"], s["T"], s["slip"]):
            plan.rupture_run(c["steps"], D, T)
            plan.rupture_slip(slip)
        return [k() for k in s["keeps"]]
    plan = s["plan"]
    _again([plan], c["steps"], c["M"])
    if kind == "run_host":
        plan.run_host(s["D"], s["T"])
        return s["T"].float() if c["precision"] != "fp64" else s["T"]
    if kind == "step":
        plan.step(s["D"], s["T"])
    elif kind == "law":
        plan.predict(s["T"])
        with torch.cuda.stream(s["stream"]):
            torch.add(s["excess"], s["T"], out=s["D"]).mul_(s["inverse"]).clamp_(min=0.0)
        plan.commit(s["D"])
    else:
        plan.run(c["steps"], s["D"], s["T"])
    return s["keep"]()


def _leaves(xy, c):
    return fdph.tree_export(xy, c["cfl"], eta=c["eta"], leaf_size=c["leaf"], lmin=c["lmin"], eta_scheme=c["scheme"],
                            extra_steps=c["extra"])


def _march_work(c, n):
    """What one chunk of steps on one fault cannot do without: every coefficient of the operator that
    is not zero read once a chunk (the window of a near pair holds its kernel from the arrival of the
    wave on, a far block its factors at a small rank and its waveforms), the slip rates in, the
    tractions out; a multiply-add of every coefficient for every step and history."""
    xy = _fault(c, n)
    tree = _leaves(xy, c)
    size = {"fp64": 8, "fp32": 4, "fp16": 2}[c["precision"]]
    far_size = 8 if size == 8 else 4
    cdt, dx = c["cfl"], 1.0
    nc = c["extra"] if c["extra"] >= 0 else math.ceil(10.0 * dx / cdt)
    mx, my = 0.5 * (xy[:, 0] + xy[:, 2]), 0.5 * (xy[:, 1] + xy[:, 3])
    # steps a near pair keeps its exact kernel after the wave has come: its passage and n_c more, or
    # until the remainder has decayed to eps_st
    if c["soe"]:
        keep = nc + 1.0 / cdt
    elif c["eps_st"] > 0:
        keep = math.sqrt(1.0 / (math.pi * cdt * c["eps_st"]))
    else:
        keep = c["M"]
    near = far = 0.0
    for lf in tree["leaves"]:
        pairs = lf["nr"] * lf["ns"]
        if lf["kind"] == 0:
            I = tree["perm"][lf["r0"]:lf["r0"] + lf["nr"]]
            J = tree["perm"][lf["s0"]:lf["s0"] + lf["ns"]]
            r = np.hypot(mx[I][:, None] - mx[J][None, :], my[I][:, None] - my[J][None, :])
            near += float(np.sum(np.maximum(np.minimum(keep, c["M"] - r / cdt), 1.0))) + pairs * (1 + c["soe"])
        else:
            far += 2.0 * 5 * (lf["nr"] + lf["ns"]) + 2.0 * float(np.sum(lf["Dm"]))
    return near, far, size, far_size


def work(case):
    c = _full(case)
    n, steps = c["n"], c["steps"] or c["M"]
    if c["kind"] == "noalloc":
        return {"bytes": 8.0 * (c["M"] * n * n + c["M"] * n + n), "flops": 2.0 * c["M"] * n * n}
    out = {"bytes": 0.0, "flops": 0.0}
    for m in _sizes(c) if c["kind"] == "serving" else [n]:
        if c["kind"] == "march":
            # lags 0 .. M - 1, and each is used from its step on
            out["bytes"] += 8.0 * (1 if c["precision"] == "fp64" else 0.5) * c["M"] * m * m + 16.0 * c["M"] * m
            out["flops"] += 1.0 * c["M"] * (c["M"] + 1) * m * m
            continue
        near, far, size, far_size = _march_work(c, m)
        out["bytes"] += near * size + far * far_size + 16.0 * steps * c["nrhs"] * m
        out["flops"] += 2.0 * (near + far) * steps * c["nrhs"]
    return out


# ---- the same outputs in 64 bits from the closed form of the kernel, all pairs and all lags

def _ramp_jump(p, seg, t1, t2):
    """R(t2) - R(t1) on the receivers' normals for unit slip rate on the segments (mu = cs = 1): the
    2-D antiplane response of a segment switched on at t = 0, from its two end points."""
    px, py, nx, ny = (v[:, None] for v in p)
    ax, ay, tx, ty, length = (v[None, :] for v in seg)
    dx, dy = px - ax, py - ay
    X, Y = dx * tx + dy * ty, dy * tx - dx * ty
    parts = []
    for end, sign in ((length - X, 1.0), (-X, -1.0)):
        r2 = end * end + Y * Y
        s1, s2 = (torch.sqrt(torch.clamp(t * t - r2, min=0.0)) for t in (t1, t2))
        ds = torch.where(s1 > 0, (t2 * t2 - t1 * t1) / torch.where(s1 > 0, s1 + s2, 1.0), s2) / r2

        def angle(t):
            R2 = t * t - Y * Y
            on = (R2 > 0) & (t > 0)
            return torch.where(on, torch.asin(torch.clamp(end / torch.sqrt(torch.where(on, R2, 1.0)), -1.0, 1.0)), 0.0)

        parts.append((sign * (angle(t2) - angle(t1) + end * ds), sign * Y * ds))
    normal = -(parts[0][0] + parts[1][0]) / (2.0 * math.pi)
    along = -(parts[0][1] + parts[1][1]) / (2.0 * math.pi)
    return nx * (along * tx - normal * ty) + ny * (along * ty + normal * tx)


def _table(xy):
    x = torch.from_numpy(np.ascontiguousarray(xy)).cuda()
    ex, ey = x[:, 2] - x[:, 0], x[:, 3] - x[:, 1]
    length = torch.sqrt(ex * ex + ey * ey)
    tx, ty = ex / length, ey / length
    return (0.5 * (x[:, 0] + x[:, 2]), 0.5 * (x[:, 1] + x[:, 3]), -ty, tx), (x[:, 0], x[:, 1], tx, ty, length)


def _plain_march(xy, dt, history, first):
    """Eq. 4 for the steps from `first` on: T[n] = sum_m K_m D[n - m], every lag and pair."""
    steps, nrhs, n = history.shape
    p, seg = _table(xy)
    T = torch.zeros((steps - first, nrhs, n), dtype=torch.float64, device="cuda")
    rows = max(1, min(n, (1 << 25) // n))
    for m in range(steps):
        lo = max(first, m)
        D = history[lo - m:steps - m].reshape(-1, n).T
        t1 = torch.tensor(m * dt, dtype=torch.float64, device="cuda")
        t2 = torch.tensor((m + 1) * dt, dtype=torch.float64, device="cuda")
        for i in range(0, n, rows):
            K = _ramp_jump(tuple(v[i:i + rows] for v in p), seg, t1, t2)
            T[lo - first:, :, i:i + rows] += (K @ D).T.reshape(-1, nrhs, K.shape[0])
    return T


def exact(case, seed):
    """Ruptures have no such value: their slip follows from the approximate operator's own tractions,
    and the plain operator gives another rupture.  The largest sizes would take minutes."""
    c = _full(case)
    kind, n = c["kind"], c["n"]
    if kind == "noalloc":
        K, hist = _noalloc_inputs(c, seed)
        # step M - 1: lag k meets row M - 1 - k
        return torch.einsum("kji,kj->i", K, hist.flip(0))
    if kind in ("rupture", "serving") or n > 5000:
        return None
    warm = 0 if kind == "march" else c["warm"]
    steps = c["M"] if kind == "march" else c["steps"]
    history = _pulses(warm + steps, c["nrhs"], n, seed)
    if kind == "law":
        p, seg = _table(_fault(c, n))
        history[warm:] = 0.0   # the step's own slip rate is what the law solves for
        T = _plain_march(_fault(c, n), c["cfl"], history, warm)
        # the instantaneous self term of a segment at its own midpoint, -1 / 2 up to its half length
        k0 = torch.full((n,), -0.5, dtype=torch.float64, device="cuda")
        excess = torch.from_numpy(_prestress(n, seed)).cuda() - 0.3
        return [torch.clamp((excess + T) / -k0, min=0.0), T]
    T = _plain_march(_fault(c, n), c["cfl"], history, warm)
    if kind == "run_host":
        return T.cpu()
    return [T]
