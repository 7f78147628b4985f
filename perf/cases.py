"""What is measured: the calls a cratering study makes, over the sizes it makes them at.

Solver cases step a run (or a batch of runs) that `prepare` has set up (where the flow
should be developed, from saved fields); every pass puts the prepared image back first, as
a restart from a checkpoint in device memory does, so that passes repeat.  Surrogate cases evaluate,
differentiate and train the crater network.
"""
import math

import numpy as np
import torch

from paper_2403_04267_gb300 import salec, surrogate, workloads as W

# --- the cases -----------------------------------------------------------------------------


def listed():
    return [
        # the smallest run: 100 x 100 cells, hydrodynamic, FP64, from impact on; every step is
        # a few short launches, so latency counts
        dict(name="plain_100_fp64", kind="step", physics="plain", nr=100, nz=100, radius=5.0, precision="fp64",
             warm=0, steps=96),
        # an ordinary full-method run: two materials, strength with damage, gravity, FP64
        dict(name="full_800_fp64", kind="step", physics="full", nr=800, nz=800, radius=20.0, precision="fp64",
             warm=48, steps=16),
        # the paper's verification grid (stretched cells, three hydrostatic layers, strength,
        # gravity, 512 x 532 cells) in the mixed form
        dict(name="layered_512x532_fp32", kind="step", physics="layered", nr=512, nz=532, radius=18.0,
             precision="fp32mix", warm=48, steps=16),
        # the large hydrodynamic run in both forms: most of the grid still at rest
        dict(name="large_4000_fp64", kind="step", physics="plain", nr=4000, nz=4000, radius=100.0, precision="fp64",
             warm=0, steps=48),
        dict(name="large_4000_fp32", kind="step", physics="plain", nr=4000, nz=4000, radius=100.0,
             precision="fp32mix", warm=0, steps=48),
        # a hydrodynamic run with much of its grid moving, on a ragged grid
        dict(name="active_1003x701_fp32", kind="step", physics="plain", nr=1003, nz=701, radius=150.0,
             precision="fp32mix", warm=96, steps=16),
        # a batch of the sampled impacts (200-800 cells a side), mixed form, one chunk of
        # batched steps: how training data and parameter studies are run
        dict(name="batch_16_fp32", kind="batch", runs=16, lo=200, hi=800, precision="fp32mix", warm=16, steps=16),
        # the surrogate asked for many draws at once, and for the held-out draws by every
        # member of an ensemble
        dict(name="infer_65536", kind="infer", members=1, batch=65536),
        dict(name="infer_8x255", kind="infer", members=8, batch=255),
        # loss and gradient of a minibatch
        dict(name="gradient_509", kind="gradient", batch=509),
        # full-batch training: one network, and the ensemble of eight in groups of two
        dict(name="train_3675", kind="train", members=1, group=1, batch=3675, steps=51),
        dict(name="train_8x3675", kind="train", members=8, group=2, batch=3675, steps=51),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "plain", "full", "layered", "batch", "infer", "gradient", "train"])
    if kind == "infer":
        members = rng.choice([1, 1, 4, 8])
        return dict(kind=kind, members=members, batch=max(1, _log(rng, 1, 65536) // members))
    if kind == "gradient":
        return dict(kind=kind, batch=_log(rng, 32, 4096))
    if kind == "train":
        members = rng.choice([1, 2, 3, 8])
        return dict(kind=kind, members=members, group=rng.choice([1, 2]) if members > 1 else 1,
                    batch=_log(rng, 256, 3675), steps=rng.choice([10, 27, 51]))
    precision = rng.choice(["fp64", "fp32mix"])
    if kind == "batch":
        return dict(kind=kind, runs=rng.randint(2, 10), lo=200, hi=rng.choice([400, 800]), precision=precision,
                    warm=16, steps=rng.choice([5, 10, 16]))
    if kind == "full":
        n = rng.randint(200, 800)
        return dict(kind="step", physics=kind, nr=n, nz=rng.randint(max(200, n // 2), n),
                    radius=float(rng.randint(8, 20)), precision=precision, warm=48, steps=rng.choice([8, 16, 21]))
    if kind == "layered":
        core = rng.randint(150, 462)
        return dict(kind="step", physics=kind, nr=core + 50, nz=core + 70, radius=18.0, precision=precision,
                    warm=48, steps=rng.choice([8, 16, 21]))
    nr, nz = _log(rng, 100, 3000), _log(rng, 100, 3000)
    n = min(nr, nz)
    if rng.random() < 0.5:
        return dict(kind="step", physics=kind, nr=nr, nz=nz, radius=float(max(4, n // 40)), precision=precision,
                    warm=0, steps=rng.choice([16, 37, 48]))
    return dict(kind="step", physics=kind, nr=min(nr, 1200), nz=min(nz, 1200), radius=float(max(4, min(n, 1200) // 5)),
                precision=precision, warm=48, steps=rng.choice([8, 16, 21]))


# --- inputs --------------------------------------------------------------------------------


def _spec(case, seed):
    """The workload dictionary of a single run: the repository's builders, with the impact
    speed (and the full method's cohesion and friction) drawn from the seed."""
    rng = np.random.default_rng([7, seed])
    nr, nz, rad = case["nr"], case["nz"], case["radius"]
    if case["physics"] == "plain":
        v = rng.uniform(8e3, 12e3)
        return W.impact(nr, nz, 10.0, W.basalt(), None, rad, v, int(round(0.7 * nz)), 16, pml_alpha=0.0)
    if case["physics"] == "full":
        tgt = W.basalt(strength=True, cohesion=math.exp(rng.uniform(math.log(3e6), math.log(3e7))),
                       friction=rng.uniform(0.4, 0.8))
        return W.impact(nr, nz, 25.0, tgt, W.iron(), rad, rng.uniform(10e3, 18e3), int(round(0.7 * nz)), 40,
                        gravity=1.62)
    w = W.chicxulub_stretched(nr - 50)
    w["projectile"]["vz"] = -rng.uniform(10e3, 14e3)
    return w


def _draws(case, seed):
    """The batch's impacts: the sampled distribution.  The sides, uniform on lo..hi cells, are
    the case's; speed, projectile and strength come from the seed."""
    out = []
    for k in range(case["runs"]):
        n = case["lo"] + int(W.uniform01(k, 0) * (case["hi"] - case["lo"] + 1))
        out.append(dict(W.batched_draw(1000 * (seed % 100000) + k), n=n))
    return out


def _net_inputs(case, seed):
    """Inputs uniform over the normalised parameter ranges and smooth targets of them."""
    g = torch.Generator(device="cuda").manual_seed(1 + seed)
    x = 2 * torch.rand(case["batch"], surrogate.N_IN, device="cuda", generator=g) - 1
    k = torch.linspace(0, 1, surrogate.N_OUT, device="cuda")
    t = torch.cos(2 * k * (x[:, :1] + 2)) * (1 + 0.3 * x[:, 1:2]) + 0.2 * k * x[:, 2:3] * x[:, 3:4] - 0.1 * x[:, 4:]
    return x.contiguous(), t.float().contiguous()


def _theta(seed, member):
    return W.mlp_init(1000 * (seed % 100000) + member).astype(np.float32)


LR = 2e-3


# --- the state buffer's fields as device tensors --------------------------------------------


def _fields(sim):
    """Views of the fields in the run's state buffer (the first checkpoint_bytes() of it):
    scalars, geometry tables, then the fields, every array on a 256-byte boundary."""
    nr, nz, nm = sim.nr, sim.nz, sim.nmat
    e = 8 if sim.precision == salec.SALEC_FP64 else 4
    T = torch.float64 if e == 8 else torch.float32
    nc, nv = nr * nz, (nr + 1) * (nz + 1)
    pb, pr = sim.grid.pml_bottom, sim.grid.pml_right
    cur = 0

    def take(n):
        nonlocal cur
        off = cur
        cur += (n + 255) // 256 * 256
        return off

    take(96)
    for n in (nr + 1, nr, nr, nr, nr, nr, nr, nz, nz):
        take(n * e)
    take(nz * 8)
    for n in (nr + 1, nr, nr, nz, nz):
        take(n * e)
    take(nz * 8)
    for n in (nz, nz + 1, nr, nr + 1):
        take(n * e)

    def view(n, w, shape, t):
        size = n * w * (8 if t == torch.float64 else 4)
        off = take(size)
        return sim.state[off:off + size].view(t).view(shape + (w,) if w > 1 else shape)

    out = {"pmax": view(nc, 1, (nz, nr), T)}
    for m in range(nm):
        fr = view(nc, 2, (nz, nr), T)
        out[f"f{m}"], out[f"rho{m}"] = fr[..., 0], fr[..., 1]
    out["I"] = view(nc, 1, (nz, nr), torch.float64)
    s01, s2d = view(nc, 2, (nz, nr), T), view(nc, 2, (nz, nr), T)
    v = view(nv, 2, (nz + 1, nr + 1), T)
    out["vr"], out["vz"] = v[..., 0], v[..., 1]
    if any(m["strength"] != "none" for m in sim.spec["materials"]):
        out.update(srr=s01[..., 0], szz=s01[..., 1], srz=s2d[..., 0], D=s2d[..., 1])
    for n in (2 * nr * pb, nr * pb, 4 * (nr + 1) * pb, 2 * pr * nz, pr * nz, 4 * pr * (nz + 1)):
        take(n * e)
    if cur != sim.checkpoint_bytes():
        raise RuntimeError("the state buffer is laid out differently")
    return out


def _typed(fields, fp64):
    """The mixed form's energies are FP64 sums of FP32 increments: returned in FP32 like its
    other fields."""
    return fields if fp64 else {k: v.float() for k, v in fields.items()}


# --- prepare and run -------------------------------------------------------------------------


def _restart(spec, precision, warm):
    """A run set up and, with `warm`, given the fields of the same impact `warm` steps on (as
    a program that resumes from saved fields does).  The saved fields are those of the plain
    FP64 cycle below."""
    sim = salec.Sim(spec, precision=precision)
    if warm:
        ref = _Cycle(spec)
        for _ in range(warm):
            ref.step()
        for name, x in dict(ref.fields(), **ref.strips()).items():
            sim.set(name, x.cpu().numpy())
        sim.set_time(ref.t, ref.dt_prev)
    return sim


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "step":
        sim = _restart(_spec(case, seed), case["precision"], case["warm"])
        s.update(sim=sim, image=sim.state[:sim.checkpoint_bytes()].clone(), fields=_fields(sim))
    elif case["kind"] == "batch":
        sims = [_restart(W.batched_run(d, d["n"]), case["precision"], case["warm"]) for d in _draws(case, seed)]
        for sim in sims:
            sim.set_end_time(20.0)
        s.update(sims=sims, batch=salec.Batch(sims), images=[x.state[:x.checkpoint_bytes()].clone() for x in sims],
                 fields=[_fields(x) for x in sims])
    else:
        x, t = _net_inputs(case, seed)
        members, n = case.get("members", 1), case["batch"]
        group = case.get("group", 1)
        streams = [torch.cuda.current_stream() if members // group <= 1 or case["kind"] != "train" else torch.cuda.Stream()
                   for _ in range(0, members, group)]
        nets = [surrogate.MLP(max(n, 128), stream=streams[k // group]) for k in range(members)]
        theta = [_theta(seed, k) for k in range(members)]
        for net, th in zip(nets, theta):
            net.set_params(th)
        s.update(x=x, t=t, nets=nets, theta=theta)
        if case["kind"] == "train":
            s["lr"] = torch.from_numpy(surrogate.cosine_lr(case["steps"], LR)).cuda()
            s["groups"] = [surrogate.Group(nets[k:k + group], stream=streams[k // group])
                           for k in range(0, members, group)] if group > 1 else None
        torch.cuda.current_stream().synchronize()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        sim, image = s["sim"], s["image"]
        sim.state[:image.numel()].copy_(image)
        sim.state_changed()
        sim.step(case["steps"])
        sums = sim.conservation()              # the run's log: it also ends the pass
        fp64 = case["precision"] == "fp64"
        return dict(_typed(s["fields"], fp64), sums=torch.tensor(list(sums.values()), dtype=torch.float64 if fp64 else torch.float32))
    if kind == "batch":
        batch = s["batch"]
        for sim, image in zip(s["sims"], s["images"]):
            sim.state[:image.numel()].copy_(image)
            sim.state_changed()
        batch.stream.wait_stream(torch.cuda.current_stream())
        batch.run(chunk=case["steps"], max_steps=case["steps"])
        fs = s["fields"]
        return _typed({k: torch.cat([f[k].reshape(-1) for f in fs]) for k in fs[0]}, case["precision"] == "fp64")
    if kind == "infer":
        return [net.forward(s["x"]) for net in s["nets"]]
    if kind == "gradient":
        loss, grad = s["nets"][0].gradient(s["x"], s["t"])
        return {"loss": np.float32(loss), "grad": grad}
    for net, th in zip(s["nets"], s["theta"]):     # training starts from the initial parameters
        net.set_params(th)
    if s["groups"]:
        for g in s["groups"]:
            g.train(s["x"], s["t"], s["lr"])
    else:
        for net in s["nets"]:
            net.train(s["x"], s["t"], s["lr"])
    return [net.get_params() for net in s["nets"]]


# --- work ------------------------------------------------------------------------------------

_PARAMS = 215874                       # of the network; its weights alone: 214784
_WEIGHTS = 214784


def _run_work(nr, nz, nm, strength, gravity, fp64, radius, warm, steps):
    """Bytes: a pass reads the fields once and writes them once.  Operations: those of the
    cycle in its plainest form (counted from its formulas: about 380 per cell and step with
    one hydrodynamic material, 90 more per further material, 200 more with strength) on the
    cells that signals can have reached (all of them under gravity)."""
    e = 8 if fp64 else 4
    cells = nr * nz
    state = cells * (2 * e * nm + 8 + e + (4 * e if strength else 0)) + (nr + 1) * (nz + 1) * 2 * e
    per = 380 + 90 * (nm - 1) + (200 if strength else 0)
    reach = 2 * radius + 0.4 * (warm + 0.5 * steps)
    active = cells if gravity else min(cells, 0.5 * math.pi * reach * reach)
    return 2.0 * state, float(per * active * steps)


def work(case):
    kind = case["kind"]
    if kind == "step":
        ph = case["physics"]
        nm = {"plain": 1, "full": 2, "layered": 3}[ph]
        b, f = _run_work(case["nr"], case["nz"], nm, ph != "plain", ph != "plain", case["precision"] == "fp64",
                         case["radius"], case["warm"], case["steps"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        n = (case["lo"] + case["hi"]) // 2
        side2 = n * n + (case["hi"] - case["lo"]) ** 2 / 12.0
        b, f = _run_work(n, n, 2, True, True, case["precision"] == "fp64", 20, case["warm"], case["steps"])
        return {"bytes": b * case["runs"] * side2 / (n * n), "flops": f * case["runs"] * side2 / (n * n)}
    B, m = case["batch"], case.get("members", 1)
    if kind == "infer":
        return {"bytes": float(B * 20 + m * (B * 264 + 4 * _PARAMS)), "flops": 2.0 * m * B * _WEIGHTS}
    passes = case.get("steps", 1)
    return {"bytes": float(B * (20 + 264) + m * 8 * _PARAMS), "flops": 6.0 * m * passes * B * _WEIGHTS}


# --- the same results in 64 bits ----------------------------------------------------------------


def exact(case, seed):
    if case["kind"] == "step":
        ref = _Cycle(_spec(case, seed))
        for _ in range(case["warm"] + case["steps"]):
            ref.step()
        return dict(ref.fields(), sums=ref.sums())
    if case["kind"] == "batch":
        runs = []
        for d in _draws(case, seed):
            ref = _Cycle(W.batched_run(d, d["n"]))
            for _ in range(case["warm"] + case["steps"]):
                ref.step()
            runs.append(ref.fields())
        return {k: torch.cat([r[k].reshape(-1) for r in runs]) for k in runs[0]}
    x, t = _net_inputs(case, seed)
    x, t = x.double(), t.double()
    members = case.get("members", 1)
    thetas = [torch.from_numpy(_theta(seed, k)).cuda().double() for k in range(members)]
    if case["kind"] == "infer":
        return [_net(th, x) for th in thetas]
    if case["kind"] == "gradient":
        loss, grad = _loss_grad(thetas[0], x, t)
        return {"loss": float(loss), "grad": grad}
    lrs = surrogate.cosine_lr(case["steps"], LR)
    out = []
    for th in thetas:
        m, v = torch.zeros_like(th), torch.zeros_like(th)
        for k, lr in enumerate(lrs):
            _, g = _loss_grad(th, x, t)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            th = th - float(lr) * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        out.append(th)
    return out


def _net(theta, x):
    h, off = x, 0
    for l in range(5):
        ni, no = surrogate.DIMS[l], surrogate.DIMS[l + 1]
        w, b = theta[off:off + ni * no].view(no, ni), theta[off + ni * no:off + ni * no + no]
        off += ni * no + no
        h = h @ w.T + b
        if l < 4:
            h = torch.nn.functional.gelu(h)
    return h


def _loss_grad(theta, x, t):
    th = theta.detach().requires_grad_(True)
    loss = ((_net(th, x) - t) ** 2).mean()
    (g,) = torch.autograd.grad(loss, th)
    return loss.detach(), g


def _sdiv(a, b, where):
    """a / b where `where` holds, else 0."""
    return torch.where(where, a / torch.where(where, b, torch.ones_like(b)), torch.zeros_like(a))


def _eos(m, rho_in, I):
    """Tillotson pressure and squared sound speed."""
    I = I.clamp_min(0.0)
    rho_f = 1e-12 * m["rho0"]
    rho = rho_in.clamp_min(rho_f)
    rho0, A, B, a, b = m["rho0"], m["A"], m["B"], m["a"], m["b"]
    mu = rho / rho0 - 1.0
    ie = rho0 * rho0 / m["E0"] / (rho * rho)
    w0 = I * ie + 1.0
    bw = b / w0
    dw = bw / w0 * I * ie
    pc = (a + bw) * rho * I + mu * (A + B * mu)
    pc_r = (a + bw) * I + 2 * dw * I + (A + 2 * B * mu) / rho0
    cc = pc_r + pc / (rho * rho) * rho * (a + bw - dw)
    x = rho0 / rho - 1.0
    x_r = -rho0 / (rho * rho)
    ea, eb = torch.exp(-m["alpha"] * x * x), torch.exp(-m["beta"] * x)
    ta = A * mu * eb
    ta_r = A / rho0 * eb - m["beta"] * x_r * ta
    tsum = bw * rho * I + ta
    pe = a * rho * I + tsum * ea
    pe_r = a * I + (bw * I + 2 * dw * I + ta_r) * ea - 2 * m["alpha"] * x * x_r * tsum * ea
    ce = pe_r + pe / (rho * rho) * rho * (a + (bw - dw) * ea)
    we = ((I - m["Eiv"]) / (m["Ecv"] - m["Eiv"])).clamp(0.0, 1.0)
    we = torch.where((rho >= rho0) | (I <= m["Eiv"]), torch.zeros_like(we), we)
    p, c2 = we * pe + (1 - we) * pc, we * ce + (1 - we) * cc
    p = torch.where(rho_in < rho_f, p * rho_in.clamp_min(0.0) / rho_f, p)
    return p, c2.clamp_min(0.01 * A / rho0)


def _expansion(m, rho):
    return (2 * rho / m["rho0"] - 1).clamp(0.0, 1.0)


class _Cycle:
    """The explicit cycle (Lagrangian step, absorbing strips, donor-cell remap, Courant
    step) on whole FP64 arrays of torch, cells [j, i] and vertices [j, i]."""

    def __init__(self, spec):
        g, self.mats = spec["grid"], spec["materials"]
        self.g = g
        nr, nz, nm = g["nr"], g["nz"], len(self.mats)
        self.nr, self.nz, self.nm = nr, nz, nm
        dev = dict(dtype=torch.float64, device="cuda")
        dr = torch.tensor(g.get("dr") or [g["dx"]] * nr, **dev)
        dz = torch.tensor(g.get("dz") or [g["dx"]] * nz, **dev)
        zero = torch.zeros(1, **dev)
        rR, zv = torch.cat([zero, dr.cumsum(0)]), torch.cat([zero, dz.cumsum(0)])
        rc = 0.5 * (rR[1:] + rR[:-1])
        self.dr, self.dz, self.rR, self.rc, self.zv = dr, dz[:, None], rR, rc, zv
        self.AZ = rc * dr
        self.V = self.AZ * self.dz
        self.AR = rR * self.dz                                # radial faces of each row
        self.L = torch.minimum(dr[None, :], self.dz)
        self.strength = any(m["strength"] != "none" for m in self.mats)
        Z = lambda *s: torch.zeros(*s, **dev)                 # noqa: E731
        self.f = [Z(nz, nr) for _ in range(nm)]
        self.rho = [Z(nz, nr) for _ in range(nm)]
        self.I, self.pmax, self.D = Z(nz, nr), Z(nz, nr), Z(nz, nr)
        self.s = [Z(nz, nr) for _ in range(3)]
        zvl = [float(z) for z in W.positions(g.get("dz") or [g["dx"]] * nz)]
        up = None                                             # pressure and weight of the row above
        for lay in spec["layers"]:
            m = self.mats[lay["mat"]]
            rows = [j for j in range(nz) if lay["zlo"] <= zvl[j] and lay["zhi"] >= zvl[j + 1]]
            for j in reversed(rows):
                rho = m["rho0"]
                if g["gravity"] > 0:                          # discrete hydrostatic balance
                    k = 0.5 * float(dz[j]) * g["gravity"]
                    rhs = 0.0 if up is None else up[0] + up[1]
                    lin, cst = m["A"] - k * m["rho0"], k * m["rho0"] + rhs
                    mu = 2 * cst / (lin + math.sqrt(lin * lin + 4 * m["B"] * cst))
                    rho = m["rho0"] * (1 + mu)
                    up = (m["A"] * mu + m["B"] * mu * mu, k * rho)
                self.f[lay["mat"]][j], self.rho[lay["mat"]][j] = 1.0, rho
        pj = spec["projectile"]                               # tangent to the surface: fills void cells only
        sub = (torch.arange(16, **dev) + 0.5) / 16
        ni = min(nr, int((rR <= pj["radius"]).sum()))
        j0, j1 = int((zv[1:] < pj["zc"] - pj["radius"]).sum()), int((zv[:-1] <= pj["zc"] + pj["radius"]).sum())
        rs = rR[:ni, None] + dr[:ni, None] * sub
        zs = zv[j0:j1, None] + dz[j0:j1, None] * sub - pj["zc"]
        inside = (rs * rs)[None, :, None, :] + (zs * zs)[:, None, :, None] < pj["radius"] ** 2
        frac = (inside * rs[None, :, None, :]).sum((2, 3)) / (16 * rs.sum(1))
        frac = torch.where(frac < g["f_min"], torch.zeros_like(frac), frac)
        k = pj["mat"]
        here = frac > 0
        self.f[k][j0:j1, :ni] = torch.where(here, frac, self.f[k][j0:j1, :ni])
        self.rho[k][j0:j1, :ni] = torch.where(here, torch.full_like(frac, self.mats[k]["rho0"]), self.rho[k][j0:j1, :ni])
        moving = torch.zeros_like(self.V)
        moving[j0:j1, :ni] = here.double()
        M = self.V * sum(f * r for f, r in zip(self.f, self.rho))
        mass, mom = self._corner(M), self._corner(M * moving)
        self.vr, self.vz = Z(nz + 1, nr + 1), _sdiv(mom, mass, mass > 0) * pj["vz"]
        self.vz[0] = 0.0
        # strips: reference rows of the outermost column, profiles, relaxation
        pr, pb = g["pml_r"], g["pml_b"]
        self.pr, self.pb = pr, pb
        c = g["pml_c"] or max(math.sqrt(m["A"] / m["rho0"]) for m in self.mats)
        phat, phi, mass = Z(nz), Z(nz), Z(nz)
        for m, f, r in zip(self.mats, self.f, self.rho):
            p, _ = _eos(m, r[:, -1], self.I[:, -1])
            p = torch.maximum(p, m["p_t"] * _expansion(m, r[:, -1]))
            phat, phi, mass = phat + f[:, -1] * torch.where(f[:, -1] > 0, p, 0 * p), phi + f[:, -1], mass + f[:, -1] * r[:, -1]
        self.p0 = _sdiv(phat, phi, phi > 0)[:, None]
        self.rho_ref = _sdiv(mass, phi, phi > 0)[:, None]
        lg = math.log(1.0 / g["pml_R"])
        prof = lambda y, d: 1.5 * c / d * (y.clamp_min(0.0) / d) ** 2 * lg   # noqa: E731
        if pb:
            d = float(zv[pb])
            self.dBc, self.dBv = prof(d - (zv[:pb] + 0.5 * dz[:pb]), d)[:, None], prof(d - zv[:pb], d)[:, None]
            self.ab = g["pml_alpha"] * c / d
        if pr:
            d, r_in = float(rR[nr] - rR[nr - pr]), rR[nr - pr]
            rows = (self.rho_ref > 0).double()
            vrows = torch.maximum(torch.cat([rows, 0 * rows[:1]]), torch.cat([0 * rows[:1], rows]))
            self.dRc, self.dRv = prof(rc[nr - pr:] - r_in, d) * rows, prof(rR[nr - pr + 1:] - r_in, d) * vrows
            self.ar = g["pml_alpha"] * c / d
        self.B = dict(phi1=Z(pb, nr), phi3=Z(pb, nr), psi2=Z(pb, nr), v=[Z(pb, nr + 1) for _ in range(4)])
        self.R = dict(phi1=Z(nz, pr), phi3=Z(nz, pr), psi2=Z(nz, pr), v=[Z(nz + 1, pr) for _ in range(4)])
        self.t, self.dt_prev = 0.0, g["dt_init"]

    @staticmethod
    def _around(x):
        """The four cells around each vertex: (i-1,j-1), (i,j-1), (i,j), (i-1,j); 0 outside."""
        p = torch.nn.functional.pad(x, (1, 1, 1, 1))
        return p[:-1, :-1], p[:-1, 1:], p[1:, 1:], p[1:, :-1]

    def _corner(self, x):
        return 0.25 * sum(self._around(x))

    def _bc(self, vr, vz):
        vr[:, 0] = 0.0
        vr[:, -1] = 0.0
        vz[0] = 0.0
        if self.g["bc_bottom"] == "noslip":
            vr[0] = 0.0
        if self.g["bc_top"] == "wall":
            vz[-1] = 0.0

    def step(self):
        g, nr, nz, pr, pb = self.g, self.nr, self.nz, self.pr, self.pb
        V, AZ, AR, dz, dr = self.V, self.AZ, self.AR, self.dz, self.dr
        zero = torch.zeros_like(V)
        # phase 0: pressure, viscosity, Courant step
        phat, phi, rhob, c2 = zero, zero, zero, zero
        for m, f, r in zip(self.mats, self.f, self.rho):
            here = f > 0
            p, c2m = _eos(m, r, self.I)
            p = torch.maximum(p, (1 - self.D) * m["p_t"] * _expansion(m, r))
            phat, phi, rhob = phat + torch.where(here, f * p, zero), phi + f, rhob + f * r
            c2 = torch.maximum(c2, torch.where(here, c2m, zero))
        matter = phi > 0
        cs = c2.sqrt()

        def faces(vr, vz):
            return (0.5 * (vr[1:, :-1] + vr[:-1, :-1]), 0.5 * (vr[1:, 1:] + vr[:-1, 1:]),
                    0.5 * (vz[:-1, :-1] + vz[:-1, 1:]), 0.5 * (vz[1:, :-1] + vz[1:, 1:]))

        def fluxes(vr, vz):
            uL, uR, uB, uT = faces(vr, vz)
            return AR[:, 1:] * uR - AR[:, :-1] * uL, AZ * (uT - uB)

        a, b = fluxes(self.vr, self.vz)
        div = ((a + b) / V).clamp_max(0.0)
        pbar, rb = _sdiv(phat, phi, matter), _sdiv(rhob, phi, matter)
        q = rb * (g["av_cq"] * (self.L * div) ** 2 - g["av_cl"] * self.L * cs * div)
        P = torch.where(matter, phat + phi * q, zero)
        M = rhob * V
        self.pmax = torch.where(matter, torch.maximum(self.pmax, pbar - self.p0), self.pmax)
        w = self.vr ** 2 + self.vz ** 2
        w = torch.maximum(torch.maximum(w[:-1, :-1], w[:-1, 1:]), torch.maximum(w[1:, :-1], w[1:, 1:]))
        rate = torch.where(matter, (w.sqrt() + cs) / self.L, zero).max()
        dt = min(g["dt_growth"] * self.dt_prev, g["cfl"] / float(rate), g["dt_max"])
        # phase 1: corner forces, strips, Lagrangian velocity
        P0, P1, P2, P3 = self._around(P)
        pad = torch.nn.functional.pad
        ARb, ARt = pad(AR, (0, 0, 1, 0)), pad(AR, (0, 0, 0, 1))
        AZl, AZr = pad(AZ, (1, 0)), pad(AZ, (0, 1))
        rad = lambda x0, x1, x2, x3: 0.5 * (ARb * (x0 - x1) + ARt * (x3 - x2))     # noqa: E731
        ver = lambda x0, x1, x2, x3: 0.5 * (AZl * (x0 - x3) + AZr * (x1 - x2))     # noqa: E731
        rr, rz, vr_, vz_ = 0.0, 0.0, 0.0, 0.0
        if self.strength:
            Srr, Szz, Srz = (phi * x for x in self.s)
            hr, hz, hoop = 0.5 * self.rc * dz, 0.5 * AZ, 0.25 * dr * dz
            left = lambda x: (lambda k: k[1] + k[2] - k[0] - k[3])(self._around(x))      # noqa: E731
            low = lambda x: (lambda k: k[2] + k[3] - k[0] - k[1])(self._around(x))       # noqa: E731
            rr = left(hr * Srr) + sum(self._around(hoop * (Srr + Szz)))
            rz, vr_, vz_ = left(hr * Srz), low(hz * Srz), low(hz * Szz)
        Fr, Fz = rad(P0, P1, P2, P3) + (rr + vr_), ver(P0, P1, P2, P3) + (rz + vz_)
        if pb or pr:
            Q = self._around(P - phi * self.p0)
        if pb:
            z, w4 = self.B["v"][2], self.B["v"][3]
            Tr = (rad(*Q) + rr)[:pb]
            Tz = rz[:pb] if self.strength else 0.0
            z, w4 = z * (1 - self.ab * dt) - dt * self.dBv * Tr, w4 * (1 - self.ab * dt) - dt * self.dBv * Tz
            self.B["v"][2:] = [z, w4]
            Fr[:pb] -= z
            Fz[:pb] -= w4
        if pr:
            z, w4 = self.R["v"][2], self.R["v"][3]
            Tz = (ver(*Q) + vz_)[:, nr - pr + 1:]
            Tr = vr_[:, nr - pr + 1:] if self.strength else 0.0
            z, w4 = z * (1 - self.ar * dt) - dt * self.dRv * Tr, w4 * (1 - self.ar * dt) - dt * self.dRv * Tz
            self.R["v"][2:] = [z, w4]
            Fr[:, nr - pr + 1:] -= z
            Fz[:, nr - pr + 1:] -= w4
        mass = self._corner(M)
        some = mass > 0
        vr = torch.where(some, self.vr + dt * _sdiv(Fr, mass, some), torch.zeros_like(mass))
        vz = torch.where(some, self.vz + dt * (_sdiv(Fz, mass, some) - g["gravity"]), torch.zeros_like(mass))
        self._bc(vr, vz)
        dK = 0.5 * mass * ((vr - self.vr) ** 2 + (vz - self.vz) ** 2)
        # phase 2: Lagrangian cells
        uL, uR, uB, uT = faces(vr, vz)
        err, ezz, ett = (uR - uL) / dr, (uT - uB) / dz, (uR + uL) / (2 * self.rc)
        a, b = fluxes(vr, vz)
        dV = dt * (a + b)
        VL = torch.where(matter, V + dV, V)
        Pr, Pv, strain = -P * a, -P * b, zero
        if self.strength:
            vr_z = 0.5 * ((vr[1:, :-1] + vr[1:, 1:]) - (vr[:-1, :-1] + vr[:-1, 1:])) / dz
            vz_r = 0.5 * ((vz[:-1, 1:] + vz[1:, 1:]) - (vz[:-1, :-1] + vz[1:, :-1])) / dr
            erz = 0.5 * (vr_z + vz_r)
            Stt = -(Srr + Szz)
            strain = dt * V * (Srr * err + Szz * ezz + Stt * ett + 2 * Srz * erz)
            Pr = Pr + V * (Srr * err + Stt * ett + Srz * vz_r)
            Pv = Pv + V * (Szz * ezz + Srz * vr_z)
        dE = -P * dV + strain
        if pb:
            a2 = self.B["psi2"] * (1 - self.ab * dt) - dt * self.dBc * Pr[:pb]
            self.B["psi2"] = torch.where(matter[:pb], a2, self.B["psi2"])
            dE[:pb] -= dt * self.B["psi2"]
        if pr:
            a2 = self.R["psi2"] * (1 - self.ar * dt) - dt * self.dRc * Pv[:, nr - pr:]
            self.R["psi2"] = torch.where(matter[:, nr - pr:], a2, self.R["psi2"])
            dE[:, nr - pr:] -= dt * self.R["psi2"]
        IL = torch.where(matter, self.I + _sdiv(dE, M, M > 0), zero)
        fL, rL = [], []
        for f, r in zip(self.f, self.rho):
            here = f > 0
            Vm = f * V
            VmL = Vm + _sdiv(f, phi, matter) * phi * dV
            fL.append(torch.where(here, VmL / VL, zero))
            rL.append(r * _sdiv(Vm, VmL, here))
        sL, DL = self.s, self.D
        if self.strength:
            G, Y, ie = zero, zero, zero
            for m, f, r in zip(self.mats, self.f, self.rho):
                if m["strength"] == "none":
                    continue
                pp = pbar.clamp_min(0.0)
                Yi = m["Yi0"] + m["mui"] * pp / (1 + m["mui"] * pp / (m["Yim"] - m["Yi0"]))
                y = (1 - DL) * Yi + DL * (m["Yd0"] + m["mud"] * pp).clamp_max(m["Ydm"])
                hot = self.I > 0
                soft = torch.tanh(1.2 * (_sdiv(torch.full_like(zero, m["Eiv"]), self.I, hot) - 1))
                y = torch.where(hot, y * soft, y) * _expansion(m, r)
                y = torch.where(hot & (self.I >= m["Eiv"]), zero, y).clamp_min(0.0)
                G, Y = G + f * m["G"], Y + f * y
                ie = ie + f / (m["B_dam"] * (pbar - m["p_bd"])).clamp_min(m["eps_fb"])
            G, Y, ie = (_sdiv(x, phi, matter) for x in (G, Y, ie))
            om, tr3 = 0.5 * (vr_z - vz_r), (err + ezz + ett) / 3
            srr, szz, srz = self.s
            n = [srr + dt * (2 * G * (err - tr3) + 2 * om * srz), szz + dt * (2 * G * (ezz - tr3) - 2 * om * srz),
                 srz + dt * (2 * G * erz + om * (szz - srr))]
            J2 = 0.5 * (n[0] ** 2 + n[1] ** 2 + (n[0] + n[1]) ** 2) + n[2] ** 2
            sq = J2.sqrt()
            flow = (J2 > Y * Y) & (G > 0)
            k = torch.where(flow, _sdiv(Y, sq, flow), torch.ones_like(sq))
            DL = torch.where(flow, (DL + _sdiv(sq - Y, math.sqrt(3.0) * G, flow) * ie).clamp_max(1.0), DL)
            sL = [torch.where(G > 0, x * k, zero) for x in n]
            DL = torch.where(matter, DL, zero)
        # phase 3a: donor-cell remap of the cells
        dVR = torch.zeros(nz, nr + 1, dtype=V.dtype, device=V.device)
        dVR[:, 1:-1] = dt * AR[:, 1:-1] * 0.5 * (vr[:-1, 1:-1] + vr[1:, 1:-1])
        dVZ = dt * AZ * 0.5 * (vz[:, :-1] + vz[:, 1:])
        dVZ[0] = 0.0
        fromL, fromB = dVR > 0, dVZ > 0
        inn = lambda x: torch.where(fromL, pad(x, (1, 0)), pad(x, (0, 1)))          # noqa: E731
        inz = lambda x: torch.where(fromB, pad(x, (0, 0, 1, 0)), pad(x, (0, 0, 0, 1)))  # noqa: E731
        net = lambda fr, fz: fr[:, :-1] - fr[:, 1:] + fz[:-1] - fz[1:]              # noqa: E731
        vm = [(dVR * inn(f), dVZ * inz(f)) for f in fL]
        mm = [(v[0] * inn(r), v[1] * inz(r)) for v, r in zip(vm, rL)]
        vR, vZ = sum(v[0] for v in vm), sum(v[1] for v in vm)
        mR, mZ = sum(m[0] for m in mm), sum(m[1] for m in mm)
        iR, iZ = inn(IL), inz(IL)
        gain = ((iR[:, :-1] - IL) * mR[:, :-1].clamp_min(0) - (iR[:, 1:] - IL) * mR[:, 1:].clamp_max(0) +
                (iZ[:-1] - IL) * mZ[:-1].clamp_min(0) - (iZ[1:] - IL) * mZ[1:].clamp_max(0))
        Mtot, keepV, keepM, fn, rn = zero, zero, zero, [], []
        for f, r, v, m in zip(fL, rL, vm, mm):
            av, am = net(*v), net(*m)
            Vm, Mm = f * VL + av, r * f * VL + am
            Mtot = Mtot + Mm
            rho = torch.where(Vm > 0, r + _sdiv(am - r * av, Vm, Vm > 0), zero)
            keep = (Vm / V >= g["f_min"]) & (Vm > 0)
            fn.append(torch.where(keep, Vm / V, zero))
            rn.append(torch.where(keep, rho, zero))
            keepV, keepM = keepV + torch.where(keep, Vm, zero), keepM + torch.where(keep, Mm, zero)
        I = torch.where(Mtot > 0, IL + _sdiv(gain, Mtot, Mtot > 0), zero)
        full = keepM > 0
        if self.strength:
            aV = net(vR, vZ)
            Vt = sum(f for f in fL) * VL + aV
            new = [x + _sdiv(net(vR * inn(x), vZ * inz(x)) - x * aV, Vt, Vt > 0) for x in (*sL, DL)]
            new = [torch.where(full & (Vt > 0), x, zero) for x in new]
            self.s, self.D = new[:3], new[3]
        I = torch.where(full, I, zero)
        dsum, p1, p3 = torch.zeros_like(V), torch.zeros_like(V), torch.zeros_like(V)
        if pb:
            out, oute = (mR[:, 1:] - mR[:, :-1])[:pb], ((mR * iR)[:, 1:] - (mR * iR)[:, :-1])[:pb]
            self.B["phi1"] = self.B["phi1"] * (1 - self.ab * dt) + self.dBc * out
            self.B["phi3"] = self.B["phi3"] * (1 - self.ab * dt) + self.dBc * oute
            dsum[:pb] += self.dBc
            p1[:pb] += self.B["phi1"]
            p3[:pb] += self.B["phi3"]
        if pr:
            c = slice(nr - pr, nr)
            out, oute = (mZ[1:] - mZ[:-1])[:, c], ((mZ * iZ)[1:] - (mZ * iZ)[:-1])[:, c]
            self.R["phi1"] = self.R["phi1"] * (1 - self.ar * dt) + self.dRc * out
            self.R["phi3"] = self.R["phi3"] * (1 - self.ar * dt) + self.dRc * oute
            dsum[:, c] += self.dRc
            p1[:, c] += self.R["phi1"]
            p3[:, c] += self.R["phi3"]
        damp = full & (dsum > 0)
        dM = torch.where(damp, -dt * (dsum * (keepM - keepV * self.rho_ref) + p1), zero)
        dEp = -dt * (dsum * keepM * I + p3)                    # the reference rows are cold
        I = torch.where(damp, I + _sdiv(dEp - I * dM, keepM + dM, damp), I)
        kappa = 1 + _sdiv(dM, keepM, damp)
        self.f, self.rho = fn, [kappa * r for r in rn]
        # phase 3b: momentum on the dual grid
        pR, pZ = pad(mR, (0, 0, 1, 1)), pad(mZ, (1, 1, 0, 0))
        col, row = pR[:-1] + pR[1:], pZ[:, :-1] + pZ[:, 1:]
        dR = 0.25 * (col[:, :-1] + col[:, 1:])                 # (i,j) -> (i+1,j)
        dZ = 0.25 * (row[:-1] + row[1:])                       # (i,j) -> (i,j+1)
        top = 0.5 * row[-1:]
        wr = [torch.where(dR > 0, x[:, :-1], x[:, 1:]) for x in (vr, vz)]
        wz = [torch.where(dZ > 0, x[:-1], x[1:]) for x in (vr, vz)]

        def dual(xr, xz, xt):
            """(in - out) through the side faces, and through the lower and upper ones"""
            h, t = pad(xr, (1, 1)), torch.cat([0 * xt, xz, xt])
            return h[:, :-1] - h[:, 1:], t[:-1] - t[1:]

        mh, mt = dual(dR, dZ, top)
        rh, rt = dual(dR * wr[0], dZ * wz[0], top * vr[-1:])
        zh, zt = dual(dR * wr[1], dZ * wz[1], top * vz[-1:])
        eh, et = dual(0.5 * dR * (wr[0] ** 2 + wr[1] ** 2), 0.5 * dZ * (wz[0] ** 2 + wz[1] ** 2),
                      0.5 * top * (vr[-1:] ** 2 + vz[-1:] ** 2))
        m = mass + mh + mt
        qr, qz = mass * vr + rh + rt, mass * vz + zh + zt
        kin = 0.5 * mass * (vr ** 2 + vz ** 2) + eh + et
        some = m > 0
        heat = _sdiv(dK + kin - 0.5 * _sdiv(qr * qr + qz * qz, m, some), m, some)
        damp_v = torch.zeros_like(m)
        ar, az = torch.zeros_like(m), torch.zeros_like(m)
        if pb:
            x = self.B["v"]
            x[0] = x[0] * (1 - self.ab * dt) - self.dBv * rh[:pb]
            x[1] = x[1] * (1 - self.ab * dt) - self.dBv * zh[:pb]
            damp_v[:pb] += self.dBv
            ar[:pb] += x[0]
            az[:pb] += x[1]
        if pr:
            x, c = self.R["v"], slice(nr - pr + 1, nr + 1)
            x[0] = x[0] * (1 - self.ar * dt) - self.dRv * rt[:, c]
            x[1] = x[1] * (1 - self.ar * dt) - self.dRv * zt[:, c]
            damp_v[:, c] += self.dRv
            ar[:, c] += x[0]
            az[:, c] += x[1]
        qr, qz = qr - dt * (damp_v * qr + ar), qz - dt * (damp_v * qz + az)
        near = some & (sum(self._around(sum(self.f))) > 0)
        self.vr, self.vz = _sdiv(qr, m, near), _sdiv(qz, m, near)
        self._bc(self.vr, self.vz)
        # phase 3c: the kinetic-energy deficit as heat
        add = 0.25 * (heat[:-1, :-1] + heat[:-1, 1:] + heat[1:, 1:] + heat[1:, :-1])
        self.I = torch.where(sum(f * r for f, r in zip(self.f, self.rho)) > 0, I + add, I)
        self.t, self.dt_prev = self.t + dt, dt

    def fields(self):
        out = {"pmax": self.pmax, "I": self.I, "vr": self.vr, "vz": self.vz}
        for k in range(self.nm):
            out[f"f{k}"], out[f"rho{k}"] = self.f[k], self.rho[k]
        if self.strength:
            out.update(srr=self.s[0], szz=self.s[1], srz=self.s[2], D=self.D)
        return out

    def strips(self):
        """The absorbing strips' auxiliaries as fields over the whole grid."""
        out = {}
        for side, d, cell, vert in (("b", self.B, (0, 0, 0, self.nz - self.pb), (0, 0, 0, self.nz + 1 - self.pb)),
                                    ("r", self.R, (self.nr - self.pr, 0), (self.nr + 1 - self.pr, 0))):
            for k in ("phi1", "phi3", "psi2"):
                out[f"{k}_{side}"] = torch.nn.functional.pad(d[k], cell)
            for k, x in zip(("phi2r", "phi2z", "psi1r", "psi1z"), d["v"]):
                out[f"{k}_{side}"] = torch.nn.functional.pad(x, vert)
        return out

    def sums(self):
        """Mass, vertical momentum, kinetic and internal energy."""
        M = self.V * sum(f * r for f, r in zip(self.f, self.rho))
        m = self._corner(M)
        return torch.stack([M.sum(), (m * self.vz).sum(), (0.5 * m * (self.vr ** 2 + self.vz ** 2)).sum(), (M * self.I).sum()])
