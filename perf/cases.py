"""Performance cases of the simulator, each through a call a user's program makes.

A case is one of these kinds of work (`kind`):

newton    one inexact Newton iteration as an outer driver runs it: the iterate goes
          in from host memory, `newton_step` assembles, sets the preconditioner up,
          solves and updates, and the new iterate comes back to the host
solve     a program with its own Newton loop: `assemble` at the current iterate,
          then `linear_solve` (preconditioner set-up and FGMRES) on device vectors
setup     a program with its own Krylov method and a new Jacobian: `precond_setup`
          and the first application
apply     the same program inside its iteration: one CPR application
assemble  the same program between solves: `assemble`, the CNV convergence test and
          one product with the Jacobian
batch     an ensemble of uneven realisations advanced one short time step in lockstep
forward   the learned pressure stage's network, inference on one grid
grad      its training: loss and parameter gradients on one grid

Rock, states and vectors are random but smooth, as reservoir fields are: log-normal
permeability with a correlation length of some cells, saturations with fronts and
(black oil) regions with and without free gas.
"""
import math

import numpy as np
import torch

from paper_1606_00548_gb300 import synth
from paper_1606_00548_gb300.sim import Batch, Net, Simulator


def listed():
    def sim(name, kind, model, nx, ny, nz, sigma, dt, mixed=False, stages=2, cycles=1, pattern="five_spot"):
        return dict(name=name, kind=kind, model=model, nx=nx, ny=ny, nz=nz, sigma=sigma, dt=dt, mixed=mixed,
                    stages=stages, cycles=cycles, pattern=pattern)

    return [
        # the quarter five-spot of the tests and the first thing a user runs: 2,000 cells, launches and latency
        sim("newton_ow_20x20x5", "newton", 2, 20, 20, 5, 0.0, 1.0),
        # the ordinary study: black oil, 200k cells, ten-day steps
        sim("newton_bo_100x100x20", "newton", 3, 100, 100, 20, 1.0, 10.0),
        # the same kind of study in the FP32-preconditioned CPR-FPF form, on a ragged grid
        sim("newton_bo_75x61x33_mixed_fpf", "newton", 3, 75, 61, 33, 1.0, 5.0, mixed=True, stages=3),
        # a ragged two-phase model solved by a program with its own Newton loop
        sim("solve_ow_57x43x17", "solve", 2, 57, 43, 17, 1.3, 1.0),
        # the large field: n^3 with 25 wells and two V-cycles per pressure stage, 4.1M cells
        sim("solve_bo_160x160x160", "solve", 3, 160, 160, 160, 1.0, 1.0, cycles=2, pattern="pattern25"),
        # a new preconditioner per Newton iteration: its cost on the ordinary study's grid
        sim("setup_bo_100x100x20", "setup", 3, 100, 100, 20, 1.0, 10.0),
        # the application inside a Krylov loop: the million-cell n^3 field, and a ragged two-phase grid
        sim("apply_bo_100x100x100", "apply", 3, 100, 100, 100, 1.0, 1.0, cycles=2, pattern="pattern25"),
        sim("apply_ow_127x101x31", "apply", 2, 127, 101, 31, 1.3, 1.0),
        # residual, Jacobian, convergence test and product on the grid the learned stage is trained on
        sim("assemble_bo_128x128x32", "assemble", 3, 128, 128, 32, 1.0, 10.0),
        # uncertainty studies: realisations of different sizes, one short step of all of them
        dict(name="batch_ow_8", kind="batch", members=8, nx_max=128, ny_max=128, nz_max=32, dt=0.01),
        # the learned pressure stage: inference on its training grid, gradients on a ragged one
        dict(name="forward_128x128x32", kind="forward", nx=128, ny=128, nz=32),
        dict(name="grad_131x67x29", kind="grad", nx=131, ny=67, nz=29),
    ]


def _grid(rng, lo, hi):
    """nx, ny, nz with a cell count spread over the logarithm of lo..hi, mostly odd and uneven"""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nz = max(3, min(120, int(round(n ** rng.uniform(0.2, 0.34)))))
    nx = max(8, int(round(math.sqrt(n / nz) * math.exp(rng.uniform(-0.3, 0.3)))))
    return nx, max(8, int(round(n / (nz * nx)))), nz


def draw(rng):
    kind = rng.choice(("newton", "newton", "solve", "solve", "setup", "apply", "apply", "assemble", "batch", "forward", "grad"))
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(3, 10), nx_max=rng.randint(40, 128), ny_max=rng.randint(40, 128),
                    nz_max=rng.randint(10, 32), dt=0.01)
    if kind in ("forward", "grad"):
        nx, ny, nz = _grid(rng, 2e3, 1.2e6)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz)
    nx, ny, nz = _grid(rng, 2e3, 1.2e6)
    model = rng.choice((2, 3))
    mixed = kind in ("newton", "solve") and rng.random() < 0.35
    return dict(kind=kind, model=model, nx=nx, ny=ny, nz=nz, sigma=round(rng.uniform(0.5, 1.4), 2),
                dt=rng.choice((1.0, 2.0, 5.0)), mixed=mixed, stages=rng.choice((2, 2, 3)), cycles=rng.choice((1, 1, 2)),
                pattern="five_spot")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rng(seed, salt):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + salt * 7919) & 0x7FFFFFFF)


def _field(nx, ny, nz, corr, seed, salt):
    """standardised Gaussian random field [N] (x fastest) with a correlation length of `corr` cells"""
    z = torch.randn((nz, ny, nx), generator=_rng(seed, salt), device="cuda", dtype=torch.float32)
    half = int(math.ceil(1.5 * corr))
    t = torch.arange(-half, half + 1, device="cuda", dtype=torch.float32)
    w = torch.exp(-2.0 * (t / corr) ** 2)
    w = (w / w.sum()).view(1, 1, -1)
    for axis in range(3):
        z = z.movedim(axis, -1)
        shape, m = z.shape, z.shape[-1]
        idx = torch.arange(-half, m + half, device="cuda")
        idx = (idx % (2 * m)).minimum((2 * m - 1) - idx % (2 * m))          # reflective edges
        rows = z.reshape(-1, m)
        out = torch.zeros_like(rows)
        for k in range(2 * half + 1):
            out += w[0, 0, k] * rows[:, idx[k:k + m]]
        z = out.reshape(shape).movedim(-1, axis)
    z = z.reshape(-1).double()
    return (z - z.mean()) / z.std().clamp_min(1e-12)


def _sim_case(c, seed):
    """the synth case of a listed or drawn one, with rock of this seed"""
    nx, ny, nz, sigma = c["nx"], c["ny"], c["nz"], c["sigma"]
    solver = dict(cpr_stages=c["stages"], amg_cycles=c["cycles"])
    if c["model"] == 2:
        case = synth.oil_water_case(nx=nx, ny=ny, nz=nz, sigma=0.0, dt=c["dt"], **solver)
    else:
        case = synth.black_oil_case(nx=nx, ny=ny, nz=nz, sigma=0.0, corr_len=0.0, dt=c["dt"], wells=c["pattern"], **solver)
    if sigma > 0.0:
        z = _field(nx, ny, nz, 10.0, seed, 1)
        k = torch.exp(4.6 + sigma * z).cpu().numpy()
        case.update(kx=k, ky=k.copy(), kz=0.1 * k, poro=(0.15 + 0.10 * torch.special.ndtr(z)).cpu().numpy())
    return case


def _state(case, seed):
    """a state in the middle of a run: p, Sw, x3, phase (numpy)"""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    a, s, g = (_field(nx, ny, nz, 6.0, seed, k).cpu().numpy() for k in (2, 3, 4))
    p = case["init"]["p"] + 8.0 * a
    sw = 0.1 + 0.45 / (1.0 + np.exp(-3.0 * s))
    if case["model"] == 2:
        return p, sw, np.zeros(N), np.ones(N, np.int8)
    ph = (g > 0.4).astype(np.int8)
    x3 = np.where(ph == 1, 0.02 + 0.1 * np.clip(g - 0.4, 0.0, 1.0), p - 5.0 - 10.0 * np.clip(0.4 - g, 0.0, 2.0))
    return p, sw, x3, ph


def _direction(case, state, seed):
    """a vector of the size of a Newton update (bar for pressures, saturation units otherwise)"""
    b, N = case["model"], state[0].size
    v = torch.randn(b * N, generator=_rng(seed, 5), device="cuda", dtype=torch.float64)
    v[N:2 * N] *= 0.05
    if b == 3:
        v[2 * N:] *= torch.from_numpy(np.where(state[3] == 1, 0.05, 1.0)).cuda()
    return v


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad"):
        N = case["nx"] * case["ny"] * case["nz"]
        net = Net(case["nx"], case["ny"], case["nz"], seed=seed)
        x = torch.stack([_field(case["nx"], case["ny"], case["nz"], 3.0, seed, 10 + k) for k in range(4)], 1).float().contiguous()
        t = (0.5 * x[:, 0] - 0.2 * x[:, 1] * x[:, 2]).contiguous()
        torch.cuda.synchronize()
        return dict(kind=kind, net=net, x=x, t=t, y=torch.empty(N, dtype=torch.float32, device="cuda"))
    if kind == "batch":
        cases = [_sim_case(m, seed) for m in _members(case, seed)]
        sims = [Simulator(c) for c in cases]
        return dict(kind=kind, batch=Batch(sims), sims=sims, dt=case["dt"], init=[c["init"] for c in cases])
    sc = _sim_case(case, seed)
    st = _state(sc, seed)
    sim = Simulator(sc, precision=1 if case["mixed"] else 0)
    sim.set_state(*st)
    s = dict(kind=kind, sim=sim, dt=case["dt"])
    if kind == "newton":
        s["x0"] = np.concatenate(st[:case["model"]])
        s["phase0"] = st[3]
        return s
    n = sim.N * sim.b
    sim.assemble(case["dt"])
    if kind == "solve":
        s["b"] = torch.from_numpy(-sim.residual()).cuda()
    elif kind == "assemble":
        s["b"] = _direction(sc, st, seed)
    else:
        s["b"] = torch.randn(n, generator=_rng(seed, 6), device="cuda", dtype=torch.float64)
        if kind == "apply":
            sim.precond_setup()
    s["z"] = torch.empty(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def _members(case, seed):
    """the realisations of an ensemble: uneven grids and heterogeneity, as synth's ensemble has"""
    u = synth.uniform01(4 * case["members"], 7)
    out = []
    for m in range(case["members"]):
        a = u[4 * m:4 * m + 4]
        out.append(dict(model=2, nx=32 + int(a[0] * (case["nx_max"] - 31)), ny=32 + int(a[1] * (case["ny_max"] - 31)),
                        nz=8 + int(a[2] * (case["nz_max"] - 7)), sigma=0.5 + 0.5 * a[3], dt=case["dt"], stages=2, cycles=1))
    return out


def run(s):
    kind = s["kind"]
    if kind == "forward":
        s["net"].forward(s["x"], s["y"])
        return {"y": s["y"]}
    if kind == "grad":
        loss, grads = s["net"].loss_grad(s["x"], s["t"])
        return {"loss": loss, "grads": grads}
    if kind == "batch":
        for m, i in zip(s["sims"], s["init"]):
            m.set_state(i["p"], i["sw"], i["x3"], i["phase"])
        s["batch"].step(s["dt"])
        return [list(m.get_state()[:2]) for m in s["sims"]]
    sim = s["sim"]
    if kind == "newton":
        sim.set_iterate(s["x0"], s["phase0"])
        sim.newton_step(s["dt"])
        x, ph = sim.get_iterate()
        return {"x": x, "phase": ph}
    if kind == "solve":
        sim.assemble(s["dt"])
        sim.linear_solve(s["b"], s["z"])
        return {"x": s["z"]}
    if kind == "setup":
        sim.precond_setup()
        sim.precond_apply(s["b"], s["z"])
        return {"z": s["z"]}
    if kind == "apply":
        sim.precond_apply(s["b"], s["z"])
        return {"z": s["z"]}
    sim.assemble(s["dt"])
    cnv = sim.cnv(s["dt"])
    sim.spmv(s["b"], s["z"])
    return {"cnv": cnv, "y": s["z"]}


def work(case):
    """bytes and operations one pass cannot do without (solves: at 25 iterations; a time step
    of the ensemble: five Newton iterations)"""
    kind = case["kind"]
    if kind in ("forward", "grad"):
        n = case["nx"] * case["ny"] * case["nz"]
        mac = 27 * (4 * 16 + 16 * 16 + 16 * 16 + 16) * n
        return dict(bytes=n * (16 + 4) if kind == "forward" else n * (16 + 4 + 3 * 32), flops=2 * mac * (1 if kind == "forward" else 3))
    if kind == "batch":
        parts = [_sim_work(dict(m, mixed=False, kind="newton"), 25) for m in _members(case, 0)]
        return {k: 5 * sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return _sim_work(case, 25)


def _sim_work(c, its):
    n, b, t = c["nx"] * c["ny"] * c["nz"], c["model"], 4 if c["mixed"] else 8
    spmv = (n * (7 * b * b + 2 * b) * 8, n * 14 * b * b)
    assemble = (n * (7 * b * b + 4 * b + 4) * 8, n * 100 * b)
    # set-up: the Jacobian in, the decoupled matrix, A_p and the diagonal inverses out
    setup = (n * (7 * b * b * (8 + t) + 7 * 8 + b * b * t), n * 30 * b * b)
    # one application: vectors, pressure block twice per cycle, the decoupled matrix once, the inverses
    apply = (n * (2 * b * 8 + c["cycles"] * 2 * 7 * t + (c["stages"] - 1) * (7 * b * b + b * b) * t),
             n * (c["cycles"] * 40 + (c["stages"] - 1) * 16 * b * b))
    orth = (n * b * 8 * (its / 2 + 2), n * b * 2 * its)
    parts = {"apply": [apply], "setup": [setup, apply], "assemble": [assemble, spmv]}.get(
        c["kind"], [assemble, setup] + [spmv, apply, orth] * its)
    return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))


# ---------------------------------------------------------------------------
# values in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "grad"):
        return _exact_net(case, seed)
    n = case.get("model", 0) * case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    if kind in ("batch", "setup", "apply") or (kind in ("newton", "solve") and n > 9000):
        # whole time steps and larger solves take minutes in plain torch, without a preconditioner; an
        # application of the preconditioner is what its hierarchy makes it, and has no value apart from it
        return None
    sc = _sim_case(case, seed)
    st = _state(sc, seed)
    if kind == "assemble":
        model = _Model(sc, st)
        v = _direction(sc, st, seed)
        R, y = torch.func.jvp(lambda x: model.residual(x, case["dt"]), (model.x0,), (v,))
        return {"cnv": float(model.cnv(R, case["dt"])), "y": y}
    model = _Model(sc, st)
    R = model.residual(model.x0, case["dt"])
    dx = torch.linalg.solve(model.jacobian(case["dt"]), -R)
    if kind == "solve":
        return {"x": dx}
    x, ph = model.update(dx)
    return {"x": x, "phase": ph}


def _exact_net(case, seed):
    s = prepare(case, seed)
    shape = (case["nz"], case["ny"], case["nx"])
    p = torch.from_numpy(s["net"].get_params()).cuda().double().requires_grad_(True)
    h, off = s["x"].double().t().reshape(1, 4, *shape), 0
    for l, (ci, co) in enumerate(((4, 16), (16, 16), (16, 16), (16, 1))):
        w = p[off:off + 27 * ci * co].view(3, 3, 3, ci, co).permute(4, 3, 0, 1, 2)
        off += 27 * ci * co
        h = torch.nn.functional.conv3d(h, w.contiguous(), p[off:off + co], padding=1)
        off += co
        h = torch.relu(h) if l < 3 else h
    y = h.reshape(-1)
    if case["kind"] == "forward":
        return {"y": y.detach()}
    loss = (y - s["t"].double()).square().mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grads": p.grad}


class _Model:
    """residual of the discrete equations at a state that is also the step's start, in torch"""

    def __init__(self, case, state):
        f = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        self.c, self.fl, self.b = case, case["fluid"], case["model"]
        self.dims = (case["nz"], case["ny"], case["nx"])
        self.N = state[0].size
        self.sat = torch.from_numpy(state[3]).cuda() == 1
        self.x0 = torch.cat([f(a) for a in state[:self.b]])
        self.pv = f(case["poro"]) * (case["dx"] * case["dy"] * case["dz"])
        self.tab = {k: f(v) for k, v in self.fl.items() if k.startswith("pvt_")}
        self.wells = [w for w in case["wells"]]
        darcy = 86400.0 * 9.869233e-16 * 1e5 / 1e-3
        d = (case["dz"], case["dy"], case["dx"])
        vol = d[0] * d[1] * d[2]
        self.T = []
        for axis, name in enumerate(("kz", "ky", "kx")):
            k = f(case[name]).view(self.dims)
            m = self.dims[axis]
            self.T.append(darcy * 2.0 * (vol / d[axis]) / (d[axis] / k.narrow(axis, 0, m - 1) + d[axis] / k.narrow(axis, 1, m - 1)))
        self.depth = case["top_depth"] + (torch.arange(self.dims[0], device="cuda", dtype=torch.float64) + 0.5) * case["dz"]
        # perforations: cell, well index, reference depth, well
        cell, wi, zh, iw = [], [], [], []
        for w, W in enumerate(self.wells):
            for kk in range(W["k0"], W["k1"] + 1):
                i = W["i"] + case["nx"] * (W["j"] + case["ny"] * kk)
                a, b = float(case["kx"][i]), float(case["ky"][i])
                ro = 0.28 * math.sqrt(math.sqrt(b / a) * case["dx"] ** 2 + math.sqrt(a / b) * case["dy"] ** 2) / ((b / a) ** 0.25 + (a / b) ** 0.25)
                cell.append(i)
                wi.append(2.0 * math.pi * darcy * math.sqrt(a * b) * case["dz"] / (math.log(ro / W["rw"]) + W["skin"]))
                zh.append(case["top_depth"] + (W["k0"] + 0.5) * case["dz"])
                iw.append(w)
        self.pcell = torch.tensor(cell, device="cuda")
        self.pwi, self.pzh = f(wi), f(zh)
        self.pbhp = f([self.wells[w]["bhp"] for w in iw])
        self.pinj = torch.tensor([self.wells[w]["type"] == synth.WATER_INJECTOR for w in iw], device="cuda")
        self.acc0 = self.props(self.x0)[0]

    def lut(self, name, x):
        xp, yp = self.tab["pvt_p"], self.tab[name]
        k = (torch.searchsorted(xp, x.detach().contiguous(), right=True) - 1).clamp(0, xp.numel() - 2)
        return (x - xp[k]) * ((yp[k + 1] - yp[k]) / (xp[k + 1] - xp[k])) + yp[k]

    def props(self, x):
        """accumulations, phase densities, (phase, component, mobility) and the total mobility"""
        c, fl, N = self.c, self.fl, self.N
        p, sw = x[:N], x[N:2 * N]
        pv = ((p - c["p_ref"]) * c["c_rock"] + 1.0) * self.pv
        corey = lambda s, n: s.clamp(0.0, 1.0) ** n  # noqa: E731
        mob = 1.0 - fl["swc"] - fl["sor"]
        krw = corey((sw - fl["swc"]) / mob, fl["nw"])
        if self.b == 2:
            rw = torch.exp((p - c["p_ref"]) * fl["c_w"]) * fl["rho_w_ref"]
            ro = torch.exp((p - c["p_ref"]) * fl["c_o"]) * fl["rho_o_ref"]
            kro = corey(1.0 - (sw - fl["swc"]) / mob, fl["now"])
            return ([pv * rw * sw, pv * ro * (1.0 - sw)], [rw, ro],
                    [(0, 0, rw * krw / fl["mu_w"]), (1, 1, ro * kro / fl["mu_o"])], krw / fl["mu_w"] + kro / fl["mu_o"])
        x3, s = x[2 * N:], self.sat
        sg = torch.where(s, x3, torch.zeros_like(x3))
        pb = torch.where(s, p, x3)
        du = p - pb
        bo = self.lut("pvt_bo", pb) * (1.0 - du * fl["bo_c_us"])
        rs = self.lut("pvt_rs", pb)
        mo = self.lut("pvt_muo", pb) * (1.0 + du * fl["muo_c_us"])
        bw = (p - fl["bw_pref"]) * fl["bw_c"] + 1.0
        bg = 1.0 / self.lut("pvt_bg", p)
        so = 1.0 - sw - sg
        krow = corey(((1.0 - fl["sor"]) - sw) / mob, fl["now"])
        krg = corey((sg - fl["sgc"]) / (1.0 - fl["swc"] - fl["sorg"] - fl["sgc"]), fl["ng"])
        krog = corey(((1.0 - fl["swc"] - fl["sorg"]) - sg) / (1.0 - fl["swc"] - fl["sorg"]), fl["nog"])
        kro = ((krow + krw) * (krog + krg) - (krw + krg)).clamp_min(0.0)
        rho = [bw * fl["rho_ws"], (rs * fl["rho_gs"] + fl["rho_os"]) / bo, bg * fl["rho_gs"]]
        lw, lo, lg = krw / fl["mu_w"], kro / mo, krg / self.lut("pvt_mug", p)
        acc = [pv * bw * sw * fl["rho_ws"], pv * so / bo * fl["rho_os"], pv * (rs * so / bo + bg * sg) * fl["rho_gs"]]
        return acc, rho, [(0, 0, rho[0] * lw), (1, 1, fl["rho_os"] / bo * lo), (1, 2, rs / bo * fl["rho_gs"] * lo),
                          (2, 2, rho[2] * lg)], lw + lo + lg

    def residual(self, x, dt):
        acc, rho, mob, lam = self.props(x)
        R = [(a - a0) / dt for a, a0 in zip(acc, self.acc0)]
        p3 = x[:self.N].view(self.dims)
        for axis in range(3):
            m = self.dims[axis]
            L = lambda a: a.view(self.dims).narrow(axis, 0, m - 1)  # noqa: E731
            U = lambda a: a.view(self.dims).narrow(axis, 1, m - 1)  # noqa: E731
            gdz = 9.80665 * self.c["dz"] / 1e5 if axis == 0 else 0.0
            for ph, comp, mo in mob:
                dphi = (U(p3) - L(p3)) - 0.5 * (L(rho[ph]) + U(rho[ph])) * gdz
                F = self.T[axis] * torch.where(dphi.detach() > 0.0, U(mo), L(mo)) * dphi     # flow into the lower cell
                pad = [0, 0] * (2 - axis)
                R[comp] = R[comp] - (torch.nn.functional.pad(F, pad + [0, 1]) - torch.nn.functional.pad(F, pad + [1, 0])).reshape(-1)
        i = self.pcell
        z = self.depth[i // (self.dims[1] * self.dims[2])]
        dh = 9.80665 * (self.pzh - z) / 1e5
        dw = self.pbhp - x[:self.N][i] - rho[0][i] * dh
        inj = self.pinj & (dw.detach() >= 0.0)
        add = [torch.zeros_like(dw) for _ in R]
        for ph, comp, mo in mob:
            drop = torch.where(self.pinj, dw, self.pbhp - x[:self.N][i] - rho[ph][i] * dh)
            add[comp] = add[comp] + torch.where(inj, torch.zeros_like(dw), self.pwi * mo[i] * drop)
        add[0] = add[0] + torch.where(inj, self.pwi * rho[0][i] * lam[i] * dw, torch.zeros_like(dw))
        return torch.cat([r.index_add(0, i, -a) for r, a in zip(R, add)])

    def jacobian(self, dt):
        n = self.x0.numel()
        J = torch.empty((n, n), dtype=torch.float64, device="cuda")
        column = lambda v: torch.func.jvp(lambda x: self.residual(x, dt), (self.x0,), (v,))[1]  # noqa: E731
        for k in range(0, n, 500):
            e = torch.zeros((min(500, n - k), n), dtype=torch.float64, device="cuda")
            e[torch.arange(e.shape[0]), k + torch.arange(e.shape[0])] = 1.0
            J[:, k:k + e.shape[0]] = torch.func.vmap(column)(e).t()
        return J

    def cnv(self, R, dt):
        return max((R[k * self.N:(k + 1) * self.N].abs() * dt / (self.pv * self.c["cnv_rho"][k])).max() for k in range(self.b))

    def update(self, dx):
        """Appleyard chop, clamp and variable switch of the Newton update"""
        N, sv = self.N, self.c["solver"]
        d, x, sat = dx.view(self.b, N), self.x0.view(self.b, N).clone(), self.sat.clone()
        ds, dp = d[1].abs(), d[0].abs()
        if self.b == 3:
            ds = torch.where(sat, torch.maximum(ds, d[2].abs()), ds)
            dp = torch.where(sat, dp, torch.maximum(dp, d[2].abs()))
        one = torch.ones_like(ds)
        fct = torch.minimum(torch.where(ds > sv["chop_ds"], sv["chop_ds"] / ds, one), torch.where(dp > sv["chop_dp"], sv["chop_dp"] / dp, one))
        x = x + fct * d
        x[1] = x[1].clamp(0.0, 1.0)
        if self.b == 3:
            zero = torch.zeros_like(x[2])
            to_us, to_sat = sat & (x[2] < 0.0), ~sat & (x[2] > x[0])
            x[2] = torch.where(to_us, x[0], torch.where(to_sat, zero, x[2]))
            sat = (sat & ~to_us) | to_sat
            dry = ~sat & (x[1] > 1.0 - 1e-6)
            x[2] = torch.where(dry, zero, x[2])
            sat = sat | dry
            x[2] = torch.where(sat, torch.minimum(x[2], 1.0 - x[1]), x[2])
        return x.reshape(-1), sat.to(torch.int8)
