"""The work that users of this library have it do, as cases for measurement.

Every case goes through the public entry points of ``paper_0807_4471_gb300``
(the lattice handle, the lattice pool, the job server, checkpoint/restart, and
the totals of device fields) with the couplings of the paper's Fig. 2 caption
and Psi = rho0 (1 - exp(-rho/rho0)).  ``exact`` restates the model in plain
torch FP64, without the library.
"""
import math

import numpy as np
import torch

import paper_0807_4471_gb300 as lb
from paper_0807_4471_gb300.serve import Server, job_params

COUPLINGS = dict(G_A1=-12.55, G_A2=11.70, G_B1=-11.80, G_B2=10.95, G_X=0.58)
AMP = 0.03                      # initial densities rho0 (1 +- 3 %)
ELEM = dict(fp64=8, fp32=4, fp16=2, bf16=2)
STEP_FLOPS = 350                # both species: moments, Psi, force of Eq. (2), collision
LIBRARY_KEYS = ("boundary", "u_wall", "init_shear", "kolmo_amp", "kolmo_k", "tau_A", "tau_B", "rho0",
                "stress_every")


def listed():
    return [
        # The plain method: one FP64 lattice at the size of the paper's shear and ageing runs.
        dict(name="plain_fp64_128", kind="lattice", precision="fp64", nx=128, ny=128, steps=100),
        # FP64 at the paper's resolution, between moving walls: the reference run of a precision study.
        dict(name="couette_fp64_512", kind="lattice", precision="fp64", nx=512, ny=512, steps=50,
             shear=1e-4),
        # The Kolmogorov-shear experiment: one small forced lattice, fields every 100 steps.
        dict(name="kolmogorov_fp32_128", kind="lattice", precision="fp32", nx=128, ny=128, steps=100,
             kolmo=0.1),
        # A single small ragged shear run with unequal relaxation times (the general collision).
        dict(name="couette_fp32_tau_300x211", kind="lattice", precision="fp32", nx=300, ny=211, steps=200,
             shear=1e-4, tau_A=0.8),
        # The headline sweep over rho0 at the paper's resolution, stepped together in one pool.
        dict(name="sweep_fp32_5x512", kind="pool", precision="fp32", count=5, nx=512, ny=512, steps=400,
             couette=0.0),
        # The shear-rate sweep in FP16 offsets: eight plane-Couette lattices in one pool.
        dict(name="couette_fp16_8x512", kind="pool", precision="fp16", count=8, nx=512, ny=512, steps=200,
             couette=1.0),
        # The batched mix: uneven lattices, half of them sheared, one launch per step.
        dict(name="batch_fp16_24_mixed", kind="mix", precision="fp16", count=24, lo=128, hi=1024, steps=150),
        # The peak-bandwidth lattice, far larger than L2, in FP32 and in FP16 offsets.
        dict(name="peak_fp32_4096", kind="lattice", precision="fp32", nx=4096, ny=4096, steps=100),
        dict(name="peak_fp16_4096", kind="lattice", precision="fp16", nx=4096, ny=4096, steps=100),
        # Rheology jobs served by continuous batching: admission, uneven step counts, results.
        dict(name="serve_fp16_16_jobs", kind="serve", precision="fp16", count=16, lo=64, hi=1024,
             steps=300),
        # A long run in pieces: restore a state, step, write the next checkpoint.
        dict(name="restart_fp32_1024", kind="restart", precision="fp32", nx=1024, ny=1024, steps=100),
        # Mass and momentum of device fields for a caller that may not allocate.
        dict(name="totals_2048", kind="totals", nx=2048, ny=2048),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "pool", "mix", "serve", "restart", "totals"])
    prec = rng.choice(["fp64", "fp32", "fp32", "fp16", "fp16", "bf16"])
    # the demixing instability amplifies each format's rounding: runs stay short enough to compare
    most = dict(fp64=100, fp32=300, fp16=200, bf16=80)
    if kind == "lattice":
        hi = 700 if prec == "fp64" else 3600
        nx, ny = _log_int(rng, 32, hi), _log_int(rng, 32, hi)
        c = dict(kind=kind, precision=prec, nx=nx, ny=ny,
                 steps=rng.randint(20, min(most[prec], 80 if nx * ny > 1 << 22 else 200)))
        option = rng.choice(["", "", "shear", "kolmo", "tau"])
        if option == "shear":
            c["shear"] = 10.0 ** rng.uniform(-6, -4)
        elif option == "kolmo":
            c["kolmo"] = rng.uniform(0.01, 0.1)
        elif option == "tau":
            c["tau_A"] = rng.uniform(0.8, 1.1)
        return c
    if kind == "totals":
        return dict(kind=kind, nx=_log_int(rng, 32, 4096), ny=_log_int(rng, 32, 4096))
    if kind == "restart":
        return dict(kind=kind, precision=prec, nx=_log_int(rng, 64, 1024), ny=_log_int(rng, 64, 1024),
                    steps=rng.randint(20, min(most[prec], 100)))
    prec = "fp32" if prec == "fp64" else prec
    if kind == "pool":
        return dict(kind=kind, precision=prec, count=rng.randint(2, 8), nx=_log_int(rng, 96, 600),
                    ny=_log_int(rng, 96, 600), steps=rng.randint(50, most[prec]), couette=rng.choice([0.0, 0.5, 1.0]))
    if kind == "mix":
        return dict(kind=kind, precision=prec, count=rng.randint(4, 24), lo=rng.randint(64, 200),
                    hi=rng.randint(256, 700), steps=rng.randint(40, min(most[prec], 150)))
    return dict(kind=kind, precision=prec, count=rng.randint(4, 16), lo=64, hi=rng.randint(128, 1000),
                steps=rng.randint(60, most[prec]))


# ------------------------------------------------------------------ inputs
def _members(case, seed):
    """The lattices of a case, each as the arguments of lb.make_params, and
    for a served job its step count and its own seed."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("lattice", "restart"):
        m = dict(nx=case["nx"], ny=case["ny"], rho0=0.70)
        if case.get("shear"):
            m.update(boundary=1, u_wall=case["shear"] * case["ny"] / 2.0, init_shear=1)
        if case.get("kolmo"):
            k = 2.0 * math.pi / case["ny"]
            m.update(kolmo_amp=k * k * case["kolmo"] / 6.0, kolmo_k=1.0)
        if case.get("tau_A"):
            m.update(tau_A=case["tau_A"], tau_B=1.0)
        return [m]
    out = []
    shape = np.random.default_rng(7919 * case["count"] + case.get("hi", 0))   # sizes belong to the case
    for j in range(case["count"]):
        if kind == "pool":
            nx, ny = case["nx"], case["ny"]
            couette = j < round(case["couette"] * case["count"])
        elif kind == "mix":
            nx = ny = int(round(math.exp(shape.uniform(math.log(case["lo"]), math.log(case["hi"])))))
            couette = j % 2 == 1
        else:   # served jobs: sides are multiples of 8, the sizes spread evenly over the range
            q = (j + shape.uniform()) / case["count"]
            nx = ny = int(math.ceil(case["lo"] * (case["hi"] / case["lo"]) ** q / 8) * 8)
            couette = j % 3 != 0
        if kind == "pool":
            rho0 = 0.55 + 0.28 * (j + 0.5) / case["count"]
        else:
            rho0 = float(rng.uniform(0.55, 0.83))
        rate = float(10.0 ** rng.uniform(-5, -4)) if couette else 0.0
        m = dict(nx=nx, ny=ny, rho0=rho0)
        if couette:   # pool members restart from densities at rest, served jobs on the shear profile
            m.update(boundary=1, u_wall=rate * ny / 2.0, init_shear=int(kind == "serve"))
        if kind == "serve":
            m.update(shear_rate=rate, seed=int(rng.integers(0, 2 ** 31)),
                     steps=int(case["steps"] * shape.uniform(0.25, 1.0)))
        out.append(m)
    return out


def _params(m, precision):
    kw = {k: m[k] for k in LIBRARY_KEYS if k in m}
    return lb.make_params(m["nx"], m["ny"], precision, psi_form=lb.LB_PSI_RHO0, init_amp=AMP, **COUPLINGS, **kw)


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()


def _densities(m, seed, j):
    """Initial densities of a pool member, FP64 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed * 1009 + j)
    u = torch.rand((2, m["ny"], m["nx"]), generator=g, device="cuda", dtype=torch.float64)
    return m["rho0"] * (1.0 + AMP * (2.0 * u - 1.0))


def _restart_state(case, seed):
    """A post-collision state f* [2][9][ny][nx]: equilibrium at rest of random
    densities, with a small random non-equilibrium part."""
    g = torch.Generator(device="cuda").manual_seed(seed + 17)
    shape = (case["ny"], case["nx"])
    rho = 0.70 * (1.0 + AMP * (2.0 * torch.rand((2, 1) + shape, generator=g, device="cuda", dtype=torch.float64) - 1.0))
    w = torch.tensor(W, device="cuda", dtype=torch.float64).view(1, 9, 1, 1)
    eps = torch.rand((2, 9) + shape, generator=g, device="cuda", dtype=torch.float64) - 0.5
    return w * rho * (1.0 + 0.01 * eps)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "totals":
        # device fields as lb_fields lays them out: densities near 0.7, velocities of a slow shear
        g = torch.Generator(device="cuda").manual_seed(seed)
        u = torch.rand((4, case["ny"], case["nx"]), generator=g, device="cuda", dtype=torch.float64)
        fields = [0.7 * (1.0 + AMP * (2.0 * u[0] - 1.0)), 0.7 * (1.0 + AMP * (2.0 * u[1] - 1.0)),
                  0.02 * u[2] - 0.005, 0.01 * u[3] - 0.002]
        # the first call on a device looks up the library's scratch array
        totals = torch.zeros(4, device="cuda", dtype=torch.float64)
        lb.load()
        return dict(kind=kind, nx=case["nx"], ny=case["ny"], fields=fields, totals=totals)
    ms = _members(case, seed)
    prec = case["precision"]
    st = dict(kind=kind, seed=seed, steps=case["steps"])
    if kind in ("lattice", "restart"):
        m = ms[0]
        st["lattice"] = lb.Lattice(_params(m, prec))
        if kind == "lattice":
            st["out"] = [_pinned((m["ny"], m["nx"])) for _ in range(4)]
        else:
            st["state"], st["out"] = _pinned((2, 9, m["ny"], m["nx"])), _pinned((2, 9, m["ny"], m["nx"]))
            st["state"][:] = _restart_state(case, seed).cpu().numpy()
        return st
    if kind == "serve":
        st["make"] = job_params(lb, dict(psi_form=lb.LB_PSI_RHO0, init_amp=AMP, **COUPLINGS), prec)
        st["specs"] = [{k: m[k] for k in ("nx", "ny", "rho0", "shear_rate", "steps", "seed")} for m in ms]
        # room for about half of the jobs: the others wait for memory, as under load
        sizes = [lb.Pool.footprint(st["make"](s)) for s in st["specs"]]
        budget = max(max(sizes), sum(sizes) // 2) + (1 << 20)
        st["stream"] = torch.cuda.Stream()
        st["pool"] = lb.Pool(st["make"](dict(nx=64, ny=64)), budget, max_jobs=64, stream=st["stream"])
        return st
    ps = [_params(m, prec) for m in ms]
    st["stream"] = torch.cuda.Stream()
    budget = sum(lb.Pool.footprint(p) for p in ps) + (16 << 20)
    st["pool"] = pool = lb.Pool(ps[0], budget, max_jobs=len(ps), stream=st["stream"])
    st["jobs"] = [pool.admit(p, seed + j, 1 << 40) for j, p in enumerate(ps)]
    st["in"] = [_pinned((2, m["ny"], m["nx"])) for m in ms]
    st["out"] = [_pinned((2, m["ny"], m["nx"])) for m in ms]
    for j, (m, a) in enumerate(zip(ms, st["in"])):
        a[:] = _densities(m, seed, j).cpu().numpy()
    pool.run(1024)       # long runs are tuned on their first steps
    st["stream"].synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "totals":
        a, b, ux, uy = st["fields"]
        lb.lb_totals_noalloc(st["nx"], st["ny"], a.data_ptr(), b.data_ptr(), ux.data_ptr(), uy.data_ptr(),
                             st["totals"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return st["totals"]
    if kind == "lattice":
        g = st["lattice"]
        g.init_seeded(st["seed"])
        g.step(st["steps"])
        lb.lb_fields(g.h, *st["out"])
        return st["out"]
    if kind == "restart":
        g = st["lattice"]
        g.resume(st["state"], 1000, 1)
        g.step(st["steps"])
        lb.lb_checkpoint(g.h, st["out"])
        return st["out"]
    pool = st["pool"]
    if kind == "serve":
        srv = Server(pool, st["make"], quantum=100, keep_fields=True)
        jobs = [srv.submit(s) for s in st["specs"]]
        srv.run_until_idle()
        return [j.result["fields"][:2] for j in jobs] + [[j.result["sigma_mean"] for j in jobs]]
    for j, a in zip(st["jobs"], st["in"]):
        pool.init_fields(j, a[0], a[1])
    pool.run(st["steps"])
    for j, a in zip(st["jobs"], st["out"]):
        lb.lb_pool_fields(pool.h, j, a[0], a[1])
    return st["out"]


def work(case):
    """Every time step reads and writes the 18 populations of every site once;
    inputs and fields that cross to or from the host count once."""
    if case["kind"] == "totals":
        n = case["nx"] * case["ny"]
        return dict(bytes=32 * n, flops=7 * n)
    steps = case["steps"]
    total = dict(bytes=0, flops=0)
    for m in _members(case, 0):
        n, k = m["nx"] * m["ny"], m.get("steps", steps)
        io = {"lattice": 32, "serve": 16, "restart": 288}.get(case["kind"], 32)
        total["bytes"] += n * (36 * ELEM[case["precision"]] * k + io)
        total["flops"] += n * STEP_FLOPS * k
    return total


# ------------------------------------------------- the model in 64 bits
C9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
W_BELT = {1: 1 / 9, 2: 1 / 36}
P_BELT = {1: 4 / 63, 2: 4 / 135, 4: 1 / 180, 5: 2 / 945, 8: 1 / 15120}


class _Model:
    """One lattice in torch FP64: state f [2][9][ny][nx] before collision."""

    def __init__(self, m):
        self.m, self.rho0 = m, m["rho0"]
        self.walls = bool(m.get("boundary"))
        self.uw = m.get("u_wall", 0.0)
        self.tau = torch.tensor([m.get("tau_A", 1.0), m.get("tau_B", 1.0)], device="cuda",
                                dtype=torch.float64).view(2, 1, 1)
        c = COUPLINGS
        self.Ga, self.Gr = (c["G_A1"], c["G_B1"]), (c["G_A2"], c["G_B2"])
        y = torch.arange(m["ny"], device="cuda", dtype=torch.float64).view(-1, 1)
        self.acc = m.get("kolmo_amp", 0.0) * torch.sin(2 * math.pi * m.get("kolmo_k", 0.0) / m["ny"] * y)
        self.y = y

    def equilibrium(self, rho, ux, uy):
        usq = 1.5 * (ux * ux + uy * uy)
        f = []
        for (cx, cy), w in zip(C9, W):
            cu = 3.0 * (cx * ux + cy * uy)
            f.append(w * rho * (1.0 + cu + 0.5 * cu * cu - usq))
        return torch.stack(f, 1)

    def start(self, rho):
        ux = torch.zeros_like(rho)
        if self.m.get("init_shear"):
            ux = ux + self.uw * (2.0 * self.y + 1.0 - self.m["ny"]) / self.m["ny"]
        self.f = self.equilibrium(rho, ux, torch.zeros_like(rho))

    def _pad(self, q):
        """Two rows beyond each edge: periodic images, or the mirror at halfway walls."""
        if self.walls:
            return torch.cat([q[:, 1:2], q[:, 0:1], q, q[:, -1:], q[:, -2:-1]], 1)
        return torch.cat([q[:, -2:], q, q[:, :2]], 1)

    def forces(self, rho):
        ny = rho.shape[1]
        psi = self.rho0 * (1.0 - torch.exp(-rho / self.rho0))
        pp, pr = self._pad(psi), self._pad(rho)
        sx, sy = torch.zeros_like(rho), torch.zeros_like(rho)
        qx, qy = torch.zeros_like(rho), torch.zeros_like(rho)
        for dy in range(-2, 3):
            for dx in range(-2, 3):
                d2 = dx * dx + dy * dy
                if d2 == 0:
                    continue
                v = torch.roll(pp[:, 2 + dy:2 + dy + ny], -dx, 2)
                for s in range(2):
                    K = self.Ga[s] * W_BELT.get(d2, 0.0) + self.Gr[s] * P_BELT[d2]
                    if dx:
                        sx[s] += K * dx * v[s]
                    if dy:
                        sy[s] += K * dy * v[s]
                if d2 <= 2:
                    r = torch.roll(pr[:, 2 + dy:2 + dy + ny], -dx, 2)
                    if dx:
                        qx += W_BELT[d2] * dx * r
                    if dy:
                        qy += W_BELT[d2] * dy * r
        g = COUPLINGS["G_X"] / self.rho0
        Fx = -psi * sx - g * rho * qx.flip(0) + rho * self.acc
        Fy = -psi * sy - g * rho * qy.flip(0)
        return Fx, Fy

    def moments(self):
        f = self.f
        jx = f[:, 1] - f[:, 3] + f[:, 5] - f[:, 6] - f[:, 7] + f[:, 8]
        jy = f[:, 2] - f[:, 4] + f[:, 5] + f[:, 6] - f[:, 7] - f[:, 8]
        return f.sum(1), jx, jy

    def collide(self):
        rho, jx, jy = self.moments()
        Fx, Fy = self.forces(rho)
        den = (rho / self.tau).sum(0)
        ux = (jx / self.tau).sum(0) / den + self.tau * Fx / rho
        uy = (jy / self.tau).sum(0) / den + self.tau * Fy / rho
        self.f = self.f + (self.equilibrium(rho, ux, uy) - self.f) / self.tau.view(2, 1, 1, 1)

    def stream(self):
        s = self.f
        out = []
        for i, (cx, cy) in enumerate(C9):
            v = torch.roll(s[:, i], (cy, cx), (1, 2))
            if self.walls and cy:
                row, u = (0, -self.uw) if cy == 1 else (-1, self.uw)
                rw = s[:, :, row].sum(1)
                v[:, row] = s[:, OPP[i], row] + 6.0 * W[i] * cx * u * rw
            out.append(v)
        self.f = torch.stack(out, 1)

    def fields(self):
        rho, jx, jy = self.moments()
        Fx, Fy = self.forces(rho)
        tot = rho.sum(0)
        return [rho[0], rho[1], (jx + 0.5 * Fx).sum(0) / tot, (jy + 0.5 * Fy).sum(0) / tot]


def _mix64(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _seeded(m, seed):
    """The densities of lb_init_seeded: rho0 (1 + amp (2u - 1)), u from the
    SplitMix64 counter generator the header documents."""
    idx = np.arange(2 * m["ny"] * m["nx"], dtype=np.uint64)
    z = _mix64(np.uint64(seed) ^ _mix64(idx + np.uint64(0x9E3779B97F4A7C15)))
    u = (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    rho = m["rho0"] * (1.0 + AMP * (2.0 * u - 1.0))
    return torch.from_numpy(rho.reshape(2, m["ny"], m["nx"])).cuda()


def exact(case, seed):
    kind = case["kind"]
    if kind == "totals":
        a, b, ux, uy = prepare(case, seed)["fields"]
        t = a + b
        return torch.stack([a.sum(), b.sum(), (t * ux).sum(), (t * uy).sum()])
    results = []
    for j, m in enumerate(_members(case, seed)):
        model = _Model(m)
        if kind == "restart":
            model.f = _restart_state(case, seed)
            for _ in range(case["steps"]):
                model.stream()
                model.collide()
            return model.f
        model.start(_seeded(m, seed if kind == "lattice" else m["seed"]) if kind in ("lattice", "serve")
                    else _densities(m, seed, j))
        for _ in range(m.get("steps", case["steps"])):
            model.collide()
            model.stream()
        f = model.fields()
        if kind == "lattice":
            return f
        results.append(f[:2] if kind == "serve" else torch.stack(f[:2]))
    if kind == "serve":
        results.append([None] * case["count"])     # the wall stress is checked against the start's
    return results
