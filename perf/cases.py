"""What the speed of liblbpc is measured on: the work its users have it do, through lbpc.Simulation and
lbpc.Batch, over the sizes, precisions, boundaries and options they use.

A pass advances one simulation by a chunk of time steps and reads its fields on the device (a run that is
watched: droplet area, vapour volume), or reads the domain sums after every step (a monitored run), or
resumes a run from a checkpoint kept on the device (a sweep that starts from one relaxed pool), or advances
a batch of uneven simulations by a service's chunk and reads back those that are done.

listed() is the list that is reported; draw() gives further cases of the same ranges. exact() evaluates the
same method in binary64 with torch operations on whole arrays, independently of the library.
"""

import numpy as np
import torch

from paper_1709_04400_gb300 import lbpc

# Working point of every case: Peng-Robinson with the default constants at T_s = 0.86 T_c.
A, B, R, OMEGA = 3.0 / 49.0, 2.0 / 21.0, 1.0, 0.344
TC = 0.0778 * A / (0.45724 * B * R)
TS = 0.86 * TC
RHO_V, RHO_L = 0.37967899939971905, 6.498945763287887  # coexistence densities at T_s
S_F = (1.0, 0.8, 0.8, 1.0, 1.1, 1.0, 1.1, 1.25, 1.25)
S_G_UNIT = (1.0,) * 9
S_G_MIXED = (1.0, 0.9, 1.05, 1.0, 1.2, 1.0, 1.2, 0.95, 0.85)
CV = 5.0

PREC = {"fp64": lbpc.FP64, "fp32": lbpc.FP32, "fp16": lbpc.FP16DEV, "df64": lbpc.DF64}
MODEL = {"improved": lbpc.IMPROVED, "compromised": lbpc.COMPROMISED, "gong_cheng": lbpc.GONG_CHENG}
KIND = {"periodic": lbpc.PERIODIC, "wall": lbpc.WALL, "pressure": lbpc.PRESSURE}
STATE_BYTES = {"fp64": 304, "df64": 304, "fp32": 152, "fp16": 96}  # state read and written once per node and step
FLOPS = 330  # operations of one coupled step at one node
RELAX = 100  # steps of a pool before its checkpoint is taken


def listed():
    return [
        # the smallest simulations: a periodic droplet in binary64, the case that pins the method's accuracy;
        # its steps take microseconds each, so launches and latency count
        dict(name="droplet_128_fp64", kind="sim", setup="droplet", nx=128, ny=128, prec="fp64", read="fields",
             steps=100),
        # D^2-law runs: droplet evaporation in a held ring, mass and heat watched after every step
        dict(name="evaporation_256_fp64", kind="sim", setup="evaporation", nx=256, ny=256, prec="fp64",
             read="sums", steps=100),
        # the same in binary64 at the size the library's own benchmark reports
        dict(name="evaporation_2048_fp64", kind="sim", setup="evaporation", nx=2048, ny=2048, prec="fp64",
             read="fields", steps=20),
        # binary64-grade accuracy at scale: double-word arithmetic
        dict(name="evaporation_2048_df64", kind="sim", setup="evaporation", nx=2048, ny=2048, prec="df64",
             read="fields", steps=60),
        # a droplet on a heated surface under an open top, a small grid in double-word arithmetic
        dict(name="surface_300x150_df64", kind="sim", setup="surface", nx=300, ny=150, prec="df64",
             read="resume", steps=100),
        # nucleation over a heated strip under a held-pressure top, binary32
        dict(name="nucleation_300x400_fp32", kind="sim", setup="open_pool", nx=300, ny=400, prec="fp32",
             read="resume", steps=200),
        # bubble departure in a closed pool: rows that are no multiple of 16 bytes, buoyancy against the mean
        dict(name="bubble_150x300_fp32", kind="sim", setup="closed_pool", nx=150, ny=300, prec="fp32",
             read="resume", steps=200),
        # a mid-size grid with odd sides and the thermal rates all different
        dict(name="evaporation_1023x1025_fp32", kind="sim", setup="evaporation", nx=1023, ny=1025, prec="fp32",
             read="fields", steps=100, rates="mixed"),
        # the large binary32 run
        dict(name="evaporation_4096_fp32", kind="sim", setup="evaporation", nx=4096, ny=4096, prec="fp32",
             read="fields", steps=150),
        # the large run with binary16 storage, which runs beside a service
        dict(name="evaporation_4096_fp16", kind="sim", setup="evaporation", nx=4096, ny=4096, prec="fp16",
             read="fields", steps=150),
        # a service's chunk: uneven requests, half evaporation and half heated pools, binary32
        dict(name="batch_64_fp32", kind="batch", count=64, lo=64, hi=512, mix=1, pools=True, prec="fp32", steps=256),
        # the same form with binary16 storage, evaporation requests only
        dict(name="batch_24_fp16", kind="batch", count=24, lo=64, hi=512, mix=2, pools=False, prec="fp16", steps=256),
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    if rng.random() < 0.2:
        lo = log_uniform(48, 128)
        return dict(kind="batch", count=log_uniform(6, 64), lo=lo, hi=log_uniform(lo + 16, 512), mix=rng.randrange(1000),
                    pools=rng.random() < 0.5, prec=rng.choice(["fp32", "fp32", "fp16", "fp64"]), steps=64)
    setup = rng.choice(["droplet", "evaporation", "evaporation", "surface", "open_pool", "closed_pool"])
    prec = rng.choice(["fp64", "df64", "fp32", "fp32", "fp16"])
    pool = setup in ("surface", "open_pool", "closed_pool")
    if setup in ("open_pool", "closed_pool") and prec == "fp16":
        prec = "fp32"
    nx = log_uniform(100, 800) if pool else log_uniform(64, {"fp64": 1500, "df64": 2048}.get(prec, 4000))
    ny = min(max(int(nx * (0.6 + 0.9 * rng.random())), 96), 4000)
    if rng.random() < 0.4:  # binary16 and binary32 rows of whole 16-byte pieces are common in practice
        nx, ny = nx & ~7, ny & ~7
    nodes = nx * ny
    steps = max(10, min(100, int((2e7 if prec == "fp64" else 8e7) / nodes)))
    read = "resume" if pool else rng.choice(["fields", "fields", "sums"])
    case = dict(kind="sim", setup=setup, nx=nx, ny=ny, prec=prec, read=read, steps=steps)
    if rng.random() < 0.2:
        case["rates"] = "mixed"
    elif not pool and rng.random() < 0.2:
        case["model"] = rng.choice(["compromised", "gong_cheng"])
    return case


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------


def _rand(seed, n):
    return np.random.RandomState(seed % (1 << 31)).random_sample(n)


def _droplet(nx, ny, radius, cx, cy):
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    r = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2)
    return 0.5 * (RHO_L + RHO_V) - 0.5 * (RHO_L - RHO_V) * torch.tanh(2.0 * (r - radius) / 4.0)


def _setup(setup, nx, ny, seed, rates="unit", model="improved"):
    """(parameters as a plain dict, rho, T): the physical set-up and its seeded start, on the device."""
    u = _rand(seed, 8)
    p = dict(nx=nx, ny=ny, s_f=S_F, s_g=S_G_MIXED if rates == "mixed" else S_G_UNIT, sigma=0.1, cV=CV, model=model,
             lambda_const=True, lam=2.0 / 3.0, chi=0.0, gy=0.0, buoyancy=0, bottom="periodic", top="periodic",
             rho_top=0.0, t_bc=(False,) * 4, T_bc=(0.0,) * 4, strip=None, G_wall=0.0)
    if setup == "droplet":  # saturated droplet, temperature with a seeded sinusoid of 0.01 T_c
        rho = _droplet(nx, ny, (0.18 + 0.04 * u[0]) * min(nx, ny), nx / 2.0, ny / 2.0)
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] / ny
        x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] / nx
        T = TS + 0.01 * TC * torch.sin(2.0 * np.pi * ((1 + int(4 * u[1])) * x + (1 + int(4 * u[2])) * y + u[3]))
    elif setup == "evaporation":  # droplet at T_s in superheated vapour inside a held ring
        dT = (0.05 + 0.15 * u[0]) * TC
        rho = _droplet(nx, ny, (0.14 + 0.04 * u[1]) * min(nx, ny), nx / 2.0 + u[2], ny / 2.0 + u[3])
        T = TS + dT * (RHO_L - rho) / (RHO_L - RHO_V)
        p.update(t_bc=(True,) * 4, T_bc=(TS + dT,) * 4)
    elif setup == "surface":  # droplet on a heated non-wetting wall under an open top
        rho = _droplet(nx, ny, (0.25 + 0.04 * u[0]) * min(nx, ny), nx / 2.0 + u[1], 12.0)
        T = torch.full((ny, nx), TS, dtype=torch.float64, device="cuda")
        p.update(lambda_const=False, chi=0.08, bottom="wall", top="pressure", rho_top=RHO_V,
                 t_bc=(False, False, True, True), T_bc=(0.0, 0.0, (0.87 + 0.005 * u[2]) * TC, TS), G_wall=0.08)
    else:  # a pool over a heated strip, with density noise
        surface = ny / 2.0 if setup == "open_pool" else ny - min(ny // 2, 40)
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
        rho = 0.5 * (RHO_L + RHO_V) - 0.5 * (RHO_L - RHO_V) * torch.tanh(2.0 * (y - surface) / 4.0)
        noise = torch.rand((ny, nx), dtype=torch.float64, device="cuda",
                           generator=torch.Generator("cuda").manual_seed(seed))
        rho = rho + 1e-4 * (2.0 * noise - 1.0)
        T = torch.full((ny, nx), TS, dtype=torch.float64, device="cuda")
        width = max(4, nx // 15)
        p.update(lambda_const=False, chi=0.06, gy=-3e-5, bottom="wall", t_bc=(False, False, True, True),
                 T_bc=(0.0, 0.0, TS, TS), strip=(nx // 2 - width // 2, nx // 2 - width // 2 + width,
                                                 TS + (0.2 + 0.1 * u[0]) * TC))
        if setup == "open_pool":
            p.update(top="pressure", rho_top=RHO_V, buoyancy=2)
        else:
            p.update(top="wall", buoyancy=1, G_wall=-0.1)
    return p, rho.contiguous(), T.contiguous()


def _params(p, prec):
    edge = (lbpc.PERIODIC, lbpc.PERIODIC, KIND[p["bottom"]], KIND[p["top"]])
    return lbpc.Params(
        nx=p["nx"], ny=p["ny"], prec=PREC[prec], model=MODEL[p["model"]], s_f=p["s_f"], s_g=p["s_g"],
        sigma=p["sigma"], lambda_mode=lbpc.LAMBDA_CONST if p["lambda_const"] else lbpc.LAMBDA_RHO_CV_CHI,
        lam=p["lam"], chi=p["chi"] or 0.06, cV=p["cV"], gy=p["gy"], buoyancy=p["buoyancy"], flow_bc=edge,
        rho_bc=(0.0, 0.0, 0.0, p["rho_top"]), t_bc=[int(b) for b in p["t_bc"]], T_bc=p["T_bc"], strip=p["strip"],
        G_wall=p["G_wall"])


def _instances(case, seed):
    """Of each instance of a batch: (set-up, nx, ny, seed). Sizes belong to the case, the rest to the seed."""
    u = _rand(7919 * case["mix"] + 13, 2 * case["count"])
    out = []
    for k in range(case["count"]):
        n = case["lo"] + int(u[2 * k] * (case["hi"] - case["lo"] + 1))
        out.append(("closed_pool" if case["pools"] and k % 2 else "evaporation", n, n, seed + 101 * k))
    return out


def _done(case):
    """The instances that are read back after a chunk: about one in eight."""
    return list(range(1, case["count"], 8)) if case["count"] > 1 else [0]


def _single(prec):
    """Fields of the types that compute in binary32 are binary32 values; the others are binary64."""
    return prec in ("fp32", "fp16")


# ------------------------------------------------------------------------------------------------
# the measured passes
# ------------------------------------------------------------------------------------------------


def prepare(case, seed):
    if case["kind"] == "batch":
        made = [(_setup(*i), i) for i in _instances(case, seed)]
        params = [_params(p, case["prec"]) for (p, _, _), _ in made]
        room = sum(lbpc.Batch.instance_bytes(q) for q in params) + 13 * 8 * case["hi"] ** 2 + (64 << 20)
        batch = lbpc.Batch(PREC[case["prec"]], room, max_instances=case["count"] + 8)
        ids = [batch.add(q, rho.cpu().numpy(), T.cpu().numpy()) for q, ((_, rho, T), _) in zip(params, made)]
        return dict(case=case, batch=batch, ids=ids)
    p, rho, T = _setup(case["setup"], case["nx"], case["ny"], seed, case.get("rates", "unit"),
                       case.get("model", "improved"))
    sim = lbpc.Simulation(_params(p, case["prec"]))
    sim.init(rho, T)
    state = dict(case=case, sim=sim)
    if case["read"] == "sums":
        state["sums"] = torch.empty((case["steps"], 2), dtype=torch.float64, pin_memory=True)
    if case["read"] == "resume":
        sim.step(RELAX)
        state["checkpoint"] = sim.save(torch.empty(sim.checkpoint_bytes(), dtype=torch.uint8, device="cuda"))
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        batch.check()
        got = [batch.fields(state["ids"][k]) for k in _done(case)]
        if _single(case["prec"]):
            got = [[x.astype(np.float32) for x in f] for f in got]
        return [list(f) for f in got]
    sim = state["sim"]
    if case["read"] == "resume":
        sim.load(state["checkpoint"])
    if case["read"] == "sums":
        sums = state["sums"]
        for k in range(case["steps"]):
            sim.step(1, sync=False)
            sim.sums_async(sums[k])
        sim.check()
    else:
        sim.step(case["steps"])
    fields = sim.fields(device=True)
    if _single(case["prec"]):
        fields = [x.to(torch.float32) for x in fields]
    out = dict(zip(("rho", "ux", "uy", "T"), fields))
    if case["read"] == "sums":
        out["sums"] = state["sums"].to(torch.float32) if _single(case["prec"]) else state["sums"]
    return out


def work(case):
    """The state is read and written once per step; what is read out is written once per pass."""
    if case["kind"] == "batch":
        sizes = [nx * ny for _, nx, ny, _ in _instances(case, 0)]
        nodes, out = sum(sizes), sum(sizes[k] for k in _done(case))
    else:
        nodes = out = case["nx"] * case["ny"]
    width = 4 if _single(case["prec"]) else 8
    return dict(bytes=nodes * case["steps"] * STATE_BYTES[case["prec"]] + out * 4 * width,
                flops=nodes * case["steps"] * FLOPS)


# ------------------------------------------------------------------------------------------------
# the same in binary64, as torch operations on whole arrays
# ------------------------------------------------------------------------------------------------

E = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))


def _basis():
    """Rows (rho, e, eps, jx, qx, jy, qy, pxx, pxy) of the D2Q9 moments, and the inverse."""
    rows = []
    for ex, ey in E:
        s = ex * ex + ey * ey
        rows.append((1, 3 * s - 4, 4 - 10.5 * s + 4.5 * s * s, ex, (3 * s - 5) * ex, ey, (3 * s - 5) * ey,
                     ex * ex - ey * ey, ex * ey))
    M = torch.tensor(rows, dtype=torch.float64, device="cuda").T.contiguous()
    return M, torch.linalg.inv(M)


def _apply(M, x):
    return torch.matmul(M, x.reshape(9, -1)).reshape(x.shape)


class _Whole:
    """One simulation as whole arrays in binary64."""

    def __init__(self, p, rho, T):
        self.p = p
        self.M, self.Mi = _basis()
        self.periodic = p["bottom"] == "periodic"
        z = torch.zeros_like(rho)
        self.f = self.close_flow(_apply(self.Mi, self.flow_eq(rho, z, z)), None)
        self.g = self.close_heat(_apply(self.Mi, self.heat_eq(T, z, z)))
        self.phi = None
        self.mean = float(self.f.sum(0).mean())

    def flow_eq(self, rho, vx, vy):
        v2 = vx * vx + vy * vy
        return torch.stack([rho, rho * (3 * v2 - 2), rho * (1 - 3 * v2), rho * vx, -rho * vx, rho * vy, -rho * vy,
                            rho * (vx * vx - vy * vy), rho * vx * vy])

    def heat_eq(self, T, vx, vy):
        if self.p["model"] == "gong_cheng":
            return self.flow_eq(T, vx, vy)
        z = torch.zeros_like(T)
        return torch.stack([T, -2 * T, 2 * T if self.p["model"] == "improved" else T, T * vx, -T * vx, T * vy, -T * vy, z, z])

    def near(self, X, dx, dy):
        """X at the neighbour (dx, dy): x wraps, y wraps or repeats the edge row."""
        X = torch.roll(X, -dx, 1) if dx else X
        if not dy:
            return X
        if self.periodic:
            return torch.roll(X, -dy, 0)
        return torch.cat([X[1:], X[-1:]]) if dy > 0 else torch.cat([X[:1], X[:-1]])

    def slope(self, X):
        n = {e: self.near(X, *e) for e in E[1:]}
        dx = (n[1, 0] - n[-1, 0]) / 3 + (n[1, 1] - n[-1, 1] + n[1, -1] - n[-1, -1]) / 12
        dy = (n[0, 1] - n[0, -1]) / 3 + (n[1, 1] + n[-1, 1] - n[1, -1] - n[-1, -1]) / 12
        lap = (n[1, 0] + n[-1, 0] + n[0, 1] + n[0, -1] - 4 * X) * 2 / 3 + (
            n[1, 1] + n[-1, 1] + n[1, -1] + n[-1, -1] - 4 * X) / 6
        return dx, dy, lap

    def close_flow(self, f, F):
        """Zou-He rows: a wall sets j to minus half the force of the step before, a held density u_x = 0."""
        if self.periodic:
            return f
        for row, kind, s, (a, b, c), (ao, bo, co) in ((0, self.p["bottom"], 1.0, (2, 5, 6), (4, 7, 8)),
                                                      (-1, self.p["top"], -1.0, (4, 7, 8), (2, 5, 6))):
            q = f[:, row].clone()
            d = 0.5 * (q[1] - q[3]) * s
            if kind == "wall":
                jx, jy = (torch.zeros_like(d), torch.zeros_like(d)) if F is None else (-0.5 * F[0][row], -0.5 * F[1][row])
            else:
                jx = torch.zeros_like(d)
                jy = s * (self.p["rho_top"] - (q[0] + q[1] + q[3] + 2 * (q[ao] + q[bo] + q[co])))
            f[a, row] = q[ao] + s * 2 / 3 * jy
            f[b, row] = q[bo] - d + s * (0.5 * jx + jy / 6)
            f[c, row] = q[co] + d - s * (0.5 * jx - jy / 6)
        return f

    def rest(self, T):
        T = torch.as_tensor(T, dtype=torch.float64, device="cuda").reshape(-1)
        z = torch.zeros_like(T)
        return torch.matmul(self.Mi, self.heat_eq(T, z, z))

    def close_heat(self, g):
        p = self.p
        low = torch.full((p["nx"],), p["T_bc"][2], dtype=torch.float64, device="cuda")
        if p["strip"] is not None:
            low[p["strip"][0]:p["strip"][1]] = p["strip"][2]
        if not self.periodic:
            for row, edge, T, new, old in ((0, 2, low, (2, 5, 6), (4, 7, 8)), (-1, 3, p["T_bc"][3], (4, 7, 8), (2, 5, 6))):
                e = self.rest(T)
                for a, b in zip(new, old):
                    g[a, row] = 2 * e[a] - g[b, row] if p["t_bc"][edge] else g[b, row]
        if p["t_bc"][0]:
            g[:, :, 0] = self.rest(p["T_bc"][0])
        if p["t_bc"][1]:
            g[:, :, -1] = self.rest(p["T_bc"][1])
        if self.periodic and p["t_bc"][2]:
            g[:, 0] = self.rest(low)
        if self.periodic and p["t_bc"][3]:
            g[:, -1] = self.rest(p["T_bc"][3])
        return g

    def fluid(self):
        """rho, T, force, velocity and what the source needs of the equation of state."""
        p, f = self.p, self.f
        rho, T = f.sum(0), self.g.sum(0)
        kappa = 0.37464 + 1.54226 * OMEGA - 0.26992 * OMEGA ** 2
        th = 1 + kappa * (1 - torch.sqrt(T / TC))
        attract = A * rho * rho / (1 + 2 * B * rho - B * B * rho * rho)
        repel = rho * R / (1 - B * rho)
        pressure = repel * T - attract * th * th
        dpdT = repel + attract * kappa * th / torch.sqrt(T * TC)
        psi = torch.sqrt(2 * (rho / 3 - pressure))
        sx, sy, _ = self.slope(psi)
        Fx, Fy = psi * sx, psi * sy
        Q = 12 * p["sigma"] / (1 / p["s_f"][1] - 0.5) * (sx * sx + sy * sy)
        if p["bottom"] == "wall":
            Fy[0] += 0.5 * p["G_wall"] * psi[0] ** 2
        if p["buoyancy"]:
            Fy = Fy + (rho - (self.mean if p["buoyancy"] == 1 else p["rho_top"])) * p["gy"]
        jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8]
        jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
        return rho, T, dpdT, Fx, Fy, Q, (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho

    def sums(self):
        return self.f.sum(), self.g.sum()

    def step(self):
        p = self.p
        rho, T, dpdT, Fx, Fy, Q, vx, vy = self.fluid()
        div = self.slope(vx)[0] + self.slope(vy)[1]
        Tx, Ty, lapT = self.slope(T)
        rcv = rho * p["cV"]
        source = T * (1 - dpdT / rcv) * div
        if p["model"] != "gong_cheng":
            if p["lambda_const"]:
                flux = p["lam"] * lapT
            else:
                rx, ry, _ = self.slope(rho)
                flux = rcv * p["chi"] * lapT + p["cV"] * p["chi"] * (rx * Tx + ry * Ty)
            source = source + flux / rcv - (1 / p["s_g"][3] - 0.5) / 3 * lapT
        S0 = source
        if p["model"] == "improved":
            S0 = source + 0.5 * (source - (source if self.phi is None else self.phi))
        self.phi = source
        vF, z = vx * Fx + vy * Fy, torch.zeros_like(rho)
        s = torch.tensor(p["s_f"], dtype=torch.float64, device="cuda")[:, None, None]
        m = _apply(self.M, self.f)
        force = torch.stack([z, 6 * vF + Q, -6 * vF - Q, Fx, -Fx, Fy, -Fy, 2 * (vx * Fx - vy * Fy), vx * Fy + vy * Fx])
        f = _apply(self.Mi, m - s * (m - self.flow_eq(rho, vx, vy)) + (1 - 0.5 * s) * force)
        m = _apply(self.M, self.g)
        off = m - self.heat_eq(T, vx, vy)
        if p["model"] == "gong_cheng":
            tau = (p["lam"] * 3 / rcv if p["lambda_const"] else 3 * p["chi"]) + 0.5
            m = m - off / tau
            m[0] += S0
            m[1] -= 2 * S0
            m[2] += S0
        else:
            r = p["s_g"]
            m = m - torch.tensor(r, dtype=torch.float64, device="cuda")[:, None, None] * off
            m[0] += S0
            if p["model"] == "improved":
                m[3] += (1 - 0.5 * r[3]) * r[4] * off[4]
                m[5] += (1 - 0.5 * r[5]) * r[6] * off[6]
        g = _apply(self.Mi, m)
        self.f = self.close_flow(torch.stack([torch.roll(f[a], (E[a][1], E[a][0]), (0, 1)) for a in range(9)]), (Fx, Fy))
        self.g = self.close_heat(torch.stack([torch.roll(g[a], (E[a][1], E[a][0]), (0, 1)) for a in range(9)]))
        self.mean = rho.mean()

    def fields(self):
        rho, T, _, _, _, _, vx, vy = self.fluid()
        return rho, vx, vy, T


def exact(case, seed):
    if case["kind"] == "batch":
        every, out = _instances(case, seed), []
        for k in _done(case):
            w = _Whole(*_setup(*every[k]))
            for _ in range(case["steps"]):
                w.step()
            out.append([x.cpu().numpy() for x in w.fields()])
        return out
    w = _Whole(*_setup(case["setup"], case["nx"], case["ny"], seed, case.get("rates", "unit"),
                       case.get("model", "improved")))
    sums = []
    for _ in range(case["steps"] + (RELAX if case["read"] == "resume" else 0)):
        w.step()
        if case["read"] == "sums":
            sums.append(torch.stack(w.sums()))
    out = dict(zip(("rho", "ux", "uy", "T"), w.fields()))
    if case["read"] == "sums":
        out["sums"] = torch.stack(sums).cpu()
    return out
