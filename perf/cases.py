"""The workloads whose speed matters to a user of the library, as cases that can be timed.

Every case is a stretch of a simulation as its user runs it: `steps` Runge-Kutta steps through
the public API and the read-out that such a run makes of them (moment fields on the device or
the host, diagnostics, the structure factor). The state lives in the handle and moves on from
pass to pass. Sizes and parameter sets are those of the repository's own runs (the parity
tests, the precision table, the coexistence, droplet and energy-drift protocols, the benchmark).

A float32 form's fields are handed on as float32 (what its state holds; a user keeps snapshots
of it in that type), a float64 form's as float64. The four moment fields come as one array.
"""
import math

import numpy as np
import torch

import paper_1403_3746_gb300 as lbm

PRECISION = {"fp64": lbm.LBM_FP64, "mixed": lbm.LBM_MIXED, "rho64": lbm.LBM_MIXED_RHO64}
# parameter sets: phase separation (the library's defaults), flat-interface coexistence, droplet
PHASE = dict(tau=1e-4, dt=1e-4, dx=1.0 / 256.0, K=5e-6, q=-0.004)
COEXISTENCE = dict(tau=1e-4, dt=5e-5, dx=0.02, K=1e-5, q=-0.004)
DROPLET = dict(tau=5e-4, dt=1e-4, dx=0.01, K=1e-5, q=-0.05)
SETS = {"phase": PHASE, "coexistence": COEXISTENCE, "droplet": DROPLET}


def _single(name, precision, nx, ny, start, T, steps, params="phase", iso=False, filtered=False, read="device"):
    """One simulation. start: slab, droplet (radius a quarter of the shorter side), layers (the
    sharp-edged coexistence layout), rectangle or spinodal. read: device (moment fields into
    device tensors), host (moment fields as numpy arrays), protocol (host fields and the
    diagnostics), monitor (the diagnostics of every step, each read while the next step runs,
    then device fields), growth (host fields, diagnostics and the structure factor), state (host
    fields and the 16 distributions)."""
    c = dict(kind="single", precision=precision, nx=nx, ny=ny, start=start, T=T, steps=steps, params=params, iso=iso,
             filtered=filtered, read=read)
    return dict(c, name=name) if name else c


def _batch(name, precision, smallest, levels, count, start, T, steps):
    """`count` instances of each of `levels` square sizes (smallest, 2 smallest, ...), one temperature each from T
    on, advanced together; every instance's fields are read to the host at the end."""
    c = dict(kind="batch", precision=precision, smallest=smallest, levels=levels, count=count, start=start, T=T,
             steps=steps)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain method on the smallest parity workload: a liquid slab with noise, where
        # launches and the few rows count; the distributions are read as the parity check does
        _single("slab-64-fp64", "fp64", 64, 64, "slab", 0.9, 20, read="state"),
        # quasi-one-dimensional coexistence runs: two rows, read to the host between checks
        _single("coexistence-512x2-mixed", "mixed", 512, 2, "layers", 0.9975, 100, params="coexistence", read="host"),
        # the plain method's quench of the parity tests
        _single("quench-256-fp64", "fp64", 256, 256, "spinodal", 0.9, 20),
        # the precision table's droplets: five instances of 128 x 128 as one batch
        _batch("droplets-5x128-mixed", "mixed", 128, 1, 5, "droplet", 0.9, 50),
        # droplet deformation at fixed temperature, sampled with host fields and diagnostics
        _single("rectangle-256-mixed-iso", "mixed", 256, 256, "rectangle", 0.95, 25, params="droplet", iso=True,
                read="protocol"),
        # energy-drift quench with the solution filter, with its growth measures
        _single("filtered-128x256-fp64", "fp64", 128, 256, "spinodal", 0.9, 10, filtered=True, read="growth"),
        # the benchmark's droplet
        _single("droplet-1024-mixed", "mixed", 1024, 1024, "droplet", 0.85, 10),
        # a wide box watched step by step
        _single("monitor-2048x512-mixed", "mixed", 2048, 512, "spinodal", 0.9, 10, read="monitor"),
        # the benchmark's droplet by the plain method
        _single("droplet-1024-fp64", "fp64", 1024, 1024, "droplet", 0.85, 2),
        # the same with the density chain in float64
        _single("droplet-1024-rho64", "rho64", 1024, 1024, "droplet", 0.85, 4),
        # ensemble of quenches of uneven sizes and temperatures
        _batch("quenches-8x128-256-512-mixed", "mixed", 128, 3, 8, "spinodal", 0.8, 60),
        # the large run
        _single("quench-4096-mixed", "mixed", 4096, 4096, "spinodal", 0.9, 4),
    ]


def draw(rng):
    """A case of the same kinds: sides are powers of two (the library takes no others) over the listed range, in
    any aspect ratio the node budget allows."""
    T = round(rng.uniform(0.86, 0.95), 4)
    if rng.random() < 0.2:
        precision = rng.choice(["mixed", "mixed", "fp64"])
        levels = rng.randint(1, 3 if precision == "mixed" else 2)
        return _batch(None, precision, 128 if precision == "mixed" else 64, levels, rng.randint(2, 6),
                      rng.choice(["spinodal", "droplet"]), round(rng.uniform(0.82, 0.9), 4), rng.randint(5, 30))
    precision = rng.choice(["fp64", "fp64", "mixed", "mixed", "mixed", "rho64"])
    top = {"fp64": 20, "mixed": 22, "rho64": 20}[precision]  # log2 of the nodes
    total = rng.randint(10, top)
    lx = rng.randint(max(4, total - 12), min(11 if precision == "rho64" else 12, total - 1))
    nx, ny = 1 << lx, 1 << (total - lx)
    most = max(2, min(40, (1 << (21 if precision == "fp64" else 23)) >> total))
    read = rng.choice(["device", "device", "host", "protocol", "monitor", "growth"])
    if precision != "fp64" and read == "growth":
        read = "device"
    if total <= 14 and rng.random() < 0.3:
        read = "state"
    small = min(nx, ny) < 32
    start = rng.choice(["slab", "spinodal"]) if small else rng.choice(["slab", "droplet", "spinodal"])
    return _single(None, precision, nx, ny, start, T, rng.randint(max(1, most // 4), most),
                   iso=rng.random() < 0.15, filtered=rng.random() < 0.15, read=read)


# ---- inputs -----------------------------------------------------------------------------


def _fields(start, nx, ny, T, seed, amplitude=0.01):
    """(rho, u_x, u_y, T) as CUDA float64 tensors (ny, nx): a phase profile between the coexisting densities, with
    seeded noise on the density, at rest."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    noise = 2.0 * torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64) - 1.0
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    if start == "spinodal":
        rho = 1.0 + amplitude * noise
    else:
        if start == "layers":
            hi, lo = 1.045, 0.955
            part = ((x >= nx // 4) & (x < 3 * nx // 4)).double()
        elif start == "rectangle":
            hi, lo = 1.462, 0.579
            cx, cy = nx / 2.0 - 0.5, ny / 2.0 - 0.5
            part = (0.5 * (1 + torch.tanh(nx * 0.2305 - (x - cx).abs()))) * (0.5 * (1 + torch.tanh(ny * 0.0273 - (y - cy).abs())))
        else:
            hi, lo = _coexisting(T)
            if start == "slab":
                part = 0.5 * (1 + torch.tanh((nx / 4.0 - (x - nx / 2.0).abs()) / 2))
            else:
                r = torch.sqrt((x - nx / 2.0) ** 2 + (y - ny / 2.0) ** 2)
                part = 0.5 * (1 + torch.tanh((min(nx, ny) / 4.0 - r) / 2))
        rho = lo + (hi - lo) * part + 1e-4 * noise
    rho = rho.expand(ny, nx).contiguous()
    z = torch.zeros_like(rho)
    return rho, z, z.clone(), torch.full_like(rho, float(T))


def _coexisting(T):
    """Liquid and vapour densities of the van der Waals fluid: equal pressure and chemical potential, by Newton's
    method from the expansion about the critical point."""
    def p(r):
        return 3 * r * T / (3 - r) - 1.125 * r * r

    def dp(r):
        return 9 * T / (3 - r) ** 2 - 2.25 * r

    def mu(r):
        return T * math.log(r / (3 - r)) + 3 * T / (3 - r) - 2.25 * r

    s = 2 * math.sqrt(1 - T)
    a, b = 1 + s + 0.4 * (1 - T), max(0.05, 1 - s + 0.4 * (1 - T))
    for _ in range(200):
        f, h = p(a) - p(b), mu(a) - mu(b)
        fa, fb, ha, hb = dp(a), -dp(b), dp(a) / a, -dp(b) / b
        det = fa * hb - fb * ha
        da, db = (f * hb - fb * h) / det, (fa * h - f * ha) / det
        k = min(1.0, 0.2 * min(b, 3 - a) / max(abs(da), abs(db), 1e-300))
        a, b = a - k * da, b - k * db
        if abs(da) + abs(db) < 1e-14:
            break
    return a, b


def _params(case):
    s = SETS[case.get("params", "phase")]
    return lbm.default_params(precision=PRECISION[case["precision"]], tau=s["tau"], dt=s["dt"], dx=s["dx"], dy=s["dx"],
                              K=s["K"], q=s["q"], flags=lbm.LBM_FLAG_ISOTHERMAL if case.get("iso") else 0,
                              T_iso=float(case["T"]) if case.get("iso") else 0.0,
                              filter_alpha=36.0 if case.get("filtered") else 0.0)


def _instances(case, seed):
    """(size, temperature, seed) of a batch's instances, size by size."""
    out = []
    for level in range(case["levels"]):
        for k in range(case["count"]):
            i = level * case["count"] + k
            spread = 0.06 * i / max(1, case["levels"] * case["count"] - 1)
            out.append((case["smallest"] << level, case["T"] + spread, int(seed) * 4096 + i))
    return out


def _bins(case):
    return max(case["nx"], case["ny"]) // 2


# ---- the passes -------------------------------------------------------------------------


def prepare(case, seed):
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    if case["kind"] == "batch":
        inst = _instances(case, seed)
        sim = lbm.Batch([(n, n) for n, _, _ in inst], _params(case))
        for k, (n, T, s) in enumerate(inst):
            sim.init(k, *[a.cpu().numpy() for a in _fields(case["start"], n, n, T, s)])
        # pinned host arrays for the fields of every instance, one block per size
        blocks = [torch.empty((case["count"], 4, case["smallest"] << v, case["smallest"] << v), dtype=torch.float64,
                              pin_memory=True) for v in range(case["levels"])]
        outs = [[b[k, j].numpy() for j in range(4)] for b in blocks for k in range(case["count"])]
        return dict(case=case, sim=sim, blocks=blocks, outs=outs, dtype=dtype)
    sim = lbm.Simulation(case["nx"], case["ny"], _params(case))
    fields = _fields(case["start"], case["nx"], case["ny"], case["T"], seed)
    sim.init(*fields)
    torch.cuda.synchronize()
    return dict(case=case, sim=sim, m=torch.empty((4, case["ny"], case["nx"]), dtype=torch.float64, device="cuda"),
                dtype=dtype)


def _numbers(d, dtype):
    return torch.tensor([d["mass"], d["px"], d["py"], d["energy"], d["umax"]], dtype=torch.float64).to(dtype)


def run(state):
    case, sim, dtype = state["case"], state["sim"], state["dtype"]
    if case["kind"] == "batch":
        sim.step(case["steps"])
        for k, out in enumerate(state["outs"]):
            sim.moments(k, out=out)
        return [b.to(dtype, copy=True) for b in state["blocks"]]
    read, watched = case["read"], []
    if read == "monitor":
        for k in range(case["steps"]):
            sim.step(1)
            sim.diagnostics_begin()
            if k:
                watched.append(_numbers(sim.diagnostics_end(), dtype))
        watched.append(_numbers(sim.diagnostics_end(), dtype))
    else:
        sim.step(case["steps"])
    if read in ("device", "monitor"):
        m = state["m"]
        sim.moments_device(m[0], m[1], m[2], m[3])
        out = {"fields": m.to(dtype)}
    else:
        out = {"fields": torch.from_numpy(np.stack(sim.moments())).to(dtype)}
    if watched:
        out["watched"] = torch.stack(watched)
    if read in ("protocol", "growth"):
        out["numbers"] = _numbers(sim.diagnostics(), dtype)
    if read == "state":
        out["f"] = torch.from_numpy(sim.get_f()).to(dtype)
    if read == "growth":
        out["S"] = torch.from_numpy(sim.structure_factor(_bins(case))[0]).to(dtype)
    return out


def work(case):
    """Per step every distribution is read once and written once in the type it is stored in; a read-out writes
    four float64 fields, or those and the distributions. Operations of a step: the line transforms (a real line's derivative costs 5 log2 n per
    point; two stages of 20.5 derivatives along each axis, a forward transform that serves two counted once) and
    about 1000 per node and stage of local arithmetic."""
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "batch":
        grids = [(case["smallest"] << v,) * 2 for v in range(case["levels"]) for _ in range(case["count"])]
    else:
        grids = [(case["nx"], case["ny"])]
    nbytes = flops = 0.0
    for nx, ny in grids:
        nodes = nx * ny
        logs = math.log2(nx) + math.log2(ny)
        nbytes += nodes * (case["steps"] * 2 * 16 * size + (20 if case.get("read") == "state" else 4) * 8)
        per = 2 * (20.5 * 5 * logs + 1000) + (16 * 5 * logs if case.get("filtered") else 0)
        flops += nodes * case["steps"] * per
    return {"bytes": nbytes, "flops": flops}


# ---- the same in plain float64 torch ----------------------------------------------------

_SERIES = [1.0, 1.0 / 6.0, 3.0 / 40.0, 5.0 / 112.0, 35.0 / 1152.0, 63.0 / 2816.0, 231.0 / 13312.0, 143.0 / 10240.0]


class _Plain:
    """The scheme in float64 by library FFTs: fields (..., ny, nx), all instances of one size at once."""

    def __init__(self, case, nx, ny):
        s = SETS[case.get("params", "phase")]
        self.tau, self.dt, self.K, self.q, self.dx = s["tau"], s["dt"], s["K"], s["q"], s["dx"]
        self.T_iso = float(case["T"]) if case.get("iso") else None
        self.nx, self.ny = nx, ny
        v = [(1, 0), (0, 1), (-1, 0), (0, -1), (6, 0), (0, 6), (-6, 0), (0, -6),
             (1, 1), (-1, 1), (-1, -1), (1, -1), (1.5, 1.5), (-1.5, 1.5), (-1.5, -1.5), (1.5, -1.5)]
        v = torch.tensor(v, dtype=torch.float64, device="cuda")
        self.vx, self.vy = v[:, 0], v[:, 1]
        x, y = self.vx, self.vy
        p = x * x + y * y
        p = p + torch.tensor([6.25] * 4 + [0.0] * 12, dtype=torch.float64, device="cuda")
        self.psi = p
        M = torch.stack([x ** 0, x, y, p, x * x, x * y, y * y, p * x, p * y, x ** 3, x * x * y, x * y * y, y ** 3,
                         p * x * x, p * x * y, p * y * y])
        self.Minv = torch.from_numpy(np.linalg.inv(M.cpu().numpy())).cuda()
        self.kx, self.ky = self._multiplier(nx), self._multiplier(ny)
        self.filt = None
        if case.get("filtered"):
            wx, wy = (torch.exp(-36.0 * (torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64) * 2) ** 36)
                      for n in (nx, ny))
            self.filt = (wx, wy)

    def _multiplier(self, n):
        m = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
        phi = torch.sin(math.pi * m / n)
        k = sum(c * phi ** (2 * j + 1) for j, c in enumerate(_SERIES)) * (2.0 / self.dx)
        k[-1] = 0.0
        return k

    def d(self, h, axis, order=1):
        n, k = (self.nx, self.kx) if axis == "x" else (self.ny, self.ky[:, None])
        dim = -1 if axis == "x" else -2
        mult = 1j * k if order == 1 else -(k * k)
        return torch.fft.irfft(torch.fft.rfft(h, dim=dim) * mult, n=n, dim=dim)

    def equilibrium(self, rho, ux, uy, T):
        uu = ux * ux + uy * uy
        e, g = 4 * T + uu, 6 * T + uu
        m = [torch.ones_like(rho), ux, uy, 2 * T + uu, T + ux * ux, ux * uy, T + uy * uy, ux * e, uy * e,
             3 * T * ux + ux ** 3, uy * (T + ux * ux), ux * (T + uy * uy), 3 * T * uy + uy ** 3,
             T * e + g * ux * ux, g * ux * uy, T * e + g * uy * uy]
        return torch.einsum("ij,j...->i...", self.Minv, torch.stack([rho * a for a in m]))

    def moments(self, f):
        rho = f.sum(0)
        ux, uy, E = (torch.einsum("i,i...->...", w, f) / rho for w in (self.vx, self.vy, self.psi))
        T = (E - ux * ux - uy * uy) / 2
        return rho, ux, uy, (T if self.T_iso is None else torch.full_like(T, self.T_iso))

    def rhs(self, f):
        rho, ux, uy, T = self.moments(f)
        feq = self.equilibrium(rho, ux, uy, T)
        d, K = self.d, self.K
        rx, ry, Tx, Ty = d(rho, "x"), d(rho, "y"), d(T, "x"), d(T, "y")
        lap = d(rho, "x", 2) + d(rho, "y", 2)
        uxx, uxy, uyx, uyy = d(ux, "x"), d(ux, "y"), d(uy, "x"), d(uy, "y")
        div = uxx + uyy
        P = 3 * rho * T / (3 - rho) - 1.125 * rho * rho
        g2 = rx * rx + ry * ry
        iso = K * (rho * lap + 0.5 * g2) - rho * K / T * (rx * Tx + ry * Ty)
        Lxx, Lxy, Lyy = K * rx * rx - iso, K * rx * ry, K * ry * ry - iso
        Pn = P - rho * T
        Bx = (d(Pn + Lxx, "x") + d(Lxy, "y")) / (rho * T)
        By = (d(Lxy, "x") + d(Pn + Lyy, "y")) / (rho * T)
        Cq = (d(self.q * rho * T * Tx, "x") + d(self.q * rho * T * Ty, "y")) / (rho * T * T)
        C = Pn * div + Lxx * uxx + Lxy * (uyx + uxy) + Lyy * uyy + 1.125 * rho * rho * div
        C = C - K * (0.5 * g2 * div + rho * (rx * d(div, "x") + ry * d(div, "y"))
                     + rx * (uxx * rx + uyx * ry) + ry * (uxy * rx + uyy * ry))
        CC = C / (2 * rho * T * T) + Cq
        out = []
        for i in range(16):
            vx, vy = float(self.vx[i]), float(self.vy[i])
            cx, cy = vx - ux, vy - uy
            r = (feq[i] - f[i]) / self.tau - (-2 * CC * T + Bx * cx + By * cy + CC * (cx * cx + cy * cy)) * feq[i]
            if vx:
                r -= vx * d(f[i], "x")
            if vy:
                r -= vy * d(f[i], "y")
            out.append(r)
        return torch.stack(out)

    def step(self, f):
        f = f + self.dt * self.rhs(f + 0.5 * self.dt * self.rhs(f))
        if self.filt is not None:
            f = torch.fft.irfft(torch.fft.rfft(f) * self.filt[0], n=self.nx)
            f = torch.fft.irfft(torch.fft.rfft(f, dim=-2) * self.filt[1][:, None], n=self.ny, dim=-2)
        return f

    def numbers(self, f):
        rho, ux, uy, T = self.moments(f)
        rx, ry = self.d(rho, "x"), self.d(rho, "y")
        uu = ux * ux + uy * uy
        e = rho * T - 1.125 * rho * rho + 0.5 * self.K * (rx * rx + ry * ry) + 0.5 * rho * uu
        cell = self.dx * self.dx
        return torch.stack([rho.sum() * cell, (rho * ux).sum() * cell, (rho * uy).sum() * cell, e.sum() * cell,
                            uu.max().sqrt()]).cpu()

    def structure(self, rho, nbins):
        n = max(self.nx, self.ny)
        power = torch.fft.fft2(rho).abs() ** 2 / (self.nx * self.ny)
        mx = torch.fft.fftfreq(self.nx, device="cuda", dtype=torch.float64) * n
        my = torch.fft.fftfreq(self.ny, device="cuda", dtype=torch.float64) * n
        shell = torch.sqrt(mx[None, :] ** 2 + my[:, None] ** 2).round().long().reshape(-1)
        keep = shell < nbins
        total = torch.zeros(nbins, dtype=torch.float64, device="cuda").index_add_(0, shell[keep], power.reshape(-1)[keep])
        count = torch.bincount(shell[keep], minlength=nbins)
        S = total / count.clamp(min=1)
        S[0] = 0.0
        return S.cpu()


def exact(case, seed):
    if case["kind"] == "batch":
        inst, out = _instances(case, seed), []
        for level in range(case["levels"]):
            n = case["smallest"] << level
            mine = [i for i in inst if i[0] == n]
            p = _Plain(case, n, n)
            fields = [torch.stack(a) for a in zip(*[_fields(case["start"], n, n, T, s) for _, T, s in mine])]
            f = p.equilibrium(*fields)
            for _ in range(case["steps"]):
                f = p.step(f)
            out.append(torch.stack(p.moments(f), dim=1).cpu())
        return out
    p = _Plain(case, case["nx"], case["ny"])
    fields = list(_fields(case["start"], case["nx"], case["ny"], case["T"], seed))
    if case["iso"]:
        fields[3] = torch.full_like(fields[3], float(case["T"]))
    f, watched = p.equilibrium(*fields), []
    del fields
    for _ in range(case["steps"]):
        f = p.step(f)
        if case["read"] == "monitor":
            watched.append(p.numbers(f))
    out = {"fields": torch.stack(p.moments(f))}
    if case["read"] not in ("device", "monitor"):
        out["fields"] = out["fields"].cpu()
    if watched:
        out["watched"] = torch.stack(watched)
    if case["read"] in ("protocol", "growth"):
        out["numbers"] = p.numbers(f)
    if case["read"] == "state":
        out["f"] = f.cpu()
    if case["read"] == "growth":
        out["S"] = p.structure(out["fields"][0].cuda(), _bins(case))
    return out
