"""The workloads whose speed this repository is held to, each a pass through
the public Python entry points (``lesbgk.Solver``, ``lesbgk.Batch``) as a
user's program calls them.

Sizes and set-ups are those of ``inputs.py``, ``serve.py``, ``bench.py`` and
the tests: the paper's channel flows on 4 columns, the force-driven channel,
the lid-driven cavity of the serving mix, the Taylor-Green vortex on every
velocity set and storage, and the batch mix.  Fields differ by seed: waves of
random phase and amplitude plus the 1e-4 density noise of those set-ups (per
row in the flows that run the printed update, which are uniform in x).

``exact`` restates the method in FP64 with torch alone (Sec. 2.2 collision,
Sec. 3.1 scheme, Sec. 3.2 walls), without this repository's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1209_6548_gb300 import inputs as I
from paper_1209_6548_gb300 import lesbgk as L

STORAGE = {"f32": L.F32, "f16": L.F16, "bf16": L.BF16, "f32c": L.F32C}
BYTES = {"f32": 4, "f16": 2, "bf16": 2, "f32c": 6}
SETS = {"d2q16": (4, 2), "d2q36": (6, 2), "d3q64": (4, 3), "d3q216": (6, 3)}
STORED = {"d2q16": 16, "d2q36": 36, "d3q64": 32, "d3q216": 108}  # values per node


def case(kind, nx, ny, steps, **kw):
    """kind: 'solve' (re-initialise, step, read the moments and, where FP32
    populations are stored, the state a checkpoint keeps; a 16-bit state is
    random in its last bits by design), 'check' (a check interval of the
    serving loop: step, the steady-state residual, the moments) or 'host'
    (from host fields to host moments).  flow: 'tgv' (periodic, split scheme),
    'channel' (walls in y, uniform in x, printed update) or 'cavity'."""
    c = {"kind": kind, "set": "d2q16", "storage": "f32", "flow": "tgv", "nx": nx, "ny": ny, "steps": steps,
         "kn": 0.05, "b": -0.5, "visc": 0.5, "gx": 0.0, "wall_u": 0.0, "wall_dT": 0.0, "specular": 0.0, "heat": 0.0}
    c.update(kw)
    return c


def listed():
    return [
        # the paper's Couette flow on 4 x 64: the smallest solve, one of
        # thousands in a parameter study; steps are bound by latency
        case("solve", 4, 64, 64, name="couette_4x64", flow="channel", kn=0.1, wall_u=0.05),
        # combined Couette-Fourier flow at high Mach number on the larger 2D
        # set (Sec. 4), an odd height, long enough to matter
        case("solve", 4, 65, 256, name="couette_fourier_4x65_d2q36", set="d2q36", flow="channel", kn=0.08,
             wall_u=0.2, wall_dT=0.15),
        # the force-driven channel of the tests: a middle size that stays in L2
        case("solve", 512, 1024, 100, name="poiseuille_512x1024", flow="channel", kn=0.2, b=0.0, gx=1e-4),
        # one check interval of a cavity in the serving loop's wide lane
        case("check", 256, 256, 256, name="cavity_256_check", flow="cavity", kn=0.1, wall_u=0.05),
        # the benchmark's vortex: throughput at a size far beyond L2
        case("solve", 4096, 4096, 40, name="tgv_4096_d2q16"),
        # the other velocity sets, one of them on a ragged grid
        case("solve", 2048, 2048, 40, name="tgv_2048_d2q36", set="d2q36"),
        case("solve", 1999, 2053, 40, name="tgv_1999x2053_d3q64", set="d3q64"),
        case("solve", 1024, 1024, 40, name="tgv_1024_d3q216", set="d3q216"),
        # 16-bit storage, the capacity option, at the benchmark's size
        case("solve", 4096, 4096, 40, name="tgv_4096_d2q16_f16", storage="f16"),
        # a whole solve between host buffers, the other 16-bit type, odd sizes
        case("host", 1021, 767, 100, name="host_1021x767_bf16", storage="bf16"),
        # compensated storage, the one that holds every field to 1e-5
        case("solve", 4096, 4096, 20, name="tgv_4096_d2q16_f32c", storage="f32c"),
        # the batch mix: admit 512 uneven channels, step all, read all
        {"name": "batch_mix_512", "kind": "batch", "set": "d2q16", "storage": "f32", "n": 512, "mix": 0,
         "ny_lo": 16, "ny_hi": 1024, "steps": 1024},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["channel", "channel", "wide_channel", "cavity", "tgv", "tgv", "tgv", "host", "batch"])
    kn = round(math.exp(rng.uniform(math.log(0.02), math.log(0.5))), 4)
    b = rng.choice([-0.5, 0.0, 0.5])
    if what == "batch":
        n = log_int(16, 512)
        return {"kind": "batch", "set": rng.choice(["d2q16", "d2q16", "d2q36", "d3q64"]),
                "storage": rng.choice(["f32", "f32", "f16", "bf16"]), "n": n, "mix": rng.randrange(1, 1000),
                "ny_lo": 16, "ny_hi": rng.choice([256, 512, 1024]) if n > 128 else 1024,
                "steps": rng.choice([100, 256, 1000])}
    vset = rng.choice(["d2q16", "d2q16", "d2q36", "d3q64", "d3q216"])
    storage = rng.choice(["f32", "f32", "f16", "bf16"] + (["f32c"] if SETS[vset][0] == 4 else []))
    if what == "channel":
        # 1D flows on few columns, with the options of the walls
        wall = rng.choice(["diffuse", "diffuse", "maxwell", "heated"])
        if wall == "maxwell":
            storage = "f32"
        return case("solve", rng.choice([1, 2, 4, 4, 4, 8, 5, 16]), log_int(16, 1024), rng.choice([16, 64, 256]),
                    set=vset, storage=storage, flow="channel", kn=kn, b=b, visc=rng.choice([0.5, 0.5, 0.75, 1.0]),
                    gx=rng.choice([0.0, 1e-4]), wall_u=rng.choice([0.0, 0.05, 0.2]),
                    wall_dT=rng.choice([0.0, 0.05]), specular=0.3 if wall == "maxwell" else 0.0,
                    heat=0.002 if wall == "heated" else 0.0)
    if what == "wide_channel":
        cap = 2 ** 19 * 16 // STORED[vset]
        nx = log_int(32, 512)
        return case("solve", nx, log_int(33, max(64, min(2048, cap // nx))), 40, set=vset, storage=storage,
                    flow="channel", kn=kn, b=b, gx=1e-4)
    if what == "cavity":
        vset = rng.choice(["d2q16", "d2q16", "d2q36"])
        return case("check", log_int(31, 512), log_int(31, 512), rng.choice([32, 128]), set=vset,
                    storage="f32" if storage == "f32c" else storage, flow="cavity", kn=max(kn, 0.05), b=b, wall_u=0.05)
    cap = 2 ** 24 * 16 // STORED[vset]  # no more values than the largest listed grid
    nx = log_int(61, 4096)
    ny = log_int(61, max(122, min(4096, cap // nx)))
    if what == "host":
        return case("host", min(nx, 2048), min(ny, 1024, cap // min(nx, 2048)), 40, set=vset, storage=storage,
                    kn=kn, b=b)
    return case("solve", nx, ny, 20 if nx * ny > 2 ** 22 else 40, set=vset, storage=storage, kn=kn, b=b)


# ------------------------------------------------------------------ set-up
def problem(c):
    nroots, dim = SETS[c["set"]]
    walls = c["flow"] != "tgv"
    cavity = c["flow"] == "cavity"
    wall_ux = (0.0, c["wall_u"]) if cavity else (-c["wall_u"], c["wall_u"])
    return I.Problem(name=c["flow"], nroots=nroots, dim=dim, nx=c["nx"], ny=c["ny"],
                     bc_y=I.DIFFUSE if walls else I.PERIODIC, bc_x=I.DIFFUSE if cavity else I.PERIODIC,
                     kn=c["kn"], b=c["b"], visc_exp=c["visc"], wall_ux=wall_ux,
                     wall_T=(1.0 - c["wall_dT"], 1.0 + c["wall_dT"]), g=(c["gx"], 0.0),
                     scheme=I.UNSPLIT if c["flow"] == "channel" else I.SPLIT,
                     wall_specular=c["specular"], wall_T_amp=c["heat"],
                     wall_T_freq=math.pi * math.sqrt(2.0) / 8.0 if c["heat"] else 0.0)


def device():
    return torch.device("cuda")


def fields(flow, nx, ny, seed):
    """(4, ny, nx) FP64 rho, u_x, u_y, T: a wave of random phase and
    amplitude, and density noise of 1e-4 (uniform in x for channels)."""
    g = torch.Generator(device=device())
    g.manual_seed(int(seed))
    r = torch.rand(4, generator=g, device=device(), dtype=torch.float64)
    tp = 2.0 * math.pi
    y = torch.arange(ny, device=device(), dtype=torch.float64) / ny
    amp, px, py = 0.04 + 0.02 * r[0], tp * r[1], tp * r[2]
    out = torch.empty((4, ny, nx), device=device(), dtype=torch.float64)
    if flow == "tgv":
        x = torch.arange(nx, device=device(), dtype=torch.float64) / nx
        sx, cx = torch.sin(tp * x + px), torch.cos(tp * x + px)
        sy, cy = torch.sin(tp * y + py), torch.cos(tp * y + py)
        noise = torch.rand((ny, nx), generator=g, device=device(), dtype=torch.float64)
        out[0] = 1.0 + 1e-4 * (2.0 * noise - 1.0)
        out[1] = amp * cy[:, None] * sx[None, :]
        out[2] = -amp * sy[:, None] * cx[None, :]
        out[3] = 1.0 + 0.01 * sy[:, None] * sx[None, :]
        return out
    noise = torch.rand((ny, nx if flow == "cavity" else 1), generator=g, device=device(), dtype=torch.float64)
    out[0] = 1.0 + 1e-4 * (2.0 * noise - 1.0)
    out[1] = (0.2 * amp * torch.sin(tp * y + py))[:, None]
    out[2] = 0.0
    out[3] = (1.0 + 0.005 * torch.cos(tp * y + px))[:, None]
    return out


def batch_problems(c):
    nroots, dim = SETS[c["set"]]
    from dataclasses import replace
    return [replace(p, nroots=nroots, dim=dim)
            for p in I.batch_mix(n=c["n"], seed=c["mix"], ny_lo=c["ny_lo"], ny_hi=c["ny_hi"])]


def params(c, prob):
    p = L.params_from_problem(prob)
    p.storage = STORAGE[c["storage"]]
    return p


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        probs = batch_problems(c)
        ps = [params(c, p) for p in probs]
        h_inits, outs, at = [], [], 0
        flat = torch.empty(sum(9 * p.cells for p in probs), device=device(), dtype=torch.float32)
        every = fields("channel", 1, sum(p.ny for p in probs), seed)[:, :, 0].cpu().numpy()
        row = 0
        for p in probs:
            col = every[:, row:row + p.ny].copy()
            h_inits.append(np.repeat(col[:, :, None], p.nx, axis=2))
            outs.append(flat[at:at + 9 * p.cells].view(9, p.ny, p.nx))
            row += p.ny
            at += 9 * p.cells
        bt = L.Batch(capacity=c["n"], nx=probs[0].nx, pool_bytes=sum(L.batch_slot_bytes(p) for p in ps))
        return {"case": c, "batch": bt, "params": ps, "h_inits": h_inits, "outs": outs, "flat": flat}
    p = params(c, problem(c))
    f = fields(c["flow"], c["nx"], c["ny"], seed)
    if c["kind"] == "host":
        pinned = torch.empty(f.shape, dtype=torch.float64, pin_memory=True)
        pinned.copy_(f)
        return {"case": c, "params": p, "h_init": pinned.numpy(), "keep": pinned}
    state = {"case": c, "solver": L.Solver(p), "fields": f}
    if c["kind"] == "check":
        state["snap"] = torch.empty((4, c["ny"], c["nx"]), dtype=torch.float32, device=device())
    return state


def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        bt = state["batch"]
        slots = bt.add_many(state["params"], state["h_inits"])
        bt.step(c["steps"])
        bt.moments_many(slots, state["outs"])
        for s in slots:
            bt.remove(s)
        return {"moments": state["flat"]}
    if c["kind"] == "host":
        s = L.Solver(state["params"], h_init=state["h_init"])
        s.step(c["steps"])
        m, sums = s.moments_host()
        return {"moments": m, "sums": sums.astype(np.float32)}
    s = state["solver"]
    s.reinit(state["fields"])
    if c["kind"] == "check":
        s.residual(state["snap"], 0)
        s.step(c["steps"])
        r, mass = s.residual(state["snap"], c["steps"], mass=True)
        return {"moments": s.moments(), "residual": r, "mass": mass}
    s.step(c["steps"])
    if BYTES[c["storage"]] >= 4:
        return {"moments": s.moments(), "populations": s.populations()}
    return {"moments": s.moments()}


def work(case):
    """Per step every stored value read and written once, the fields read
    once, the moments written once, and the state where it is returned.  Operations: about 30 per stored value
    (two sweeps with their limiters, the two Hermite transforms, the update)
    and 80 per node for the coefficients."""
    c = case
    cells = sum(p.cells for p in batch_problems(c)) if c["kind"] == "batch" else c["nx"] * c["ny"]
    q = STORED[c["set"]]
    state = 4.0 * q if c["kind"] == "solve" and BYTES[c["storage"]] >= 4 else 0.0
    return {"bytes": cells * (2.0 * q * BYTES[c["storage"]] * c["steps"] + 32 + 36 + state),
            "flops": cells * c["steps"] * (30.0 * q + 80.0)}


# --------------------------------------------------- the method in 64 bits
class Exact:
    """B solves side by side, populations f[B, Z, R, R, Y, X] (z-even half of
    the D = 3 sets).  rows: per solve the number of rows it has (Y the
    largest), only for channels side by side."""

    def __init__(self, nroots, dim, flow, split, steps_dt, dx, dy, kn, b, visc, g, wall_T, wall_u, spec, heat, freq,
                 rows=None):
        dev = device()
        self.t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=dev)
        c, w = np.polynomial.hermite_e.hermegauss(nroots)
        w = w / math.sqrt(2.0 * math.pi)
        self.R, self.D, self.N = nroots, dim, 3 if nroots == 4 else 4
        self.Z = nroots // 2 if dim == 3 else 1
        self.flow, self.split, self.rows = flow, split, rows
        self.c = c
        he = np.stack([np.ones_like(c), c, c ** 2 - 1, c ** 3 - 3 * c, c ** 4 - 6 * c ** 2 + 3])
        ls = (0, 2, 4) if dim == 3 else (0,)
        self.mom = [(m, k, l) for l in ls for m in range(4) for k in range(4) if m + k + l <= 3]
        self.ev = [(m, k, l) for l in ls for m in range(5) for k in range(5) if m + k + l <= self.N]
        hz = he[:, nroots // 2:] if dim == 3 else np.ones((5, 1))
        wz = w[nroots // 2:] if dim == 3 else np.ones(1)
        two = 2.0 if dim == 3 else 1.0
        fac = [1, 1, 2, 6, 24]
        q = self.Z * nroots * nroots
        self.M = self.t(np.stack([np.einsum("z,i,j->zij", two * hz[l], he[m], he[k]).reshape(q)
                                  for m, k, l in self.mom]))
        self.E = self.t(np.stack([np.einsum("z,i,j->zij", wz * hz[l] / fac[l], w * he[m] / fac[m],
                                            w * he[k] / fac[k]).reshape(q) for m, k, l in self.ev], axis=1))
        col = lambda v: self.t(v).reshape(-1, 1, 1)  # [B, 1, 1] against [B, coefficient, node]
        self.dt, self.dx, self.dy = col(steps_dt), col(dx), col(dy)
        self.kn, self.b, self.visc = col(kn), col(b), visc
        self.gx, self.gy = col(g[0]), col(g[1])
        self.wall_T, self.wall_u, self.spec, self.heat, self.freq = wall_T, wall_u, spec, heat, freq
        self.time = 0.0

    def gauss(self, rho, ux, uy, lxx, lxy, lyy, lzz):
        """The coefficients of rho N(u, I + L) for the terms of self.ev."""
        e = {(0, 0): rho}
        for n in range(1, self.N + 1):
            for m in range(n + 1):
                k = n - m
                if m:
                    v = ux * e[m - 1, k]
                    if m >= 2:
                        v = v + (m - 1) * lxx * e[m - 2, k]
                    if k:
                        v = v + k * lxy * e[m - 1, k - 1]
                else:
                    v = uy * e[0, k - 1]
                    if k >= 2:
                        v = v + (k - 1) * lyy * e[0, k - 2]
                e[m, k] = v
        zf = {0: 1.0, 2: lzz, 4: 3.0 * lzz * lzz}
        return [e[m, k] * zf[l] for m, k, l in self.ev]

    def start(self, fld):
        """fld [B, 4, Y, X]."""
        B, _, Y, X = fld.shape
        self.B, self.Y, self.X = B, Y, X
        rho, ux, uy, T = (fld[:, i].reshape(B, Y * X) for i in range(4))
        th, zero = T - 1.0, torch.zeros_like(T)
        co = torch.stack(self.gauss(rho, ux, uy, th, zero, th, th), dim=1)
        f = torch.matmul(self.E, co)
        ny = self.t(self.rows if self.rows is not None else [Y] * B).long()
        j = torch.arange(Y, device=ny.device)
        if self.flow == "tgv":
            self.idx = lambda s: (j + s) % Y
        else:
            self.idx = lambda s: torch.minimum((j + s).clamp(min=0)[None], ny[:, None] - 1)
        self.last = ny - 1
        f = f.reshape(B, self.Z, self.R, self.R, Y, X)
        return self.walls(f)

    def shift_y(self, f, s):
        """f_{j+s} along the rows."""
        if self.flow == "tgv":
            return torch.roll(f, -s, dims=-2)
        idx = self.idx(s)
        if self.B == 1:
            return f.index_select(-2, idx[0])
        return f.gather(-2, idx.reshape(self.B, 1, 1, 1, -1, 1).expand(f.shape))

    def shift_x(self, f, s):
        if self.flow != "cavity":
            return torch.roll(f, -s, dims=-1)
        i = (torch.arange(self.X, device=f.device) + s).clamp(0, self.X - 1)
        return f.index_select(-1, i)

    @staticmethod
    def minmod(a, b):
        return torch.where(a * b > 0.0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))

    def flux(self, f, shift, up, k):
        """(F_{+1/2} - F_{-1/2}) / c of the second-order upwind scheme."""
        s = 1 if up else -1
        f1 = shift(f, -s)  # the upwind neighbour
        d = f - f1
        diff = (f + k * self.minmod(d, shift(f, s) - f)) - (f1 + k * self.minmod(f1 - shift(f, -2 * s), d))
        return diff if up else -diff

    def sweep(self, f, axis):
        """-(c dt/dh) dF along one axis for every population."""
        R, H = self.R, self.R // 2
        dh, shift = (self.dx, self.shift_x) if axis == "x" else (self.dy, self.shift_y)
        nu = (self.t(self.c) * (self.dt / dh))  # [B, 1, R]
        out = torch.empty_like(f)
        for i in range(R):
            n = nu[:, 0, i].reshape(-1, 1, 1, 1, 1)
            k = 0.5 * (1.0 - n.abs())
            if axis == "x":
                out[:, :, i] = -n * self.flux(f[:, :, i], self.sub(shift), i >= H, k)
            else:
                out[:, :, :, i] = -n * self.flux(f[:, :, :, i], self.sub(shift), i >= H, k)
        return out

    @staticmethod
    def sub(shift):
        return lambda v, s: shift(v.unsqueeze(2), s).squeeze(2)

    def moments_of(self, f):
        a = torch.matmul(self.M, f.reshape(self.B, -1, self.Y * self.X))
        a = {key: a[:, i:i + 1] for i, key in enumerate(self.mom)}
        rho = a[0, 0, 0]
        ux, uy = a[1, 0, 0] / rho, a[0, 1, 0] / rho
        mxx, mxy, myy = a[2, 0, 0] - rho * ux * ux, a[1, 1, 0] - rho * ux * uy, a[0, 2, 0] - rho * uy * uy
        mzz = a[0, 0, 2] if self.D == 3 else torch.zeros_like(rho)
        # He_2 moments count from rho: M = P - rho I
        return a, rho, ux, uy, mxx, mxy, myy, mzz

    def step(self, f):
        B, q = self.B, self.Z * self.R * self.R
        a, rho, ux, uy, mxx, mxy, myy, mzz = self.moments_of(f)
        tr = mxx + myy + mzz
        th = tr / (self.D * rho)
        om = self.dt / (self.kn * (1.0 - self.b)) * rho * (1.0 + th) ** (1.0 - self.visc)
        l = lambda m: (1.0 - self.b) * th + self.b * m / rho
        co = self.gauss(rho, ux, uy, l(mxx), self.b * mxy / rho, l(myy), l(mzz))
        for i, (m, k, z) in enumerate(self.ev):
            v = om * co[i]
            if m:
                v = v + m * self.dt * self.gx * a[m - 1, k, z]
            if k:
                v = v + k * self.dt * self.gy * a[m, k - 1, z]
            co[i] = v
        src = torch.matmul(self.E, torch.cat(co, dim=1))
        new = (src + (1.0 - om) * f.reshape(B, q, -1)).reshape(f.shape)
        del src, co, a
        dy = self.sweep(f, "y")
        new += dy
        new += self.sweep(f + dy if self.split else f, "x")
        self.time += float(self.dt[0]) if self.heat else 0.0
        return self.walls(new)

    def wall_eq(self, T, u):
        """S_a(T_w, u_w) [B, Z, R, R] for per-solve T, u."""
        T, u = self.t(T).reshape(-1, 1), self.t(u).reshape(-1, 1)
        one, zero = torch.ones_like(T), torch.zeros_like(T)
        co = torch.stack(self.gauss(one, u, zero, T - 1.0, zero, T - 1.0, T - 1.0), dim=1)
        return torch.matmul(self.E, co).reshape(-1, self.Z, self.R, self.R)

    def walls(self, f):
        if self.flow == "tgv":
            return f
        H, R = self.R // 2, self.R
        cy = self.t(np.abs(self.c))
        bi = torch.arange(self.B, device=f.device)
        dT = self.heat * math.sin(self.freq * self.time)
        cols = slice(1, -1) if self.flow == "cavity" else slice(None)
        old = f.clone() if self.flow == "cavity" else None
        for side in (0, 1):
            at = torch.zeros_like(self.last) if side == 0 else self.last
            node = f[bi, :, :, :, at]  # [B, Z, R, R, X]
            inc, outg = (slice(0, H), slice(H, R)) if side == 0 else (slice(H, R), slice(0, H))
            S = self.wall_eq(np.asarray(self.wall_T[side]) + dT, self.wall_u[side])[..., None]
            num = (cy[inc][:, None] * node[:, :, :, inc]).sum(dim=(1, 2, 3), keepdim=True)
            den = (cy[outg][:, None] * S[:, :, :, outg]).sum(dim=(1, 2, 3), keepdim=True)
            emit = (1.0 - self.spec) * (num / den) * S + self.spec * node.flip(3)
            node[:, :, :, outg] = emit[:, :, :, outg]
            if self.flow == "cavity":  # the corners belong to the side walls' rule
                f[bi, :, :, :, at, 1:-1] = node[..., cols]
            else:
                f[bi, :, :, :, at] = node
        if self.flow == "cavity":
            S = self.wall_eq([1.0], [0.0])[..., None]
            c = self.t(self.c)
            for xs in (0, 1):
                i = 0 if xs == 0 else self.X - 1
                cin = (c < 0) if xs == 0 else (c > 0)
                node = old[..., i].clone()  # [B, Z, R, R, Y]
                kept = cin.double()[:, None, None] * torch.ones(R, 1, device=f.device, dtype=torch.float64)
                cn = c.abs()[:, None, None] * torch.ones(R, 1, device=f.device, dtype=torch.float64)
                kept, cn = kept.repeat(1, 1, self.Y), cn.repeat(1, 1, self.Y)
                outk = 1.0 - kept
                for ys in (0, 1):  # corner nodes keep what arrives towards both walls
                    j = 0 if ys == 0 else self.Y - 1
                    both = cin[:, None] & ((c < 0) if ys == 0 else (c > 0))[None, :]
                    kept[:, :, j] = both.double()
                    cn[:, :, j] = (c[:, None] * (1 if xs == 0 else -1) + c[None, :] * (1 if ys == 0 else -1)).abs()
                    outk[:, :, j] = both.double()  # for a wall at rest: sum over kept of |c.n| S
                num = (kept * cn * node).sum(dim=(1, 2, 3), keepdim=True)
                den = (outk * cn * S).sum(dim=(1, 2, 3), keepdim=True)
                f[..., i] = kept * node + (1.0 - kept) * (num / den) * S
        return f

    def deviations(self, f):
        """f - w per stored population, [B, Z R R, Y, X]."""
        return f.reshape(self.B, -1, self.Y, self.X) - self.E[:, 0].reshape(-1, 1, 1)

    def nine(self, f):
        a, rho, ux, uy, mxx, mxy, myy, mzz = self.moments_of(f)
        tr = mxx + myy + mzz
        hx, hy = a[3, 0, 0] + a[1, 2, 0], a[0, 3, 0] + a[2, 1, 0]
        if self.D == 3:
            hx, hy = hx + a[1, 0, 2], hy + a[0, 1, 2]
        u2 = ux * ux + uy * uy
        qx = 0.5 * (hx - 2.0 * (mxx * ux + mxy * uy) - ux * tr - rho * ux * u2)
        qy = 0.5 * (hy - 2.0 * (mxy * ux + myy * uy) - uy * tr - rho * uy * u2)
        out = [rho, ux, uy, 1.0 + tr / (self.D * rho), mxx - tr / self.D, mxy, myy - tr / self.D, qx, qy]
        return torch.cat(out, dim=1).reshape(self.B, 9, self.Y, self.X)


def time_step(p, tmax=1.0, rmax=1.0):
    """(dt, dx, dy) of a Problem: CFL bound or the relaxation time."""
    wy, wx = p.bc_y == I.DIFFUSE, p.bc_x == I.DIFFUSE
    dx, dy = 1.0 / (p.nx - (1 if wx else 0)) if (wx or not wy) else None, 1.0 / (p.ny - (1 if wy else 0))
    dx = dy if dx is None else dx
    if wy:
        tmax = max(tmax, max(p.wall_T) + abs(p.wall_T_amp))
    cmax = float(np.polynomial.hermite_e.hermegauss(p.nroots)[0][-1])
    tau = p.kn * (1.0 - p.b) * tmax ** (p.visc_exp - 1.0) / rmax
    return min(p.cfl * min(dx, dy) / cmax, tau), dx, dy


def exact(case, seed):
    c = case
    with torch.no_grad():
        if c["kind"] == "batch":
            probs = batch_problems(c)
            Y = max(p.ny for p in probs)
            if len(probs) * Y * STORED[c["set"]] * c["steps"] > 1e10:
                return None  # more than the time allowed
            every = fields("channel", 1, sum(p.ny for p in probs), seed)[:, :, 0]
            fld = torch.zeros((len(probs), 4, Y, 1), dtype=torch.float64, device=device())
            fld[:, 0] = fld[:, 3] = 1.0
            row, sp = 0, []
            for i, p in enumerate(probs):
                col = every[:, row:row + p.ny]
                fld[i, :, :p.ny, 0] = col
                sp.append(time_step(p, float(col[3].max()), float(col[0].max())))
                row += p.ny
            ex = Exact(probs[0].nroots, probs[0].dim, "channel", False, [s[0] for s in sp], [s[1] for s in sp],
                       [s[2] for s in sp], [p.kn for p in probs], [p.b for p in probs], probs[0].visc_exp,
                       ([p.g[0] for p in probs], [p.g[1] for p in probs]),
                       [[p.wall_T[s] for p in probs] for s in (0, 1)],
                       [[p.wall_ux[s] for p in probs] for s in (0, 1)], 0.0, 0.0, 0.0, rows=[p.ny for p in probs])
            f = ex.start(fld)
            for _ in range(c["steps"]):
                f = ex.step(f)
            m = ex.nine(f)
            return {"moments": torch.cat([m[i, :, :p.ny].expand(9, p.ny, p.nx).reshape(-1)
                                          for i, p in enumerate(probs)])}
        cells = c["nx"] * c["ny"]
        if cells * STORED[c["set"]] * c["steps"] > 1.2e10 or c["steps"] > 1000:
            return None
        p = problem(c)
        fld = fields(c["flow"], c["nx"], c["ny"], seed)
        if c["kind"] == "host":
            dt, dx, dy = time_step(p, float(fld[3].max()), float(fld[0].max()))
        else:
            dt, dx, dy = time_step(p)
        ex = Exact(p.nroots, p.dim, c["flow"], p.scheme == I.SPLIT, [dt], [dx], [dy], [p.kn], [p.b], p.visc_exp,
                   ([p.g[0]], [p.g[1]]), [[p.wall_T[0]], [p.wall_T[1]]], [[p.wall_ux[0]], [p.wall_ux[1]]],
                   p.wall_specular, p.wall_T_amp, p.wall_T_freq)
        f = ex.start(fld[None])
        for _ in range(c["steps"]):
            f = ex.step(f)
        m = ex.nine(f)[0]
        if c["kind"] == "solve" and BYTES[c["storage"]] >= 4:
            return {"moments": m, "populations": ex.deviations(f)[0]}
        if c["kind"] == "solve":
            return {"moments": m}
        rho = m[0].sum()
        if c["kind"] == "check":
            return {"moments": m, "residual": None, "mass": float(rho)}
        energy = (m[0] * (0.5 * (m[1] ** 2 + m[2] ** 2) + 0.5 * p.dim * m[3])).sum()
        sums = torch.stack([rho, (m[0] * m[1]).sum(), (m[0] * m[2]).sum(), energy])
        return {"moments": m.cpu().numpy(), "sums": sums.cpu().numpy()}
