"""Performance cases of the library: what users have it do, through its public entry points.

Every case is a job as a user's program runs it: initial fields in, a number of time steps with
the FP64 diagnostics read at the program's own interval, the macroscopic fields out (`kind` "run":
one simulation; "batch": a ragged batch of members advancing together; "serve": requests served
by the continuous-batching server).  A job always starts from its initial fields, so it can be
run any number of times on the same handles.
"""
from __future__ import annotations

import math
import random
import types

import numpy as np
import torch

import paper_1110_5004_gb300 as lbm
from paper_1110_5004_gb300 import serve

STORAGE = {"fp32": lbm.LBM_FP32, "fp16": lbm.LBM_FP16_DEV, "bf16": lbm.LBM_BF16_DEV}
FIELDS = ("phi", "rho", "ux", "uy", "p")
DIAG = ("sum_phi", "liquid_area", "centroid_x", "centroid_y", "vel_x", "vel_y", "spread_radius", "max_u",
        "p_liquid", "p_gas")

# One simulation, with the defaults that most users leave alone: a drop between two walls.
DEFAULTS = dict(kind="run", setup="falling", storage="fp32", steps=100, diag_every=0, remove_Fa=0, wall_x=False,
                wall_y=True, sigma=0.005, W=4.0, nu_A=0.025, nu_B=0.025, rho_A=1.0, rho_B=0.1, gravity=1e-6,
                tau_f=0.8, ch_conservative=0, fs_form=0, s_form=0, f_form=0, host=False, force=False)


def _case(name, nx, ny, **kw):
    return dict(DEFAULTS, name=name, nx=nx, ny=ny, **kw)


def listed():
    return [
        # The smallest call: a program that single-steps a small box and looks at the diagnostics
        # after every step (interactive use, tests, parameter checks).
        _case("look_64", 64, 64, setup="static", wall_y=False, gravity=0.0, steps=4, diag_every=1),
        # The static droplet of the Laplace-law check (128 x 128 periodic, density ratio 10).
        _case("static_128", 128, 128, setup="static", wall_y=False, gravity=0.0, sigma=0.01, nu_A=0.1, nu_B=0.1,
              steps=200),
        # The paper's falling droplet at its own size (odd width, corrected scheme), logged.
        _case("paper_drop_150x450", 150, 450, rho_A=5.0, rho_B=1.0, sigma=0.002, W=3.0, gravity=8.3e-6, remove_Fa=1,
              steps=100, diag_every=50),
        # Falling droplet, 256 x 1024, density ratio 50, centroid velocity logged every 50 steps.
        _case("falling_256x1024", 256, 1024, rho_B=0.02, nu_B=0.125, steps=100, diag_every=50),
        # A closed box (walls on all four sides) of odd size, the other forms of the surface force
        # and of the Cahn-Hilliard equation, fields in and out of pinned host memory in one block.
        _case("box_601x437", 601, 437, wall_x=True, fs_form=1, ch_conservative=1, remove_Fa=1, host=True, steps=40),
        # Droplet splashing on a film on the headline workload's grid, FP32.  (Density ratio 10, the
        # paper's: at the headline's 1000 the scheme itself leaves the finite range within 20 steps.)
        _case("splash_2048x512", 2048, 512, setup="splash", sigma=1e-4, W=5.0, nu_A=0.016, nu_B=0.016, gravity=0.0,
              steps=40),
        # The same splash stored in FP16, corrected scheme.
        _case("splash_2048x512_fp16", 2048, 512, setup="splash", storage="fp16", sigma=1e-4, W=5.0, nu_A=0.016,
              nu_B=0.016, gravity=0.0, remove_Fa=1, steps=40),
        # The mass defect taken from the stored density and flux, odd sizes, and the interfacial
        # force as a field (the paper's Fig. 3).
        _case("direct_1000x701", 1000, 701, remove_Fa=1, s_form=1, force=True, steps=30),
        # A grid far beyond the L2 cache (2.4 GB of populations), periodic.
        _case("large_4096", 4096, 4096, setup="static", wall_y=False, gravity=0.0, sigma=0.01, nu_A=0.1, nu_B=0.1,
              steps=10),
        # Ragged batch of static and falling droplets, grids of 64^2 to 512^2, FP32 and BF16.
        dict(kind="batch", name="batch_fp32", members=48, steps=48, storage="fp32", max_side=512),
        dict(kind="batch", name="batch_bf16", members=48, steps=48, storage="bf16", max_side=512),
        # Falling-drop requests of 128 x 256 to 1024 x 4096 cells served by continuous batching,
        # initial fields from and results to host memory.
        dict(kind="serve", name="serve_6", requests=6, steps=60, storage="fp32", max_side=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """A case of the listed ranges: grids of 64 x 64 to 4096 x 4096 cells of any aspect up to 4,
    mostly not multiples of anything; batches of 4 to 48 members; 1 to 6 served requests."""
    kind = rng.choices(("run", "batch", "serve"), (8, 2, 1))[0]
    storage = rng.choices(("fp32", "fp16", "bf16"), (5, 2, 2))[0]
    if kind == "batch":
        return dict(kind="batch", members=_log_int(rng, 4, 48), steps=_log_int(rng, 5, 48), storage=storage,
                    max_side=512)
    if kind == "serve":
        return dict(kind="serve", requests=rng.randint(1, 6), steps=_log_int(rng, 10, 60), storage=storage,
                    max_side=4096)
    cells = math.exp(rng.uniform(math.log(64 * 64), math.log(3000 * 3000)))
    aspect = math.exp(rng.uniform(-math.log(4.0), math.log(4.0)))
    nx = max(32, min(4096, int(round(math.sqrt(cells * aspect)))))
    ny = max(32, min(4096, int(round(cells / nx))))
    if rng.random() < 0.4:
        nx = max(32, nx // 32 * 32)
    setup = rng.choice(("static", "falling", "splash"))
    wall_y = setup != "static" or rng.random() < 0.3
    # within the range in which the scheme stays stable over the job at these interface widths
    ratio = math.exp(rng.uniform(math.log(3.0), math.log(30.0)))
    nu_A = rng.uniform(0.02, 0.1)
    # about the work of the listed jobs of the same size
    steps = max(4, min(rng.randint(20, 200), int(1.2e8 / (nx * ny))))
    forms = rng.random() < 0.3
    f_form = int(forms and storage == "fp32" and rng.random() < 0.3)
    return dict(DEFAULTS, nx=nx, ny=ny, setup=setup, storage=storage, steps=steps,
                diag_every=rng.choice((0, 0, max(1, steps // 2), 25)), remove_Fa=rng.randint(0, 1),
                wall_x=rng.random() < 0.2, wall_y=wall_y, sigma=rng.uniform(1e-3, 1e-2),
                W=rng.choice((3.0, 4.0, 5.0)), nu_A=nu_A,
                nu_B=nu_A * (1.0 if setup == "splash" else rng.choice((1.0, 1.0, 5.0))), rho_B=1.0 / ratio,
                gravity=1e-6 if setup == "falling" else 0.0, ch_conservative=int(forms and rng.random() < 0.5),
                fs_form=int(forms and rng.random() < 0.5), s_form=int(forms and rng.random() < 0.4), f_form=f_form,
                host=rng.random() < 0.25, force=rng.random() < 0.15)


# ------------------------------------------------------------------------------ inputs

def _members(case, seed):
    """The single simulations of a batch or serving case, each as a run case."""
    rng = random.Random(1000003 * seed + 17 * case.get("members", case.get("requests", 0)))
    out = []
    for i in range(case["members"] if case["kind"] == "batch" else case["requests"]):
        if case["kind"] == "batch":
            # the sizes depend on the case alone: another seed brings other fields, not other work
            size = random.Random(4242 + 97 * i)
            area = size.uniform(64 * 64, case["max_side"] ** 2)
            nx = max(32, int(round(math.sqrt(area * size.uniform(1.0, 4.0)) / 32.0)) * 32)
            if i % 4 == 3:
                nx -= size.randint(1, 31)
            ny = max(64, int(round(area / nx)))
            falling = size.random() < 0.5
            m = dict(DEFAULTS, setup="falling" if falling else "static", wall_y=falling,
                     gravity=1e-6 if falling else 0.0, sigma=rng.uniform(1e-3, 1e-2), nu_A=0.1, nu_B=0.1,
                     rho_B=1.0 / rng.choice((5.0, 10.0, 20.0)), remove_Fa=i % 2, steps=case["steps"])
        else:
            size = random.Random(977 + 89 * i)
            nx = size.randint(4, 32) * 32
            ny = min(max(nx * size.randint(2, 4), 256), case["max_side"])
            m = dict(DEFAULTS, rho_B=1.0 / math.exp(rng.uniform(math.log(10.0), math.log(50.0))), nu_B=0.1,
                     steps=case["steps"] + 20 * (i % 3))
        m.update(nx=nx, ny=ny, storage=case["storage"])
        out.append(m)
    return out


def _physical(case):
    """The physical parameters as lbm.params_from_physical takes them."""
    wall = lambda w: lbm.LBM_WALL if w else lbm.LBM_PERIODIC
    keys = ("sigma", "W", "nu_A", "nu_B", "rho_A", "rho_B", "gravity", "tau_f", "remove_Fa", "ch_conservative",
            "fs_form", "s_form", "f_form")
    return types.SimpleNamespace(phi_star=1.0, theta_M=0.1, bc_x=wall(case["wall_x"]), bc_y=wall(case["wall_y"]),
                                 **{k: case[k] for k in keys})


def _fields(case, seed, device):
    """phi0, ux0, uy0, p0 as one (4, ny, nx) float32 tensor: a drop (for "splash" above a film and
    moving down at it) in a weak smooth stream, place, size and stream drawn from the seed."""
    nx, ny = case["nx"], case["ny"]
    rng = random.Random(7919 * seed + nx + 31 * ny)
    y = torch.arange(ny, dtype=torch.float64, device=device)[:, None]
    x = torch.arange(nx, dtype=torch.float64, device=device)[None, :]
    side, W = min(nx, ny), case["W"]
    R = side * rng.uniform(0.15, 0.22)
    xc = nx * rng.uniform(0.4, 0.6)
    film = 0.1 * side if case["setup"] == "splash" else 0.0
    yc = {"static": ny * rng.uniform(0.4, 0.6), "falling": ny * rng.uniform(0.6, 0.7),
          "splash": film + R + W}[case["setup"]]
    dx, dy = x - xc, y - yc
    if not case["wall_x"]:
        dx = dx - nx * torch.round(dx / nx)
    if not case["wall_y"]:
        dy = dy - ny * torch.round(dy / ny)
    phi = torch.tanh(2.0 * (R - torch.sqrt(dx * dx + dy * dy)) / W)
    drop = phi
    if film:
        phi = torch.maximum(phi, torch.tanh(2.0 * (film - y) / W).expand(ny, nx))
    # a weak stream that vanishes at the walls
    amp = 1e-3
    kx, ky = 2.0 * math.pi / nx, 2.0 * math.pi / ny
    env = torch.ones_like(phi)
    if case["wall_x"]:
        env = env * torch.sin(math.pi * (x + 0.5) / nx)
    if case["wall_y"]:
        env = env * torch.sin(math.pi * (y + 0.5) / ny)
    a = [rng.uniform(-1.0, 1.0) for _ in range(4)]
    ux = amp * env * (a[0] * torch.sin(ky * y + a[1]) + 0.0 * x)
    uy = amp * env * (a[2] * torch.sin(kx * x + a[3]) + 0.0 * y)
    if case["setup"] == "splash":
        uy = uy - torch.where(drop >= 0.0, 0.04, 0.0)
    return torch.stack([phi, ux, uy, torch.zeros_like(phi)]).to(torch.float32).contiguous()


def prepare(case, seed):
    dev = torch.device("cuda")
    stream = torch.cuda.current_stream()
    if case["kind"] == "serve":
        reqs = []
        for i, m in enumerate(_members(case, seed)):
            f = _fields(m, seed + 101 * i, dev).cpu().numpy()
            w = types.SimpleNamespace(nx=m["nx"], ny=m["ny"], cells=m["nx"] * m["ny"], phys=_physical(m), phi0=f[0],
                                      ux0=f[1], uy0=f[2], p0=f[3])
            reqs.append(serve.Request(i, w, m["steps"], 0.0, STORAGE[m["storage"]]))
        # a server that lives as long as the program, with the defaults a user gets
        return {"case": case, "requests": reqs,
                "server": serve.Server(budget_bytes=20 * 10 ** 9, keep_fields=True, stream=stream)}
    members = _members(case, seed) if case["kind"] == "batch" else [case]
    sims, ins, outs = [], [], []
    for i, m in enumerate(members):
        sims.append(lbm.Sim(m["nx"], m["ny"], lbm.params_from_physical(_physical(m), STORAGE[m["storage"]]),
                            stream=stream))
        f = _fields(m, seed + 101 * i, dev)
        o = torch.zeros((5, m["ny"], m["nx"]), dtype=torch.float32, device=dev)
        if m["host"]:
            f, o = f.cpu().pin_memory(), torch.zeros(o.shape, dtype=torch.float32).pin_memory()
        ins.append(f)
        outs.append(o)
    st = {"case": case, "sims": sims, "in": ins, "out": outs}
    if case["kind"] == "batch":
        st["batch"] = lbm.Batch(stream=stream)
        for s in sims:
            st["batch"].add(s)
    elif case["force"]:
        shape = (case["ny"], case["nx"])
        st["force"] = {k: torch.zeros(shape, dtype=torch.float32, device=dev) for k in ("fax", "fay")}
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------------------ one pass

def _out_dict(t):
    return {k: t[i] for i, k in enumerate(FIELDS)}


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        results = state["server"].run(state["requests"], realtime=False)
        return [dict(r.fields, diag=np.array([r.diagnostics[k] for k in DIAG])) for r in results]
    if case["kind"] == "batch":
        for s, f in zip(state["sims"], state["in"]):
            s.init_fields(f[0], f[1], f[2], f[3])
        state["batch"].step(case["steps"])
        return [s.moments_packed(o) for s, o in zip(state["sims"], state["out"])]
    sim, f, o = state["sims"][0], state["in"][0], state["out"][0]
    if case["host"]:
        sim.init_fields_packed(f)
    else:
        sim.init_fields(f[0], f[1], f[2], f[3])
    log, done = [], 0
    while done < case["steps"]:
        n = min(case["diag_every"] or case["steps"], case["steps"] - done)
        sim.step(n)
        done += n
        if case["diag_every"]:
            d = sim.diagnostics()
            log.append([d[k] for k in DIAG])
    if case["host"]:
        sim.moments_packed(o)
        out = _out_dict(o)
    else:
        out = sim.moments(_out_dict(o))
    if log:
        out = dict(out, diag=np.array(log))
    if case["force"]:
        out = dict(out, **sim.interfacial_force(state["force"]))
    return out


# ------------------------------------------------------------------------------ what a pass needs

def work(case):
    """A time step reads and writes the 18 populations of every cell once (4 bytes each, or 2 with
    16-bit storage); the initial fields are read and the results written once.  The arithmetic of
    a cell's step (both equilibria, the forcing, the stencils of phi, mu, p and u) is about 430
    operations."""
    members = _members(case, 0) if case["kind"] != "run" else [case]
    nbytes = flops = 0
    for m in members:
        cells = m["nx"] * m["ny"]
        pop = 18 * (4 if m["storage"] == "fp32" else 2)
        nbytes += cells * (2 * pop * m["steps"] + 4 * 4 + 5 * 4 + (8 if m["force"] else 0))
        flops += 430 * cells * m["steps"]
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------ 64-bit answer

_E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
_WT = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4


class _Exact:
    """The scheme in plain float64 torch operations."""

    def __init__(self, case, fields):
        self.c = c = case
        self.wx, self.wy = c["wall_x"], c["wall_y"]
        self.kappa = 3.0 * c["sigma"] * c["W"] / 8.0
        self.beta = 3.0 * c["sigma"] / (4.0 * c["W"])
        self.thM, self.wf = 0.1, 1.0 / c["tau_f"]
        self.gam = self.thM / (c["tau_f"] - 0.5)
        self.drho = c["rho_A"] - c["rho_B"]
        self.eta = {k: c["rho_" + k] * c["nu_" + k] for k in "AB"}
        phi, u, v, p = (t.to(torch.float64) for t in fields)
        mu = self.chem(phi)
        rho = self.density(phi)[1]
        poly = [self.poly(a, u, v) for a in range(9)]
        self.f = [_WT[a] * (phi * (1.0 + poly[a]) if c["f_form"] else 3.0 * self.gam * mu + phi * poly[a])
                  for a in range(9)]
        self.f[0] = phi - sum(self.f[1:])
        self.g = [_WT[a] * (p + rho / 3.0 * poly[a]) for a in range(9)]
        if c["s_form"]:
            self.last = (rho, self.div(rho * u, rho * v))

    @staticmethod
    def poly(a, u, v):
        eu = _E[a][0] * u + _E[a][1] * v
        return 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u + v * v)

    def near(self, q):
        """3x3 neighbourhood views n(dx, dy); beyond a wall the mirrored row or column."""
        q = torch.cat([q[:1], q, q[-1:]] if self.wy else [q[-1:], q, q[:1]], 0)
        q = torch.cat([q[:, :1], q, q[:, -1:]] if self.wx else [q[:, -1:], q, q[:, :1]], 1)
        ny, nx = q.shape
        return lambda dx, dy: q[1 + dy:ny - 1 + dy, 1 + dx:nx - 1 + dx]

    def lap(self, q):
        n = self.near(q)
        return (4.0 * (n(1, 0) + n(-1, 0) + n(0, 1) + n(0, -1)) + n(1, 1) + n(1, -1) + n(-1, 1) + n(-1, -1)
                - 20.0 * q) / 6.0

    def ddx(self, q):
        n = self.near(q)
        return (4.0 * (n(1, 0) - n(-1, 0)) + n(1, 1) - n(-1, 1) + n(1, -1) - n(-1, -1)) / 12.0

    def ddy(self, q):
        n = self.near(q)
        return (4.0 * (n(0, 1) - n(0, -1)) + n(1, 1) - n(1, -1) + n(-1, 1) - n(-1, -1)) / 12.0

    def div(self, a, b):
        return self.ddx(a) + self.ddy(b)

    def chem(self, phi):
        return 4.0 * self.beta * phi * (phi * phi - 1.0) - self.kappa * self.lap(phi)

    def density(self, phi):
        cl = ((phi + 1.0) / 2.0).clamp(0.0, 1.0)
        return cl, self.c["rho_B"] + cl * self.drho

    def macro(self):
        c = self.c
        phi = sum(self.f)
        mu = self.chem(phi)
        cl, rho = self.density(phi)
        gx, gy = self.ddx(phi), self.ddy(phi)
        if c["fs_form"]:
            fx, fy = mu * gx, mu * gy
        else:
            fx, fy = -phi * self.ddx(mu), -phi * self.ddy(mu)
        fy = fy - c["gravity"] * rho
        lapmu = self.lap(mu)
        s = (rho - self.last[0]) + self.last[1] if c["s_form"] else self.drho / 2.0 * self.thM * lapmu
        g = self.g
        jx = g[1] - g[3] + g[5] - g[6] - g[7] + g[8]
        jy = g[2] - g[4] + g[5] + g[6] - g[7] - g[8]
        den = rho - 0.5 * s if c["remove_Fa"] else rho
        u, v = (3.0 * jx + 0.5 * fx) / den, (3.0 * jy + 0.5 * fy) / den
        rx, ry = self.drho / 2.0 * gx, self.drho / 2.0 * gy
        p = sum(g) + (u * rx + v * ry) / 6.0
        return dict(phi=phi, mu=mu, cl=cl, rho=rho, gx=gx, gy=gy, fx=fx, fy=fy, lapmu=lapmu, s=s, ux=u, uy=v, rx=rx,
                    ry=ry, p=p)

    def step(self):
        c, m = self.c, self.macro()
        u, v, rho, phi, p, s = m["ux"], m["uy"], m["rho"], m["phi"], m["p"], m["s"]
        fx, fy = (m["fx"] + u * s, m["fy"] + v * s) if c["remove_Fa"] else (m["fx"], m["fy"])
        dx, dy = fx - (self.ddx(p) - m["rx"] / 3.0), fy - (self.ddy(p) - m["ry"] / 3.0)
        visc = self.eta["B"] + m["cl"] * (self.eta["A"] - self.eta["B"])
        wg = 1.0 / (3.0 * visc / rho + 0.5)
        phid = 0.0 if c["ch_conservative"] else phi * self.div(u, v)
        uf, ud = u * fx + v * fy, u * dx + v * dy
        h = 1.0 - 0.5 * self.wf
        fs, gs = [None] * 9, [None] * 9
        for a, (ex, ey) in enumerate(_E):
            w, poly = _WT[a], self.poly(a, u, v)
            src = w * (ex * fx + ey * fy - uf) + w * poly * (ex * dx + ey * dy - ud)
            gs[a] = (1.0 - wg) * self.g[a] + wg * w * (p + rho / 3.0 * poly) + (1.0 - 0.5 * wg) * src
            if a:
                if c["f_form"]:
                    eq = w * (1.0 + poly) * (self.wf * phi + h * ((ex - u) * m["gx"] + (ey - v) * m["gy"])
                                             + self.thM * m["lapmu"])
                else:
                    eq = self.wf * w * (3.0 * self.gam * m["mu"] + phi * poly)
                fs[a] = (1.0 - self.wf) * self.f[a] + eq + w * phid
        total = phi + phid + (self.thM * m["lapmu"] if c["f_form"] else 0.0)
        fs[0] = total - sum(fs[1:])
        if c["s_form"]:
            self.last = (rho, self.div(rho * u, rho * v))
        self.f, self.g = self.stream(fs), self.stream(gs)

    def stream(self, post):
        out = []
        for a, (ex, ey) in enumerate(_E):
            q = torch.roll(post[a], (ey, ex), (0, 1))
            back = post[_OPP[a]]
            if ey and self.wy:
                r = 0 if ey > 0 else -1
                q[r] = back[r]
            if ex and self.wx:
                r = 0 if ex > 0 else -1
                q[:, r] = back[:, r]
            out.append(q)
        return out

    def diag(self):
        m = self.macro()
        phi, c, u, v, p = m["phi"], m["cl"], m["ux"], m["uy"], m["p"]
        ny, nx = phi.shape
        x = torch.arange(nx, dtype=torch.float64, device=phi.device)[None, :]
        y = torch.arange(ny, dtype=torch.float64, device=phi.device)[:, None]
        sc = c.sum()
        liq, gas = phi > 0.9, phi < -0.9
        mean = lambda mask: p[mask].mean() if bool(mask.any()) else torch.zeros((), dtype=torch.float64)
        row = [phi.sum(), sc, (c * x).sum() / sc, (c * y).sum() / sc, (c * u).sum() / sc, (c * v).sum() / sc,
               0.5 * c.sum(1).max(), torch.sqrt(u * u + v * v).max(), mean(liq), mean(gas)]
        return [float(t) for t in row]


def _exact_run(case, seed, dev, final_diag=False):
    sim = _Exact(case, _fields(case, seed, dev))
    log = []
    for i in range(1, case["steps"] + 1):
        sim.step()
        if case["diag_every"] and (i % case["diag_every"] == 0 or i == case["steps"]):
            log.append(sim.diag())
    m = sim.macro()
    out = {k: m[k] for k in FIELDS}
    if final_diag:
        out["diag"] = np.array(sim.diag())
    elif log:
        out["diag"] = np.array(log)
    if case["force"]:
        out.update(fax=-m["ux"] * m["s"], fay=-m["uy"] * m["s"])
    return out


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "run":
        return _exact_run(case, seed, dev)
    outs = [_exact_run(m, seed + 101 * i, dev, final_diag=case["kind"] == "serve")
            for i, m in enumerate(_members(case, seed))]
    return [torch.stack([o[k] for k in FIELDS]) for o in outs] if case["kind"] == "batch" else outs
