"""Performance cases: the solver's work as its users call it, over the range of sizes it is used on.

Every case goes through the public binding (`janc.Grid`, `janc.janc_*`, `janc.Amr`). The states are
detonation-like: a hot, radical-rich, fast and compressed zone behind a front a few cells wide, fresh
gas ahead of it, and smooth seeded waves in every field, so that the WENO5 weights, the Newton
iterations, the stiff kinetics and the refinement all meet the values they meet in a running solve.
`exact` is an independent plain torch FP64 statement of the method (arXiv 2504.13750, Sec. 3-4); the
gradients of the adjoint cases come from torch autograd through it.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2504_13750_gb300 import inputs, janc

RU, P_REF, ATM = 8.314472, 101325.0, 101325.0
WALL, ZEROGRAD, PERIODIC = 0, 1, 2
# boundary sets by name: left, right, bottom, top
BCS = {"walls": (0, 0, 0, 0), "open": (1, 1, 1, 1), "channel": (2, 2, 0, 1), "duct": (0, 1, 2, 2)}
CHEM = {"off": janc.CHEM_OFF, "lie": janc.CHEM_LIE, "strang": janc.CHEM_STRANG, "explicit": janc.CHEM_EXPLICIT}
H2AIR, GLOBAL, GAS = "h2air_synth", "global_h2o2_g129", "ideal_gamma14"
LX = 0.05          # length of every domain, m
SPEED = 2600.0     # above every |u| + c of the states, m/s: fixed steps take 0.4 h / SPEED
_mechs = {}


def _mech(name):
    if name not in _mechs:
        _mechs[name] = inputs.load_mechanism(name)
    return _mechs[name]


def listed():
    return [
        # the smallest solve of the serving mix: a step is seven short launches, latency is everything
        dict(name="step_128x16", kind="step", mech=H2AIR, nx=128, ny=16, chem="lie", bc="walls", aspect=1.0, steps=20),
        # an everyday resolution of a detonation tube
        dict(name="step_512x64", kind="step", mech=H2AIR, nx=512, ny=64, chem="lie", bc="walls", aspect=1.0, steps=8),
        # the benchmark's production grid, the largest call
        dict(name="step_4096x512", kind="step", mech=H2AIR, nx=4096, ny=512, chem="lie", bc="walls", aspect=1.0, steps=2),
        # second-order splitting on an odd, ragged grid with stretched cells and mixed sides
        dict(name="step_strang_383x97", kind="step", mech=H2AIR, nx=383, ny=97, chem="strang", bc="duct", aspect=1.7, steps=5),
        # inert gas dynamics (one species), the validation cases' gas, on an odd grid
        dict(name="step_gas_1021x257", kind="step", mech=GAS, nx=1021, ny=257, chem="off", bc="open", aspect=1.0, steps=6),
        # the forward model of the inverse problem: one-step mechanism as an explicit source
        dict(name="step_channel_1000x400", kind="step", mech=GLOBAL, nx=1000, ny=400, chem="explicit", bc="channel", aspect=1.0, steps=4),
        # one right-hand side with its face fluxes, for a caller's own time integrator
        dict(name="rhs_2048x256", kind="rhs", mech=H2AIR, nx=2048, ny=256, chem="lie", bc="walls", aspect=1.0, steps=1),
        # a field of constant-volume reactors: the stiff chemistry alone
        dict(name="reactors_300x101", kind="reactors", mech=H2AIR, nx=300, ny=101, chem="lie", bc="open", aspect=1.0, steps=6),
        # a gradient through the reacting tube, linearisation kept, two checkpoint segments
        dict(name="adjoint_512x64", kind="adjoint", mech=H2AIR, nx=512, ny=64, chem="lie", bc="walls", aspect=1.0, steps=6, ckpt=3, store=True),
        # one descent iteration's gradient of the inverse problem, whole trajectory kept
        dict(name="adjoint_channel_1000x400", kind="adjoint", mech=GLOBAL, nx=1000, ny=400, chem="explicit", bc="channel", aspect=1.0, steps=2, ckpt=2, store=True),
        # a batch of mixed solves through the continuous-batching server, host arrays in and out
        dict(name="serve_16", kind="serve", mech=H2AIR, nx=512, ny=64, chem="lie", bc="walls", aspect=1.0, steps=12, requests=16),
        # block-structured refinement following the front, two layers, one regrid on the way
        dict(name="amr_512x128", kind="amr", mech=H2AIR, nx=512, ny=128, chem="lie", bc="walls", aspect=1.0, steps=6, levels=2, every=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["rhs", "reactors", "adjoint", "adjoint", "serve", "amr"])
    nx, ny = _log_int(rng, 96, 4096), _log_int(rng, 7, 512)
    aspect = rng.choice([1.0, 1.0, rng.uniform(0.6, 1.7)])
    c = dict(kind=kind, mech=H2AIR, nx=nx, ny=ny, chem="lie", bc=rng.choice(sorted(BCS)), aspect=aspect)
    if kind == "step":
        c["mech"], c["chem"] = rng.choice([(H2AIR, "lie"), (H2AIR, "lie"), (H2AIR, "strang"), (H2AIR, "off"), (H2AIR, "explicit"),
                                           (GLOBAL, "explicit"), (GLOBAL, "lie"), (GAS, "off")])
    if kind == "rhs":
        c["mech"] = rng.choice([H2AIR, GLOBAL, GAS])
        c["chem"] = "off"
    if kind == "adjoint":
        c["mech"], c["chem"] = rng.choice([(H2AIR, "lie"), (H2AIR, "off"), (GLOBAL, "explicit"), (GAS, "off")])
        c["nx"], c["ny"] = min(c["nx"], 700), min(c["ny"], 128)
        c["ckpt"] = rng.choice([2, 3, 8])
        c["store"] = rng.random() < 0.5
    if kind == "serve":
        c.update(nx=min(nx, 700), ny=min(max(ny, 8), 96), bc="walls", requests=rng.randint(2, 16))
    if kind == "amr":
        c.update(nx=8 * max(16, min(nx, 640) // 8), ny=8 * max(2, min(ny, 128) // 8), bc="walls", aspect=1.0, levels=rng.choice([1, 2]), every=5)
    c["steps"] = 1 if kind == "rhs" else max(1, min(rng.randint(2, 12), 4_000_000 // (c["nx"] * c["ny"])))
    if kind == "adjoint":
        c["steps"] = max(1, min(c["steps"], 5))
    return c


# ---- what a user has in hand -----------------------------------------------------------------


def _fields(c, seed, nx=None, ny=None):
    """T, p, u, v [ny, nx] and Y [ns, ny, nx] on the GPU, and dx, dy: a front at a seeded place."""
    nx, ny = nx or c["nx"], ny or c["ny"]
    m = _mech(c["mech"])
    r = np.random.default_rng([seed, nx, ny])
    dx = LX / nx
    dy = c["aspect"] * dx
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny

    def wave():
        w = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
        for _ in range(3):
            kx, ky = int(r.integers(1, 6)), int(r.integers(0, 4))
            w += math.sqrt(1 / 3) * torch.sin(2 * math.pi * (kx * x[None, :] + ky * y[:, None]) + float(r.uniform(0, 6.28)))
        return w

    xf = float(r.uniform(0.25, 0.7)) + 0.02 * torch.sin(2 * math.pi * (int(r.integers(1, 4)) * y[:, None]) + float(r.uniform(0, 6.28)))
    hot = torch.sigmoid((xf - x[None, :]) * nx / 1.2)       # the front: about 5 cells
    T = (300.0 * (1 - hot) + 2300.0 * hot) * (1 + 0.015 * wave())
    p = ATM * ((1 - hot) + 14.0 * hot) * (1 + 0.02 * wave())
    u = 800.0 * hot * (1 + 0.05 * wave()) + 15.0 * wave()
    v = 30.0 * wave()
    fresh = torch.zeros(m["ns"], dtype=torch.float64, device="cuda")
    burnt = torch.zeros_like(fresh)
    if m["ns"] == 9:
        fresh += torch.from_numpy(inputs.h2air_Y(m, float(r.uniform(0.6, 1.4)))).cuda()
        part = {"H2": 0.006, "O2": 0.03, "H": 1e-3, "O": 5e-3, "OH": 0.02, "HO2": 1e-4, "H2O2": 1e-5, "H2O": 0.19, "N2": 0.747}
        burnt += torch.from_numpy(inputs.premix_Y(m, part)).cuda()
    elif m["ns"] == 3:
        phi = float(r.uniform(0.8, 1.2))
        fresh += torch.tensor([2 * phi * m["M"][0], m["M"][1], 0.0], dtype=torch.float64, device="cuda")
        fresh /= fresh.sum()
        burnt += torch.tensor([0.02, 0.12, 0.86], dtype=torch.float64, device="cuda")
    else:
        fresh += 1.0
        burnt += 1.0
    mix = hot * (1 + 0.03 * wave()).clamp(max=1.0)
    Y = fresh[:, None, None] * (1 - mix) + burnt[:, None, None] * mix
    Y = Y / Y.sum(0, keepdim=True)
    return [t.contiguous() for t in (T, p, u, v, Y)], dx, dy


def _grid(c, dx, dy):
    return janc.Grid(_mech(c["mech"]), c["nx"], c["ny"], dx, dy, BCS[c["bc"]], chemistry=CHEM[c["chem"]])


def _serve_list(c, seed):
    """(nx, ny, steps, seed of the fields) of every request: the sizes by the case, the fields by the seed."""
    r = np.random.default_rng([c["nx"], c["ny"], c["requests"]])
    out = []
    for k in range(c["requests"]):
        s = 2 ** int(r.integers(0, 3))
        nx, ny = max(24, c["nx"] // s - int(r.integers(0, 4))), max(8, c["ny"] // s - int(r.integers(0, 4)))
        out.append((nx, ny, int(r.integers(max(1, c["steps"] // 2), c["steps"] + 1)), seed * 1000 + k))
    return out


def _fixed_dt(dx, dy):
    return 0.4 * min(dx, dy) / SPEED


def prepare(c, seed):
    kind = c["kind"]
    if kind == "serve":
        reqs = []
        for nx, ny, steps, s in _serve_list(c, seed):
            f, dx, dy = _fields(c, s, nx, ny)
            desc = janc.make_desc(nx, ny, dx, dy, BCS[c["bc"]], chemistry=True)
            nv = _mech(c["mech"])["ns"] + 3
            reqs.append((desc, [t.cpu().numpy() for t in f], steps, np.empty((nv, ny, nx)), np.empty((ny, nx))))
        mech = janc.Mechanism(_mech(c["mech"]))
        server = janc.janc_server_create(mech, chemistry=True, pool_bytes=1 << 29, max_active=32)
        return {"c": c, "reqs": reqs, "mech": mech, "server": _Server(server)}
    f, dx, dy = _fields(c, seed)
    s = {"c": c, "f": f}
    if kind == "amr":
        grid = inputs.grid_dict(c["nx"], c["ny"], dx, dy, BCS[c["bc"]])
        # refine where T rises by more than about 120 K a base cell: the front
        s["g"] = janc.Amr(_mech(c["mech"]), grid, chemistry=True, levels=c["levels"], threshold=120.0 / dx, n_buffer=2, regrid_every=c["every"])
        # host arrays for the blocks of each layer, with room for every block it can have
        s["layers"] = []
        for k in range(1, c["levels"] + 1):
            n = (c["nx"] << k) // 16 * ((c["ny"] << k) // 16)
            s["layers"].append((np.zeros((n, 2), np.int32), np.zeros((n, s["g"].nv, 16, 16)), np.zeros((n, 16, 16))))
    else:
        s["g"] = _grid(c, dx, dy)
    nv, nx, ny = s["g"].nv, c["nx"], c["ny"]
    new = lambda *shape: torch.empty(shape, dtype=torch.float64, device="cuda")  # noqa: E731
    s["U"], s["T"] = new(nv, ny, nx), new(ny, nx)
    s["dt"] = _fixed_dt(dx, dy)
    if kind == "rhs":
        s["g"].set_primitive(*f)
        s["out"] = {"Fx": new(nv, ny, nx + 1), "Gy": new(nv, ny + 1, nx), "L": new(nv, ny, nx), "alpha": new(2)}
    if kind == "adjoint":
        h = s["g"].handle
        janc.janc_set_adjoint_mode(h, janc.ADJ_STORE_FACES if c["store"] else janc.ADJ_RECOMPUTE)
        s["nbytes"] = janc.janc_adjoint_workspace_bytes(h, c["steps"], c["ckpt"])
        s["ws"] = torch.empty(s["nbytes"] + 256, dtype=torch.uint8, device="cuda")
        s["wp"] = (s["ws"].data_ptr() + 255) & ~255
        s["seed"] = _cotangent(c, seed, nv)
        s["gU0"] = new(nv, ny, nx)
    return s


def _cotangent(c, seed, nv):
    """dL/dU^N of a loss that weighs every conserved variable by its own size."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 11)
    w = torch.randn(nv, c["ny"], c["nx"], dtype=torch.float64, device="cuda", generator=gen)
    size = torch.tensor([1.0, 1e3, 1e3, 1e6] + [0.1] * (nv - 4), dtype=torch.float64, device="cuda")
    return w / size[:, None, None]


class _Server:
    def __init__(self, h):
        self.h = h

    def __del__(self):
        janc.janc_server_destroy(self.h)


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "serve":
        h = s["server"].h
        ids = [janc.janc_server_submit(h, d, *f, n, cfl=0.5) for d, f, n, _, _ in s["reqs"]]
        left = set(ids)
        while left:
            done, _ = janc.janc_server_run_until(h)
            left -= set(done)
        out = []
        for rid, (_, _, _, U, T) in zip(ids, s["reqs"]):
            janc.janc_server_fetch(h, rid, U, T)
            out.append({"U": U, "T": T})
        return out
    g = s["g"]
    if kind == "rhs":
        o = s["out"]
        janc.janc_rhs(g.handle, o["Fx"], o["Gy"], o["L"], o["alpha"])
        return o
    if kind == "amr":
        g.set_primitive(*s["f"])
        t = g.step(c["steps"], cfl=0.5)
        janc.janc_amr_get_base(g.handle, s["U"], s["T"])
        for k, arrays in enumerate(s["layers"]):
            rc = janc.lib().janc_amr_get_layer(g.handle, k + 1, *[a.ctypes.data for a in arrays])
            if rc:
                raise janc.JancError(rc, janc.janc_last_error())
        return {"U": s["U"], "T": s["T"], "t": t, "layers": s["layers"]}
    g.set_primitive(*s["f"])
    if kind == "adjoint":
        janc.janc_adjoint_forward(g.handle, c["steps"], s["dt"], c["ckpt"], janc.LOSS_SEEDED, s["wp"], s["nbytes"])
        janc.janc_get_state(g.handle, s["U"], s["T"])
        janc.janc_adjoint_reverse(g.handle, s["seed"], s["gU0"])
        return {"U": s["U"], "T": s["T"], "gU0": s["gU0"]}
    if kind == "reactors":
        janc.janc_source_step(g.handle, c["steps"], s["dt"])
    else:
        g.step(c["steps"], cfl=0.5)
    janc.janc_get_state(g.handle, s["U"], s["T"])
    return {"U": s["U"], "T": s["T"]}


# ---- work ------------------------------------------------------------------------------------

WENO_FLOPS = 69  # one textbook WENO5 reconstruction


def _chem_flops(m):
    """Point-implicit chemistry of one cell: rates, Jacobian, solve (a fused multiply-add is 2)."""
    ns, nr = m["ns"], m["nr"]
    n = ns - 1
    part = int((m["nuf"] > 0).sum() + (m["nub"] > 0).sum())
    return 17 * ns + 8 * nr + 4 * part + 6 * part + 2 * n * nr + 2 * n ** 3 // 3 + 4 * n * n


def work(c):
    """Per step: the state read and written once, the face reconstructions, update and chemistry."""
    m = _mech(c["mech"])
    ns = m["ns"]
    nv = ns + 3
    stage = 2 * nv * (2 * WENO_FLOPS + 6) + 12 * nv + 20 * ns + 60
    chem = {"off": 0, "lie": 1, "strang": 2, "explicit": 1}[c["chem"]] * _chem_flops(m)
    state = 8 * (nv + 1)
    kind = c["kind"]
    if kind == "serve":
        fl = by = 0
        for nx, ny, steps, _ in _serve_list(c, 0):
            fl += nx * ny * steps * (3 * stage + chem)
            by += nx * ny * (state + 8 * (ns + 4))
        return {"bytes": by, "flops": fl}
    n = c["nx"] * c["ny"]
    if kind == "rhs":
        return {"bytes": 8 * n * (nv + 2 + 3 * nv), "flops": n * 2 * nv * (2 * WENO_FLOPS + 6)}
    if kind == "reactors":
        return {"bytes": n * (state + 8 * (ns + 4)), "flops": n * c["steps"] * _chem_flops(m)}
    step = 3 * stage + chem * (3 if c["chem"] == "explicit" else 1)
    by = n * (state + 8 * (ns + 4))
    if kind == "adjoint":  # a forward and a reverse sweep of twice its operations
        return {"bytes": by + n * 16 * nv, "flops": 3 * n * c["steps"] * step}
    if kind == "amr":      # the front's blocks: about a tenth of each layer, 2^k substeps each
        extra = sum(0.1 * 8 ** k for k in range(1, c["levels"] + 1))
        return {"bytes": by, "flops": n * (1 + extra) * c["steps"] * step}
    return {"bytes": by, "flops": n * c["steps"] * step}


# ---- the method in plain torch, 64 bits ------------------------------------------------------


class _Ref:
    def __init__(self, c, nx, ny, dx, dy):
        m = _mech(c["mech"])
        dev = lambda a: torch.as_tensor(np.asarray(a), device="cuda")  # noqa: E731
        self.ns, self.nr, self.nv = m["ns"], m["nr"], m["ns"] + 3
        self.M, self.nasa, self.nuf, self.nub = dev(m["M"]), dev(m["nasa"]), m["nuf"], m["nub"]
        self.A, self.b, self.Ea, self.tb, self.eff = m["A"], m["b"], m["Ea"], m["tb"], dev(m["eff"])
        self.net = dev((m["nub"] - m["nuf"]).astype(np.float64))
        self.nx, self.ny, self.dx, self.dy, self.bc, self.chem = nx, ny, dx, dy, BCS[c["bc"]], c["chem"]

    def z(self, U):
        """rho Y_k / M_k of all species."""
        last = U[0] - U[4:].sum(0) if self.ns > 1 else U[0]
        return torch.cat([U[4:], last[None]]) / self.M[:, None, None]

    def conserved(self, T, p, u, v, Y):
        z = Y / self.M[:, None, None]
        rho = p / (RU * z.sum(0) * T)
        h = RU * (z * self.h(T)).sum(0)
        U = [rho, rho * u, rho * v, rho * h - p + 0.5 * rho * (u * u + v * v)]
        return torch.cat([torch.stack(U), (rho * Y)[:-1]])

    def h(self, T):
        """h_k M_k / Ru of every species, [ns, ...]."""
        a = self.nasa
        return torch.stack([T * (a[k, 0] + T * (a[k, 1] / 2 + T * (a[k, 2] / 3 + T * (a[k, 3] / 4 + T * a[k, 4] / 5)))) + a[k, 5] for k in range(self.ns)])

    def cp(self, T):
        a = self.nasa
        return torch.stack([a[k, 0] + T * (a[k, 1] + T * (a[k, 2] + T * (a[k, 3] + T * a[k, 4]))) for k in range(self.ns)])

    def temperature(self, U, Tw):
        rhoe = (U[3] - 0.5 * (U[1] ** 2 + U[2] ** 2) / U[0]) / RU

        def parts(T, z):
            W = z.sum(0)
            return (z * self.h(T)).sum(0) - W * T - rhoe, (z * self.cp(T)).sum(0) - W

        with torch.no_grad():
            T, z = Tw, self.z(U)
            for _ in range(7):
                F, D = parts(T, z)
                T = T - F / D
        z = self.z(U)
        F, D = parts(T, z)
        return T - F / D.detach()   # the implicit function's value and derivative

    def aux(self, U, T):
        z = self.z(U)
        W = z.sum(0)
        cp = (z * self.cp(T)).sum(0)
        p = RU * W * T
        c = torch.sqrt(cp / (cp - W) * p / U[0])
        u, v = U[1] / U[0], U[2] / U[0]
        return u, v, p, (u.abs() + c).amax(), (v.abs() + c).amax()

    @staticmethod
    def ghosts(n, lo, hi):
        i = torch.arange(-3, n + 3)
        flip = ((i < 0) & (lo == WALL)) | ((i >= n) & (hi == WALL))
        at = torch.where(i < 0, -1 - i if lo == WALL else (i * 0 if lo == ZEROGRAD else i + n), i)
        at = torch.where(i >= n, 2 * n - 1 - i if hi == WALL else (i * 0 + n - 1 if hi == ZEROGRAD else i - n), at)
        return at.cuda(), torch.where(flip, -1.0, 1.0).to(torch.float64).cuda()

    @staticmethod
    def weno(v0, v1, v2, v3, v4):
        eps = 1e-6
        b0 = 13 / 12 * (v0 - 2 * v1 + v2) ** 2 + 0.25 * (v0 - 4 * v1 + 3 * v2) ** 2
        b1 = 13 / 12 * (v1 - 2 * v2 + v3) ** 2 + 0.25 * (v1 - v3) ** 2
        b2 = 13 / 12 * (v2 - 2 * v3 + v4) ** 2 + 0.25 * (3 * v2 - 4 * v3 + v4) ** 2
        a0, a1, a2 = 0.1 / (eps + b0) ** 2, 0.6 / (eps + b1) ** 2, 0.3 / (eps + b2) ** 2
        q0, q1, q2 = (2 * v0 - 7 * v1 + 11 * v2) / 6, (-v1 + 5 * v2 + 2 * v3) / 6, (2 * v2 + 5 * v3 - v4) / 6
        return (a0 * q0 + a1 * q1 + a2 * q2) / (a0 + a1 + a2)

    def faces(self, U, un, p, alpha, axis):
        """Face fluxes along axis 0 (y) or 1 (x) of the [ny, nx] planes."""
        n = self.nx if axis == 1 else self.ny
        at, sign = self.ghosts(n, *(self.bc[:2] if axis == 1 else self.bc[2:]))
        sign = sign[None, :] if axis == 1 else sign[:, None]
        mom = 1 if axis == 1 else 2
        pad = lambda a: a.index_select(axis, at)  # noqa: E731
        ug, pg = pad(un) * sign, pad(p)
        out = []
        for k in range(self.nv):
            q = pad(U[k])
            if k == mom:
                q = q * sign
            f = ug * q + (pg if k == mom else pg * ug if k == 3 else 0.0)
            plus, minus = 0.5 * (f + alpha * q), 0.5 * (f - alpha * q)
            w = lambda a, s: a.narrow(axis, s, n + 1)  # noqa: E731
            out.append(self.weno(*[w(plus, s) for s in range(5)]) + self.weno(*[w(minus, 5 - s) for s in range(5)]))
        return torch.stack(out)

    def rhs(self, U, T):
        u, v, p, ax, ay = self.aux(U, T)
        Fx, Gy = self.faces(U, u, p, ax, 1), self.faces(U, v, p, ay, 0)
        L = -(Fx[:, :, 1:] - Fx[:, :, :-1]) / self.dx - (Gy[:, 1:] - Gy[:, :-1]) / self.dy
        return L, Fx, Gy, ax, ay

    def kinetics(self, X, T):
        """Rates of progress [nr, cells], dq/dX [nr, ns, cells] of concentrations X [ns, cells]."""
        a = self.nasa
        G = [a[k, 0] * (torch.log(T) - 1) + T * (a[k, 1] / 2 + T * (a[k, 2] / 6 + T * (a[k, 3] / 12 + T * a[k, 4] / 20))) - a[k, 5] / T + a[k, 6] for k in range(self.ns)]
        qs, dqs = [], []
        for i in range(self.nr):
            kf = self.A[i] * torch.exp(self.b[i] * torch.log(T) - self.Ea[i] / (RU * T))
            nu = self.nub[i] - self.nuf[i]
            lnK = sum(int(nu[j]) * G[j] for j in range(self.ns) if nu[j]) + int(nu.sum()) * torch.log(P_REF / (RU * T))
            kb = kf / torch.exp(lnK)
            part = lambda k, c: k * math.prod([X[j] ** int(c[j]) for j in range(self.ns) if c[j]])  # noqa: E731

            def slope(k, c, j):
                d = k * int(c[j])
                for l in range(self.ns):
                    e = int(c[l]) - (l == j)
                    if c[l] and e:
                        d = d * X[l] ** e
                return d

            net = part(kf, self.nuf[i]) - part(kb, self.nub[i])
            body = (self.eff[i][:, None] * X).sum(0) if self.tb[i] else torch.ones_like(T)
            d = []
            for j in range(self.ns):
                t = torch.zeros_like(T)
                if self.nuf[i][j]:
                    t = t + slope(kf, self.nuf[i], j)
                if self.nub[i][j]:
                    t = t - slope(kb, self.nub[i], j)
                t = body * t
                d.append(t + self.eff[i, j] * net if self.tb[i] else t)
            qs.append(body * net)
            dqs.append(torch.stack(d))
        return torch.stack(qs), torch.stack(dqs)

    def source(self, U, T):
        X = self.z(U)
        q, _ = self.kinetics(X.reshape(self.ns, -1), T.reshape(-1))
        return (self.M[:-1, None] * (self.net[:, :-1].T @ q)).reshape(self.ns - 1, *T.shape)

    def implicit(self, U, T, dt):
        """Point-implicit chemistry and the new T."""
        n = self.ns - 1
        X = self.z(U).reshape(self.ns, -1)
        parts = []
        for X0, T0 in zip(X.split(1 << 18, 1), T.reshape(-1).split(1 << 18)):
            q, dq = self.kinetics(X0, T0)
            S = self.M[:n, None] * (self.net[:, :n].T @ q)
            dX = dq / self.M[None, :, None]
            J = torch.einsum("rk,rjc->ckj", self.net[:, :n], dX[:, :n] - dX[:, n:]) * self.M[:n][None, :, None]
            A = torch.eye(n, dtype=torch.float64, device="cuda") - dt * J
            parts.append(torch.linalg.solve(A, (dt * S).T[:, :, None])[:, :, 0].T)
        V = torch.cat([U[:4], U[4:] + torch.cat(parts, 1).reshape(n, *T.shape)])
        return V, self.temperature(V, T)

    def stage(self, k, U0, U, T, dt):
        W = U + dt * self.rhs(U, T)[0]
        if self.chem == "explicit":
            W = torch.cat([W[:4], W[4:] + dt * self.source(U, T)])
        W = (W, 0.75 * U0 + 0.25 * W, U0 / 3 + 2 / 3 * W)[k]
        return W, self.temperature(W, T)

    def step(self, U, T, dt=None):
        if dt is None:
            _, _, _, ax, ay = self.aux(U, T)
            dt = 0.5 * min(self.dx, self.dy) / torch.maximum(ax, ay)
        call = (lambda f, *a: checkpoint(f, *a, use_reentrant=False)) if torch.is_grad_enabled() else (lambda f, *a: f(*a))
        if self.chem == "strang":
            U, T = self.implicit(U, T, 0.5 * dt)
        V, S = U, T
        for k in range(3):
            V, S = call(self.stage, k, U, V, S, dt)
        if self.chem in ("lie", "strang"):
            V, S = call(self.implicit, V, S, dt if self.chem == "lie" else 0.5 * dt)
        return V, S


def exact(c, seed):
    kind = c["kind"]
    if kind == "amr":
        return None  # block-structured refinement has no short plain statement
    with torch.set_grad_enabled(kind == "adjoint"):
        if kind == "serve":
            out = []
            for nx, ny, steps, s in _serve_list(c, seed):
                f, dx, dy = _fields(c, s, nx, ny)
                ref = _Ref(c, nx, ny, dx, dy)
                U, T = ref.conserved(*f), f[0]
                for _ in range(steps):
                    U, T = ref.step(U, T)
                out.append({"U": U, "T": T})
            return out
        f, dx, dy = _fields(c, seed)
        ref = _Ref(c, c["nx"], c["ny"], dx, dy)
        U, T = ref.conserved(*f), f[0]
        dt = _fixed_dt(dx, dy)
        if kind == "rhs":
            L, Fx, Gy, ax, ay = ref.rhs(U, T)
            return {"Fx": Fx, "Gy": Gy, "L": L, "alpha": torch.stack([ax, ay])}
        if kind == "adjoint":
            U0 = U.detach().requires_grad_(True)
            V, S = U0, ref.temperature(U0, T)
            for _ in range(c["steps"]):
                V, S = ref.step(V, S, dt)
            (g,) = torch.autograd.grad(V, U0, _cotangent(c, seed, ref.nv))
            return {"U": V.detach(), "T": S.detach(), "gU0": g}
        for _ in range(c["steps"]):
            U, T = ref.implicit(U, T, dt) if kind == "reactors" else ref.step(U, T, None)
        return {"U": U, "T": T}
