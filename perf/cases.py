"""Performance cases: the work users of the library have it do, through the
public binding (paper_1808_10633_gb300.wombat), with FP64 references.

Each case is a program's inner call: load a state, advance it, read it back
(`kind` "grid", "patches", "bricks"), read the diagnostics of a state
("monitor"), or train the weight networks ("train").  Sizes are those of the
repository's tests and benchmark legs (1-D waves, the 64^2 field loop, 64^3 to
256^3 turbulence, uneven patches of 16 to 64 cells, linked bricks, the
networks' minibatches of 4096 records) and odd ones between them.

`exact` is a plain torch FP64 solver of the same scheme (characteristic
WENO5 sweeps, constrained transport, SSP-RK3 / RK4) on flat cell arrays with
neighbour tables, so that one grid, a set of periodic patches and a cut world
all take the same code; it shares nothing with the library.
"""
import math

import numpy as np
import torch

from paper_1808_10633_gb300 import bricks, inputs, wombat

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
GAMMA = 5.0 / 3.0
CFL = 0.4
EPS = 1e-6                      # epsilon of the WENO weights (Sec. 2.1)


# ---- the cases -----------------------------------------------------------------
def listed():
    return [
        # the smallest call: a 1-D Alfven wave of the accuracy suites, fixed dt
        {"name": "wave1d_fp32", "kind": "grid", "state": "alfven", "nx": 32, "ny": 1, "nz": 1,
         "precision": "fp32", "integrator": "ssprk3", "weights": "js", "steps": 8, "host": "numpy"},
        # a 2-D test problem in FP64 with the paper's RK4
        {"name": "loop2d_fp64_rk4", "kind": "grid", "state": "field_loop", "nx": 64, "ny": 64, "nz": 1,
         "precision": "fp64", "integrator": "rk4", "weights": "js", "steps": 4, "host": "numpy"},
        # an ordinary FP64 run (the accuracy reference of the FP32 path)
        {"name": "turb64_fp64", "kind": "grid", "state": "turbulence", "nx": 64, "ny": 64, "nz": 64,
         "precision": "fp64", "integrator": "ssprk3", "weights": "js", "steps": 2, "host": "pinned"},
        # a large FP64 run
        {"name": "turb144_fp64", "kind": "grid", "state": "turbulence", "nx": 144, "ny": 144, "nz": 144,
         "precision": "fp64", "integrator": "ssprk3", "weights": "js", "steps": 1, "host": "pinned"},
        # odd, ragged extents with the other integrator and the other weights
        {"name": "odd_fp32_z_rk4", "kind": "grid", "state": "blasts", "nx": 119, "ny": 93, "nz": 70,
         "precision": "fp32", "integrator": "rk4", "weights": "z", "steps": 3, "host": "pinned"},
        # the benchmark's headline: 256^3 turbulence in FP32, totals of every step
        {"name": "turb256_fp32", "kind": "grid", "state": "turbulence", "nx": 256, "ny": 256, "nz": 256,
         "precision": "fp32", "integrator": "ssprk3", "weights": "js", "steps": 6, "host": "pinned",
         "totals": True},
        # the benchmark's end-to-end leg: the state in and out around every step
        {"name": "e2e192_fp32", "kind": "grid", "state": "blasts", "nx": 192, "ny": 192, "nz": 192,
         "precision": "fp32", "integrator": "ssprk3", "weights": "js", "steps": 1, "host": "pinned"},
        # many uneven periodic patches advanced together
        {"name": "patches320_fp32", "kind": "patches", "npatch": 320, "lo": 16, "hi": 64,
         "precision": "fp32", "integrator": "ssprk3", "weights": "js", "steps": 2, "host": "pinned"},
        # a world cut into 64 bricks that read their neighbours' cells
        {"name": "bricks64_fp32", "kind": "bricks", "nx": 160, "ny": 160, "nz": 160, "cuts": 4,
         "precision": "fp32", "integrator": "ssprk3", "weights": "js", "steps": 3, "host": "pinned"},
        # the learned weights on turbulence with blasts
        {"name": "learned112_fp32", "kind": "grid", "state": "blasts", "nx": 112, "ny": 112, "nz": 112,
         "precision": "learned", "integrator": "ssprk3", "weights": "js", "steps": 2, "host": "pinned"},
        # training of the weight networks and the full-batch loss and gradient after it
        {"name": "train4096", "kind": "train", "records": 120000, "steps": 60, "batch": 4096},
        # what a monitored run reads between its steps: dt, conserved totals, div b
        {"name": "monitor192_fp32", "kind": "monitor", "state": "turbulence", "nx": 192, "ny": 192, "nz": 192,
         "precision": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "grid", "learned", "patches", "bricks", "train", "monitor", "flat"])
    run = {"precision": rng.choice(["fp32", "fp32", "fp64"]), "integrator": rng.choice(["ssprk3", "ssprk3", "rk4"]),
           "weights": rng.choice(["js", "js", "js", "z"]), "host": rng.choice(["pinned", "pinned", "numpy"])}
    if kind == "flat":
        two_d = rng.random() < 0.5
        n = _log(rng, 16, 128)
        return {"kind": "grid", "state": "field_loop" if two_d else "alfven", "nx": n, "ny": n if two_d else 1,
                "nz": 1, **run, "steps": rng.randint(1, 8)}
    if kind == "patches":
        return {"kind": kind, "npatch": _log(rng, 6, 300), "lo": 16, "hi": 64, **run, "precision": "fp32",
                "steps": rng.randint(1, 2)}
    if kind == "train":
        return {"kind": kind, "records": _log(rng, 20000, 120000), "steps": rng.randint(10, 60),
                "batch": _log(rng, 500, 4096)}
    n = [_log(rng, 20, 100 if run["precision"] == "fp64" else 190) for _ in range(3)]
    if rng.random() < 0.4:      # cubes of even sizes are as common as ragged boxes
        n = [max(16, n[0] // 8 * 8)] * 3
    dims = {"nx": n[0], "ny": n[1], "nz": n[2]}
    if kind == "monitor":
        return {"kind": kind, "state": rng.choice(["turbulence", "blasts"]), **dims, "precision": run["precision"]}
    if kind == "bricks":
        dims = {k: max(24, min(v, 120)) for k, v in dims.items()}
        return {"kind": kind, **dims, "cuts": rng.randint(2, 4), **run, "steps": rng.randint(1, 2)}
    if kind == "learned":
        dims = {k: min(v, 100) for k, v in dims.items()}
        run.update(precision="learned", weights="js")
    return {"kind": "grid", "state": rng.choice(["turbulence", "turbulence", "blasts"]), **dims, **run,
            "steps": rng.randint(1, 3), "totals": rng.random() < 0.3}


# ---- inputs ----------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _gauss(dims, g, kmax=8):
    """Unit-variance Gaussian random field, modes 1 <= |k| <= 8 of variance |k|^(-11/3)."""
    nx, ny, nz = dims
    k = torch.arange(-kmax, kmax + 1, device=DEV, dtype=F64)
    kx = torch.arange(0, kmax + 1, device=DEV, dtype=F64)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2
    ok = (k2 >= 1) & (k2 <= kmax * kmax)
    amp = torch.where(ok, k2.clamp(min=1).pow(-11.0 / 12.0), torch.zeros_like(k2))
    C = torch.complex(torch.randn(k2.shape, device=DEV, dtype=F64, generator=g) * amp,
                      torch.randn(k2.shape, device=DEV, dtype=F64, generator=g) * amp)

    def wave(kk, n):
        return torch.polar(torch.ones(len(kk), n, device=DEV, dtype=F64),
                           2 * math.pi * kk[:, None] * torch.arange(n, device=DEV, dtype=F64)[None] / n)
    f = torch.matmul(C, wave(kx, nx))                               # [kz, ky, x]
    f = torch.matmul(wave(k, ny).T[None], f)                        # [kz, y, x]
    z = wave(k, nz).T                                               # [z, kz]
    f = f.reshape(len(k), -1)
    f = (z.real @ f.real - z.imag @ f.imag).reshape(nz, ny, nx)
    f = f - f.mean()
    s = f.std()
    return f / s if float(s) > 0 else f


def _curl(A, h):
    r = lambda a, d: torch.roll(a, -1, 2 - d)                      # noqa: E731  (next cell along axis d)
    return [(r(A[(d + 2) % 3], (d + 1) % 3) - A[(d + 2) % 3]) / h[(d + 1) % 3]
            - (r(A[(d + 1) % 3], (d + 2) % 3) - A[(d + 1) % 3]) / h[(d + 2) % 3] for d in range(3)]


def _assemble(rho, v, p, b):
    B = [0.5 * (b[d] + torch.roll(b[d], -1, 2 - d)) for d in range(3)]
    E = p / (GAMMA - 1) + 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) + 0.5 * (B[0] ** 2 + B[1] ** 2 + B[2] ** 2)
    return torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], *B, E]), torch.stack(b)


def _turbulence(dims, h, seed, blasts=0):
    """The repository's decaying-turbulence state (rms Mach 0.5, 10 % magnetic
    energy), optionally with over-pressured spheres."""
    g = _gen(seed)
    v = [_gauss(dims, g) for _ in range(3)]
    s = 0.5 * math.sqrt(GAMMA) / max(math.sqrt(sum(float((c * c).mean()) for c in v)), 1e-30)
    v = [c * s for c in v]
    rho = torch.exp(0.1 * _gauss(dims, g) - 0.005)
    db = _curl([_gauss(dims, g) for _ in range(3)], h)
    ek = 0.5 * float((rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)).mean())
    em = 0.5 * float((db[0] ** 2 + db[1] ** 2 + db[2] ** 2).mean())
    s = math.sqrt(0.1 * ek / em) if em > 0 else 0.0
    b = [0.1 + s * db[0], s * db[1], s * db[2]]
    p = torch.ones_like(rho)
    if blasts:
        c = torch.rand(blasts, 4, device=DEV, dtype=F64, generator=g)
        for q in c.tolist():
            d2 = torch.zeros((), device=DEV, dtype=F64)
            for d in range(3):
                x = (torch.arange(dims[d], device=DEV, dtype=F64) + 0.5) / dims[d]
                e = (x - q[d]).abs()
                e = torch.minimum(e, 1 - e) ** 2
                d2 = d2 + e.reshape([-1 if a == 2 - d else 1 for a in range(3)])
            p = torch.where(d2 < (0.02 + 0.03 * q[3]) ** 2, torch.full_like(p, 100.0), p)
    return _assemble(rho, v, p, b)


def _brio_wu(dims, h, seed):
    """Rotated periodic Brio-Wu tube: left (1, 1, 1), right (0.125, 0.1, -1),
    B_n = 0.75, and a guide field of 0.3 along the third direction (without
    it the direction of B_perp inside the reversal is set by rounding)."""
    r = np.random.default_rng(seed)
    m = np.zeros(3)
    while not m.any():
        m = r.integers(-1, 2, 3).astype(float)
    k = 2 * math.pi * m / (np.array(dims) * h)
    K = np.linalg.norm(k)
    n = k / K
    t = np.cross(n, [1.0, 0, 0] if abs(n[0]) < 0.9 else [0, 1.0, 0])
    t /= np.linalg.norm(t)
    q = np.cross(t, n)

    def phase(o):
        ax = [(torch.arange(dims[d], device=DEV, dtype=F64) + o[d]) * (h * k[d]) for d in range(3)]
        return ax[2][:, None, None] + ax[1][None, :, None] + ax[0][None, None, :]

    def tri(a):
        a = torch.remainder(a, 2 * math.pi)
        return torch.where(a < math.pi, a, 2 * math.pi - a) / K
    A = [float(q[d]) * tri(phase([0.5 if e == d else 0.0 for e in range(3)])) for d in range(3)]
    b = _curl(A, (h, h, h))
    b = [b[d] + 0.75 * float(n[d]) + 0.3 * float(t[d]) for d in range(3)]
    left = torch.sin(phase((0.5, 0.5, 0.5))) >= 0
    one = torch.ones_like(b[0])
    zero = torch.zeros_like(one)
    return _assemble(torch.where(left, one, 0.125 * one), [zero] * 3, torch.where(left, one, 0.1 * one), b)


def _patch_dims(case, seed):
    r = np.random.default_rng(1808)               # sizes belong to the case, not to the seed
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    out = []
    while len(out) < case["npatch"]:
        e = np.clip(np.rint(np.exp(r.uniform(lo, hi, 3))), case["lo"], case["hi"]).astype(int)
        if e.max() / e.min() <= 2.0:
            out.append(tuple(int(v) for v in e))
    return out


def _cuts(case):
    return tuple([round(case[a] * i / case["cuts"] + (0.03 * case[a] if 0 < i < case["cuts"] and i % 2 else 0))
                  for i in range(case["cuts"] + 1)] for a in ("nx", "ny", "nz"))


def _initial(case, seed):
    """dims of every patch, cell sizes, cuts (or None), and the flat
    patch-major U and b (FP64 values, rounded to FP32 for FP32 grids)."""
    cuts, kind = None, case["kind"]
    if kind == "patches":
        dims, h = _patch_dims(case, seed), (1 / 64.0,) * 3
        parts = [_brio_wu(d, h[0], seed * 1009 + p) if p % 2 else _turbulence(d, h, seed * 1009 + p)
                 for p, d in enumerate(dims)]
    else:
        dims = [(case["nx"], case["ny"], case["nz"])]
        h = tuple(1.0 / n for n in dims[0])
        r = np.random.default_rng(seed)
        state = case.get("state", "turbulence")
        if state in ("turbulence", "blasts"):
            parts = [_turbulence(dims[0], h, seed, 64 if state == "blasts" else 0)]
        else:
            if state == "alfven":
                st = inputs.alfven_wave(*dims[0], amp=0.1, t=float(r.uniform(0, 1)))
            else:
                st = inputs.field_loop(case["nx"], amp=1e-3, radius=float(r.uniform(0.25, 0.35)),
                                       v=tuple(r.uniform(0.7, 1.3, 2)))
            h = (st.dx, st.dy, st.dz)
            parts = [(torch.from_numpy(st.U).to(DEV), torch.from_numpy(np.stack([st.bx, st.by, st.bz])).to(DEV))]
        if kind == "bricks":
            cuts = _cuts(case)
            U, b = parts[0]
            xs, ys, zs = cuts
            sl = [(slice(None), slice(zs[k], zs[k + 1]), slice(ys[j], ys[j + 1]), slice(xs[i], xs[i + 1]))
                  for k in range(len(zs) - 1) for j in range(len(ys) - 1) for i in range(len(xs) - 1)]
            parts = [(U[s], b[s]) for s in sl]
            dims = bricks.brick_dims(cuts)
    U = torch.cat([p[0].reshape(-1) for p in parts])
    b = torch.cat([p[1].reshape(-1) for p in parts])
    if case["precision"] != "fp64":
        U, b = U.float(), b.float()
    return dims, h, cuts, U, b


def _networks(seed):
    """Random networks near the linear weights (7 x 1379 parameters)."""
    r = np.random.default_rng(seed)
    P = []
    for _ in range(7):
        P.append(np.concatenate([(r.standard_normal((32, 6)) * 0.4).ravel(), r.standard_normal(32) * 0.1,
                                 (r.standard_normal((32, 32)) * 0.18).ravel(), r.standard_normal(32) * 0.1,
                                 (r.standard_normal((3, 32)) * 0.1).ravel(), np.log([0.1, 0.6, 0.3])]))
    return np.array(P, dtype=np.float32)


def _records(case, seed):
    """Training records (field, x[6], q[3], T, flag) of smooth and jumping stencils."""
    r = np.random.default_rng(seed)
    n = case["records"]
    m = np.arange(6)
    ph, fr, am = r.uniform(0, 2 * np.pi, n), r.uniform(0.05, 1.2, n), r.standard_normal((n, 2))
    v = np.sin(ph[:, None] + fr[:, None] * m) + 0.3 * am[:, :1] * np.cos(2 * fr[:, None] * m) \
        + np.where(r.uniform(size=n) < 0.1, 2.0, 0.02)[:, None] * r.standard_normal((n, 6))
    v = v - v.mean(1, keepdims=True)
    v /= np.abs(v).max(1, keepdims=True) + 1e-12
    q = np.stack([(2 * v[:, 0] - 7 * v[:, 1] + 11 * v[:, 2]) / 6, (-v[:, 1] + 5 * v[:, 2] + 2 * v[:, 3]) / 6,
                  (2 * v[:, 2] + 5 * v[:, 3] - v[:, 4]) / 6], 1)
    T = q @ np.array([0.1, 0.6, 0.3]) + 0.05 * r.standard_normal(n)
    rec = np.zeros((n, 12), dtype=np.float32)
    rec[:, 0] = r.integers(0, 7, n)
    rec[:, 1:7], rec[:, 7:10], rec[:, 10] = v, q, T
    rec[:, 11] = r.uniform(size=n) < 0.1
    return rec


# ---- what a program holds, and one pass ---------------------------------------------
def prepare(case, seed):
    if case["kind"] == "train":
        return {"case": case, "records": _records(case, seed), "params": _networks(seed), "seed": int(seed)}
    dims, h, cuts, U, b = _initial(case, seed)
    fp32 = case["precision"] != "fp64"
    dt = torch.float32 if fp32 else F64
    kw = {"precision": case["precision"]}
    if case["kind"] != "monitor":
        kw.update(integrator=case["integrator"], weights=case["weights"])
    if cuts is not None:
        kw["links"] = bricks.brick_links(cuts)
    g = wombat.Grid(dims, *h, U.double().cpu().numpy(), b.double().cpu().numpy(), gamma=GAMMA, **kw)
    s = {"case": case, "grid": g}
    if case["kind"] == "monitor":
        return s
    if case["precision"] == "learned":
        g.set_mlp(_networks(seed), 4.0, 0.5)
    if case.get("totals"):
        g.set_step_totals(True)
    if case["host"] == "pinned":
        def hold(t):
            o = torch.empty(t.shape, dtype=dt, pin_memory=True)
            return o.copy_(t) if t.numel() else o
        s["U"], s["b"] = hold(U), hold(b)
        s["Uo"], s["bo"] = (torch.empty(t.shape, dtype=dt, pin_memory=True) for t in (U, b))
    else:
        s["U"], s["b"] = U.cpu().numpy(), b.cpu().numpy()
    return s


def _fixed_dt(case):
    """dt of a run at a fixed step (the accuracy suites): well inside the CFL limit."""
    return 0.1 / max(case["nx"], case["ny"])


def run(s):
    case = s["case"]
    if case["kind"] == "train":
        params, hist = wombat.mlp_train(s["records"], s["params"], case["steps"], case["batch"], lr=2e-3, lam=1e-3,
                                        seed=s["seed"])
        loss, grad = wombat.mlp_loss_grad(s["records"], params, 1e-3)
        return {"params": params, "history": hist, "loss": loss, "grad": grad}
    g = s["grid"]
    if case["kind"] == "monitor":
        return {"dt": g.cfl_dt(CFL), "totals": g.totals(), "div_b": np.array(g.div_b())}
    g.set_state(s["U"], s["b"])
    if case.get("state") in ("alfven", "field_loop"):
        g.step(_fixed_dt(case), case["steps"])
    else:
        g.step_cfl(CFL, case["steps"])
    if case["host"] == "pinned":
        U, b = g.get_state(s["Uo"], s["bo"])
    else:
        U, b = g.get_state(dtype=s["U"].dtype)
    return {"U": U, "b": b, "totals": g.step_totals()} if case.get("totals") else {"U": U, "b": b}


def _cells(case):
    if case["kind"] == "patches":
        return sum(a * b * c for a, b, c in _patch_dims(case, 0))
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    if case["kind"] == "train":
        # forward 2.6, backward 5.2 kflop per record; records and parameters once
        n = 7 * case["batch"] * case["steps"] + case["records"]
        return {"bytes": 48.0 * case["records"] + 4 * 7 * 1379 * 3, "flops": 7.9e3 * n}
    n, t = _cells(case), 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "monitor":
        return {"bytes": 8.0 * n * t, "flops": 110.0 * n}
    stages = case["steps"] * (4 if case["integrator"] == "rk4" else 3)
    # 8 values in, 11 out per cell; per stage three interfaces of about 1 600
    # flops and a cell update of about 100, plus the networks' 2.6 kflop for
    # some 40 % of the 14 weight decisions of an interface
    per = 3 * (1600 + (14700 if case["precision"] == "learned" else 0)) + 100
    return {"bytes": 19.0 * n * t, "flops": float(stages) * per * n}


# ---- FP64 reference: plain torch, flat cells and neighbour tables ---------------------
class _Reference:
    def __init__(self, case, seed):
        self.case = case
        self.dims, self.h, cuts, U, b = _initial(case, seed)
        n = [a * c * d for a, c, d in self.dims]
        off = np.concatenate([[0], np.cumsum(n)])
        self.N = int(off[-1])
        new = lambda: torch.empty(self.N, dtype=torch.int64, device=DEV)      # noqa: E731
        self.up, self.dn = [new() for _ in range(3)], [new() for _ in range(3)]
        ids = [torch.arange(off[p], off[p + 1], device=DEV).reshape(d[2], d[1], d[0])
               for p, d in enumerate(self.dims)]
        if cuts is not None:               # the bricks' cells in their places in the world
            nb = [len(c) - 1 for c in cuts]
            rows = [[torch.cat([ids[a + nb[0] * (j + nb[1] * k)] for a in range(nb[0])], 2) for j in range(nb[1])]
                    for k in range(nb[2])]
            ids = [torch.cat([torch.cat(r, 1) for r in rows], 0)]
        for w in ids:
            for d in range(3):
                self.up[d][w.reshape(-1)] = torch.roll(w, -1, 2 - d).reshape(-1)
                self.dn[d][w.reshape(-1)] = torch.roll(w, 1, 2 - d).reshape(-1)
        # flat index of (field f of nf, cell) in the patch-major arrays
        self.base = torch.cat([torch.arange(m, device=DEV) for m in n])
        self.size = torch.cat([torch.full((m,), m, device=DEV) for m in n])
        self.off = torch.cat([torch.full((m,), int(o), device=DEV) for o, m in zip(off, n)])
        U, b = U.double(), b.double()
        get = lambda a, nf, f: a[nf * self.off + f * self.size + self.base]   # noqa: E731
        self.q = torch.stack([get(U, 8, f) for f in (0, 1, 2, 3, 7)] + [get(b, 3, f) for f in range(3)])
        self.mlp = torch.from_numpy(_networks(seed)).double().to(DEV) if case["precision"] == "learned" else None

    def out(self, q):
        U = torch.empty(8 * self.N, dtype=F64, device=DEV)
        b = torch.empty(3 * self.N, dtype=F64, device=DEV)
        B = self.cell_b(q)
        for f, v in enumerate([q[0], q[1], q[2], q[3], B[0], B[1], B[2], q[4]]):
            U[8 * self.off + f * self.size + self.base] = v
        for f in range(3):
            b[3 * self.off + f * self.size + self.base] = q[5 + f]
        return U, b

    def cell_b(self, q):
        return [0.5 * (q[5 + d] + q[5 + d][self.up[d]]) for d in range(3)]

    def prims(self, q):
        B = self.cell_b(q)
        v = [q[1 + d] / q[0] for d in range(3)]
        bb = B[0] ** 2 + B[1] ** 2 + B[2] ** 2
        p = (GAMMA - 1) * (q[4] - 0.5 * q[0] * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) - 0.5 * bb)
        return v, B, bb, p

    @staticmethod
    def speeds(rho, bn, b1, b2, p):
        """a^2, ca^2, cf^2, cs^2, D = cf^2 - cs^2 and t = B_perp^2 / rho, free of cancellation."""
        a2, ca2, t = GAMMA * p / rho, bn * bn / rho, (b1 * b1 + b2 * b2) / rho
        D = torch.sqrt((a2 - ca2) ** 2 + t * (2 * (a2 + ca2) + t))
        cf2 = 0.5 * (a2 + ca2 + t + D)
        return a2, ca2, cf2, torch.where(cf2 > 0, a2 * ca2 / cf2, torch.zeros_like(cf2)), D, t

    def dt(self, q):
        v, B, bb, p = self.prims(q)
        s = 0
        for d in range(3):
            cf2 = self.speeds(q[0], B[d], B[(d + 1) % 3], B[(d + 2) % 3], p)[2]
            s = s + (v[d].abs() + torch.sqrt(cf2)) / self.h[d]
        return CFL / float(s.max())

    def phi_js(self, a, b, c, d):
        i0 = 13 * (a - b) ** 2 + 3 * (a - 3 * b) ** 2
        i1 = 13 * (b - c) ** 2 + 3 * (b + c) ** 2
        i2 = 13 * (c - d) ** 2 + 3 * (3 * c - d) ** 2
        if self.case["weights"] == "z":
            tau = (i0 - i2).abs()
            a0, a1, a2 = 1 + tau / (EPS + i0), 6 * (1 + tau / (EPS + i1)), 3 * (1 + tau / (EPS + i2))
        else:
            a0, a1, a2 = (EPS + i0) ** -2, 6 * (EPS + i1) ** -2, 3 * (EPS + i2) ** -2
        r = 1 / (a0 + a1 + a2)
        ph = a0 * r * (a - 2 * b + c) / 3 + (a2 * r - 0.5) * (b - 2 * c + d) / 6
        return ph, (i0, i1, i2)

    def phi(self, s, v, pjump):
        """phi_N of one side: v the six split fluxes in upwind order."""
        D = [v[k + 1] - v[k] for k in range(4)]
        ph, IS = self.phi_js(*D)
        if self.mlp is None:
            return ph
        ab = torch.stack([x.abs() for x in D])
        mx = ab.max(0).values
        I3 = torch.stack(IS)
        js = pjump | (mx > 4.0 * (ab.sum(0) - mx) / 3 + 1e-30)
        js = js | ~(EPS + I3.max(0).values > 1.03 * (EPS + I3.min(0).values))
        V = torch.stack(v)
        V = V - V.mean(0)
        x = (V / (V.abs().max(0).values + 1e-12)).T
        P = self.mlp[s]
        W1, b1, W2 = P[:192].reshape(32, 6), P[192:224], P[224:1248].reshape(32, 32)
        b2, W3, b3 = P[1248:1280], P[1280:1376].reshape(3, 32), P[1376:]
        gelu = lambda z: z * torch.sigmoid(1.702 * z)                         # noqa: E731
        om = torch.softmax(gelu(gelu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3, 1)
        net = om[:, 0] * (D[0] - 2 * D[1] + D[2]) / 3 + (om[:, 2] - 0.5) * (D[1] - 2 * D[2] + D[3]) / 6
        return torch.where(js, ph, net)

    def sweep(self, q, n):
        """Fluxes (rho, mx, my, mz, E, B_t1, B_t2) through the lower faces along axis n."""
        t1, t2 = (n + 1) % 3, (n + 2) % 3
        v, B, bb, p = self.prims(q)
        u, v1, v2, bn, b1, b2 = v[n], v[t1], v[t2], B[n], B[t1], B[t2]
        pt, vb = p + 0.5 * bb, u * bn + v1 * b1 + v2 * b2
        U = torch.stack([q[0], q[1 + n], q[1 + t1], q[1 + t2], b1, b2, q[4]])
        F = torch.stack([q[1 + n], q[1 + n] * u + pt - bn * bn, q[1 + t1] * u - bn * b1, q[1 + t2] * u - bn * b2,
                         u * b1 - v1 * bn, u * b2 - v2 * bn, (q[4] + pt) * u - bn * vb])
        a2, ca2, cf2, cs2, _, _ = self.speeds(q[0], bn, b1, b2, p)
        c = [cf2.sqrt(), ca2.sqrt(), cs2.sqrt()]
        lam = torch.stack([u - c[0], u - c[1], u - c[2], u, u + c[2], u + c[1], u + c[0]]).abs()
        W = torch.stack([q[0], u, v1, v2, bn, b1, b2, p])
        out = torch.empty(7, self.N, dtype=F64, device=DEV)
        step = 1 << 20 if self.mlp is not None else 1 << 22
        for c0 in range(0, self.N, step):
            at = torch.arange(c0, min(self.N, c0 + step), device=DEV)
            st = [None] * 6
            st[3] = at
            for m in (2, 1, 0):
                st[m] = self.dn[n][st[m + 1]]
            for m in (4, 5):
                st[m] = self.up[n][st[m - 1]]
            f = self.interface(U, F, lam, W, st)
            g = [None] * 7
            g[0], g[4], g[5], g[6] = f[0], f[6], f[4], f[5]
            g[1 + n], g[1 + t1], g[1 + t2] = f[1], f[2], f[3]
            out[:, c0:c0 + len(at)] = torch.stack(g)
        return out

    def interface(self, U, F, lam, W, st):
        rho, u, v1, v2, bn, b1, b2, p = 0.5 * (W[:, st[2]] + W[:, st[3]])
        a2, ca2, cf2, cs2, D, t = self.speeds(rho, bn, b1, b2, p)
        bp2 = b1 * b1 + b2 * b2
        bt2 = bn * bn + bp2
        w = bp2 > 1e-24 * bt2.clamp(min=1.0)
        ib = torch.where(w, bp2, torch.ones_like(bp2)).rsqrt()
        half = torch.full_like(b1, math.sqrt(0.5))
        be1, be2 = torch.where(w, b1 * ib, half), torch.where(w, b2 * ib, half)
        x, y = 0.5 * (D + (a2 - ca2) - t), 0.5 * (D - (a2 - ca2) + t)
        big = x >= y
        x, y = torch.where(big, x, a2 * t / y), torch.where(big, a2 * t / x, y)
        deg = D <= 1e-12 * (a2 + bt2 / rho)
        one, zero = torch.ones_like(D), torch.zeros_like(D)
        iD = 1 / torch.where(deg, one, D)
        hot = torch.where(a2 >= ca2, one, zero)
        af = torch.where(deg, hot, (x * iD).clamp(min=0).sqrt())
        as_ = torch.where(deg, 1 - hot, (y * iD).clamp(min=0).sqrt())
        a, cf, cs, ca, sr = a2.sqrt(), cf2.sqrt(), cs2.sqrt(), ca2.sqrt(), rho.sqrt()
        S = torch.where(bn >= 0, one, -one)
        g1 = GAMMA - 1
        X = 2 * rho * (af ** 2 * cf2 + as_ ** 2 * cs2)
        hv2 = 0.5 * (u * u + v1 * v1 + v2 * v2)
        # left eigenvectors acting on conserved differences: primitive
        # differences at the interface state, then the Roe-Balsara rows
        al = []
        cc = {0: -cf, 1: -ca, 2: -cs, 3: zero, 4: cs, 5: ca, 6: cf}
        for s in range(7):
            m = (u + cc[s]).abs()
            for k in st:
                m = torch.maximum(m, lam[s, k])
            al.append(m)
        pr = W[7]
        pjump = None
        if self.mlp is not None:
            ps = torch.stack([pr[k] for k in st])
            pjump = ps.max(0).values > 1.5 * ps.min(0).values

        def project(z):
            du, d1, d2 = (z[1] - u * z[0]) / rho, (z[2] - v1 * z[0]) / rho, (z[3] - v2 * z[0]) / rho
            dp = g1 * (z[6] + hv2 * z[0] - u * z[1] - v1 * z[2] - v2 * z[3] - b1 * z[4] - b2 * z[5])
            vpar, vper = be1 * d1 + be2 * d2, be1 * d2 - be2 * d1
            bpar, bper = be1 * z[4] + be2 * z[5], be1 * z[5] - be2 * z[4]
            f1 = rho * (af * cf * du - as_ * cs * S * vpar) / X
            f2 = as_ * bpar / (2 * a * sr) + af * dp / (2 * rho * a2)
            s1 = rho * (as_ * cs * du + af * cf * S * vpar) / X
            s2 = -af * bpar / (2 * a * sr) + as_ * dp / (2 * rho * a2)
            w1, w2 = 0.5 * vper, 0.5 * S * bper / sr
            return [f2 - f1, w1 + w2, s2 - s1, z[0] - dp / a2, s2 + s1, w1 - w2, f2 + f1]
        pu = [project(U[:, k]) for k in st]
        pf = [project(F[:, k]) for k in st]
        cor = []
        for s in range(7):
            gp = [0.5 * (pf[m][s] + al[s] * pu[m][s]) for m in range(6)]
            gm = [0.5 * (pf[m][s] - al[s] * pu[m][s]) for m in range(6)][::-1]
            # the reversed minus side's differences are -D-, and phi is odd
            cor.append(-self.phi(s, gm, pjump) - self.phi(s, gp, pjump))
        # right eigenvectors in primitive variables, then dU/dW
        fp, fm, sp, sm = cor[6] + cor[0], cor[6] - cor[0], cor[4] + cor[2], cor[4] - cor[2]
        ap, am = cor[5] + cor[1], cor[5] - cor[1]
        fs = af * fp + as_ * sp
        dr = rho * fs + cor[3]
        du = af * cf * fm + as_ * cs * sm
        vpar = S * (af * cf * sm - as_ * cs * fm)
        bpar = a * sr * (as_ * fp - af * sp)
        bper = -S * sr * am
        dp = rho * a2 * fs
        d1, d2 = be1 * vpar - be2 * ap, be2 * vpar + be1 * ap
        e1, e2 = be1 * bpar - be2 * bper, be2 * bpar + be1 * bper
        cen = (7 * (F[:, st[2]] + F[:, st[3]]) - (F[:, st[1]] + F[:, st[4]])) / 12
        return [cen[0] + dr, cen[1] + u * dr + rho * du, cen[2] + v1 * dr + rho * d1, cen[3] + v2 * dr + rho * d2,
                cen[4] + e1, cen[5] + e2,
                cen[6] + hv2 * dr + rho * (u * du + v1 * d1 + v2 * d2) + b1 * e1 + b2 * e2 + dp / g1]

    def rate(self, q):
        F = [self.sweep(q, n) for n in range(3)]
        up, dn = self.up, self.dn
        L = torch.zeros_like(q)
        for d in range(3):
            L[:5] -= (F[d][:5][:, up[d]] - F[d][:5]) / self.h[d]
        v, B, _, _ = self.prims(q)
        E = []
        for d in range(3):
            e, f = (d + 1) % 3, (d + 2) % 3
            # E_d on the edge: -F_e(B_f) on the two e faces, F_f(B_e) on the two f faces
            P, Q = -F[e][5], F[f][6]
            c = v[f] * B[e] - v[e] * B[f]
            E.append(0.5 * (P + P[dn[f]] + Q + Q[dn[e]]) - 0.25 * (c + c[dn[e]] + c[dn[f]] + c[dn[e]][dn[f]]))
        for d in range(3):
            e, f = (d + 1) % 3, (d + 2) % 3
            L[5 + d] = -((E[f][up[e]] - E[f]) / self.h[e] - (E[e][up[f]] - E[e]) / self.h[f])
        return L

    def advance(self):
        q, case = self.q, self.case
        for _ in range(case["steps"]):
            self.start = q
            dt = _fixed_dt(case) if case.get("state") in ("alfven", "field_loop") else self.dt(q)
            if case["integrator"] == "rk4":
                k1 = self.rate(q)
                k2 = self.rate(q + 0.5 * dt * k1)
                k3 = self.rate(q + 0.5 * dt * k2)
                q = q + dt / 6 * (k1 + 2 * k2 + 2 * k3 + self.rate(q + dt * k3))
            else:
                a = q + dt * self.rate(q)
                a = 0.75 * q + 0.25 * (a + dt * self.rate(a))
                q = q / 3 + 2 / 3 * (a + dt * self.rate(a))
        return q

    def totals(self, q):
        s = q.sum(1) * (self.h[0] * self.h[1] * self.h[2])
        return s[[0, 1, 2, 3, 5, 6, 7, 4]]


def _exact_train(case, seed):
    rec, par = _records(case, seed), torch.from_numpy(_networks(seed)).double().to(DEV)
    d = torch.tensor([0.1, 0.6, 0.3], dtype=F64, device=DEV)
    by = [torch.from_numpy(rec[(rec[:, 0] == f) & (rec[:, 11] == 0)]).double().to(DEV) for f in range(7)]

    def loss_grad(p, r):
        p = p.detach().requires_grad_(True)
        g = lambda z: z * torch.sigmoid(1.702 * z)                            # noqa: E731
        z = g(r[:, 1:7] @ p[:192].reshape(32, 6).T + p[192:224])
        z = g(z @ p[224:1248].reshape(32, 32).T + p[1248:1280])
        w = torch.softmax(z @ p[1280:1376].reshape(3, 32).T + p[1376:], 1)
        lo = (((w * r[:, 7:10]).sum(1) - r[:, 10]) ** 2 + lam * (d * (d.log() - w.log())).sum(1)).mean()
        return lo.detach(), torch.autograd.grad(lo, p)[0]

    lam = float(np.float32(1e-3))
    m, v = torch.zeros_like(par), torch.zeros_like(par)
    lr, b1, b2 = float(np.float32(2e-3)), float(np.float32(0.9)), float(np.float32(0.999))
    hist = torch.zeros(case["steps"], 7, dtype=F64)
    old = np.seterr(over="ignore")

    def mix(z):                        # splitmix64
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))
    slot = np.arange(case["batch"], dtype=np.uint64)
    for t in range(case["steps"]):
        grad = torch.empty_like(par)
        for f in range(7):
            h = mix(np.uint64(seed) ^ mix(np.uint64(t * 131071 + f * 8191) + slot))
            pick = torch.from_numpy((h % np.uint64(len(by[f]))).astype(np.int64)).to(DEV)
            hist[t, f], grad[f] = loss_grad(par[f], by[f][pick])
        m, v = b1 * m + (1 - b1) * grad, b2 * v + (1 - b2) * grad * grad
        par = par - lr * (m / (1 - b1 ** (t + 1))) / ((v / (1 - b2 ** (t + 1))).sqrt() + 1e-8)
    np.seterr(**old)
    full = [loss_grad(par[f], by[f]) for f in range(7)]
    return {"params": par, "history": hist, "loss": torch.stack([x[0] for x in full]),
            "grad": torch.stack([x[1] for x in full])}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "monitor":
        r = _Reference(case, seed)
        div = sum((r.q[5 + d][r.up[d]] - r.q[5 + d]) / r.h[d] for d in range(3)).abs().max()
        return {"dt": r.dt(r.q), "totals": r.totals(r.q), "div_b": torch.stack([div, r.q[5:].abs().max()])}
    stages = case["steps"] * (4 if case["integrator"] == "rk4" else 3)
    if _cells(case) * stages * (8 if case["precision"] == "learned" else 1) > 3.2e8:
        return None
    r = _Reference(case, seed)
    q = r.advance()
    U, b = r.out(q)
    if case.get("totals"):            # of the last step's start state
        return {"U": U, "b": b, "totals": r.totals(r.start)}
    return {"U": U, "b": b}
