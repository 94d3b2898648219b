"""The calls of this library that are timed and compared: what each is, its
inputs, one pass through the public entry points, and its result in 64 bits.

A case is a dict of plain values; ``kind`` names the path:

  mesh      batched solves along one or more axes of a 2D / 3D mesh (trid.solve)
  varlen    systems of different lengths in one call (trid.solve_varlen)
  adi       time steps of one mesh (trid.adi_step)
  adi_batch time steps of many small meshes (trid.adi_step_batched)
  grad      a differentiable solve, forward and backward (tridiag_solve)
  adi2d     a training step through 2D ADI with a diffusivity field (adi2d)

Coefficients follow the recipe of the library's own inputs (diagonally
dominant, margin at least 0.5); ADI fields are sums of sine eigenmodes.  All
inputs are made on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2201_03950_gb300 import trid
from paper_2201_03950_gb300.autograd import adi2d, tridiag_solve

DEV = "cuda"
DT = {"f32": torch.float32, "f64": torch.float64}
ESZ = {"f32": 4, "f64": 8}


def listed():
    return [
        # the smallest use: 64 systems of 64 rows along x, then y; latency of two calls
        {"name": "mesh_64x64_f32", "kind": "mesh", "dims": "64,64", "axes": "xy", "dtype": "f32",
         "acc": False},
        # the ordinary use: each direction of a 256^3 mesh, single precision ...
        {"name": "mesh_256cube_f32", "kind": "mesh", "dims": "256,256,256", "axes": "xyz",
         "dtype": "f32", "acc": False},
        # ... and double precision
        {"name": "mesh_256cube_f64", "kind": "mesh", "dims": "256,256,256", "axes": "xyz",
         "dtype": "f64", "acc": False},
        # a mesh of no convenient size (rows that are no multiple of 16 bytes, odd
        # lines), each direction adding into the field, as the end of an ADI step does
        {"name": "mesh_201x187x233_f32_acc", "kind": "mesh", "dims": "201,187,233", "axes": "xyz",
         "dtype": "f32", "acc": True},
        # few, long systems: both directions of a large 2D mesh, single precision
        {"name": "mesh_4096sq_f32", "kind": "mesh", "dims": "4096,4096", "axes": "xy",
         "dtype": "f32", "acc": False},
        # long systems in double precision, neither direction a power of two
        {"name": "mesh_3000x1400_f64", "kind": "mesh", "dims": "3000,1400", "axes": "xy",
         "dtype": "f64", "acc": False},
        # uneven batch: 8192 systems of 16 to 16384 rows
        {"name": "varlen_8192_f32", "kind": "varlen", "nsys": 8192, "lo": 16, "hi": 16384,
         "dtype": "f32"},
        # heat diffusion on one large mesh, 100 time steps in one call
        {"name": "adi_256cube_100_f32", "kind": "adi", "dims": "256,256,256", "lam": 0.1,
         "steps": 100, "dtype": "f32"},
        # many small 3D meshes stepped together
        {"name": "adi_48cube_x72_f32", "kind": "adi_batch", "dims": "48,48,48", "nb": 72,
         "lam": 0.1, "steps": 100, "dtype": "f32"},
        # many small 2D meshes stepped together
        {"name": "adi_96sq_x3000_f32", "kind": "adi_batch", "dims": "96,96", "nb": 3000,
         "lam": 0.1, "steps": 120, "dtype": "f32"},
        # a solve inside a trained model: forward and the gradients of a, b, c and d
        {"name": "grad_256cube_z_f32", "kind": "grad", "dims": "256,256,256", "axes": "z",
         "dtype": "f32"},
        # fitting a diffusivity field: 50 steps forward, checkpoints every 10, backward
        {"name": "adi2d_1024sq_50_f32", "kind": "adi2d", "dims": "1024,1024", "lam": 0.2,
         "steps": 50, "every": 10, "dtype": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, lo, hi):
    """An extent of [lo, hi], log-uniform; every other one a multiple of 8."""
    n = _log_int(rng, lo, hi)
    if rng.random() < 0.5:
        n = max(lo, min(hi // 8 * 8, (n + 4) // 8 * 8))
    return n


def _text(dims):
    return ",".join(str(n) for n in dims)


def draw(rng):
    dtype = "f64" if rng.random() < 0.3 else "f32"
    r = rng.random()
    if r < 0.3:    # a 3D mesh
        dims = [_extent(rng, 16, 256) for _ in range(3)]
        return {"kind": "mesh", "dims": _text(dims), "axes": rng.choice(["x", "y", "z", "xyz"]),
                "dtype": dtype, "acc": rng.random() < 0.25}
    if r < 0.45:   # a 2D mesh, systems up to 8000 rows, at most 16M unknowns
        nx, ny = _extent(rng, 32, 8000), _extent(rng, 32, 8000)
        if nx * ny > 1 << 24:
            ny = max(32, (1 << 24) // nx)
        return {"kind": "mesh", "dims": _text([nx, ny]), "axes": rng.choice(["x", "y", "xy"]),
                "dtype": dtype, "acc": rng.random() < 0.25}
    if r < 0.55:
        lo = _log_int(rng, 2, 64)
        hi = _log_int(rng, 256, 16384)
        return {"kind": "varlen", "nsys": _log_int(rng, 64, 8192), "lo": lo, "hi": hi,
                "dtype": dtype}
    lam = rng.choice([0.05, 0.1, 0.1, 0.2, 0.3])
    if r < 0.7:
        return {"kind": "adi", "dims": _text([_extent(rng, 24, 256) for _ in range(3)]),
                "lam": lam, "steps": rng.randint(1, 40), "dtype": dtype}
    if r < 0.85:
        if rng.random() < 0.5:
            return {"kind": "adi_batch", "dims": _text([_extent(rng, 16, 96) for _ in range(3)]),
                    "nb": rng.choice([8, 24, 24, 72]), "lam": lam, "steps": rng.randint(5, 40),
                    "dtype": dtype}
        return {"kind": "adi_batch", "dims": _text([_extent(rng, 32, 128) for _ in range(2)]),
                "nb": _log_int(rng, 100, 2000), "lam": lam, "steps": rng.randint(10, 40),
                "dtype": dtype}
    if r < 0.94:
        dims = [_extent(rng, 16, 256) for _ in range(3)]
        return {"kind": "grad", "dims": _text(dims), "axes": rng.choice("xyz"), "dtype": dtype}
    return {"kind": "adi2d", "dims": _text([_extent(rng, 64, 1024) for _ in range(2)]),
            "lam": 0.2, "steps": rng.randint(10, 50), "every": 10, "dtype": dtype}


# ---- inputs -----------------------------------------------------------------
def _dims(case):
    return tuple(int(v) for v in case["dims"].split(","))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(n, g):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _system(n, g, dt, nrhs=1):
    """a, b, c and nrhs right-hand sides, drawn in 64 bits and rounded once."""
    a = -0.1 - 0.9 * _rand(n, g)
    c = -0.1 - 0.9 * _rand(n, g)
    b = a.abs() + c.abs() + 0.5 + _rand(n, g)
    d = [(2.0 * _rand(n, g) - 1.0).to(dt) for _ in range(nrhs)]
    return a.to(dt), b.to(dt), c.to(dt), d


def _sine_fields(dims, nb, rng, dt, kmax=16):
    """nb fields, each a sum of three Dirichlet sine eigenmodes (x contiguous)."""
    total = None
    for _ in range(3):
        term = torch.as_tensor(rng.uniform(0.5, 1.5, nb), device=DEV).reshape(
            [nb] + [1] * len(dims))
        for ax, n in enumerate(dims):
            k = torch.as_tensor(rng.integers(1, max(2, min(kmax, n - 2) + 1), nb), device=DEV)
            i = torch.arange(n, device=DEV, dtype=torch.float64)
            s = torch.sin(math.pi * k[:, None] * i / (n - 1))
            s[:, 0] = 0.0
            s[:, -1] = 0.0
            shape = [nb] + [1] * len(dims)
            shape[len(dims) - ax] = n
            term = term * s.reshape(shape)
        total = term if total is None else total + term
    return total.reshape(-1).to(dt)


def _lengths(case, rng):
    """Log-uniform lengths in random order; the same lengths for every seed."""
    n, lo, hi = case["nsys"], case["lo"], case["hi"]
    u = (np.arange(n) + 0.5) / n
    v = np.clip(np.rint(np.exp(math.log(lo) + u * math.log(hi / lo))), lo, hi).astype(np.int64)
    return v if rng is None else rng.permutation(v)


def _kappa(nx, ny, rng):
    """exp of Gaussian noise, smoothed by three passes of a 3 x 3 box."""
    k = torch.as_tensor(np.exp(rng.normal(0.0, 0.3, (ny, nx))), device=DEV)
    for _ in range(3):
        p = torch.nn.functional.pad(k[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        k = sum(p[1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]
                for dy in (-1, 0, 1) for dx in (-1, 0, 1)) / 9.0
    return k.reshape(-1)


def prepare(case, seed):
    kind, dt = case["kind"], DT[case["dtype"]]
    g, rng = _gen(seed), np.random.default_rng(int(seed))
    s = {"kind": kind}
    if kind == "varlen":
        lens = _lengths(case, rng)
        off = np.concatenate([[0], np.cumsum(lens)])
        a, b, c, d = _system(int(off[-1]), g, dt)
        s.update(a=a, b=b, c=c, d=d[0], offsets=torch.from_numpy(off).to(DEV),
                 max_len=int(lens.max()),
                 ws=torch.empty(trid.varlen_workspace_bytes(len(lens)), dtype=torch.uint8,
                                device=DEV))
        return s
    dims = _dims(case)
    n = math.prod(dims)
    s["dims"] = dims
    if kind == "mesh":
        s["axes"] = ["xyz".index(k) for k in case["axes"]]
        a, b, c, s["d"] = _system(n, g, dt, len(s["axes"]))
        s["u"] = (2.0 * _rand(n, g) - 1.0).to(dt) if case["acc"] else None
        # scratch for lines that need some, kept by the caller (0 bytes for short lines)
        need = max(trid.solve_workspace_bytes(dims, k, dt) for k in s["axes"])
        s["ws"] = torch.empty(need, dtype=torch.uint8, device=DEV) if need else None
        s.update(a=a, b=b, c=c)
    elif kind == "adi":
        s.update(u=_sine_fields(dims, 1, rng, dt), lam=case["lam"], steps=case["steps"],
                 ws=torch.empty(trid.adi_workspace_bytes(dims, dt), dtype=torch.uint8, device=DEV))
    elif kind == "adi_batch":
        s.update(u=_sine_fields(dims, case["nb"], rng, dt), lam=case["lam"], steps=case["steps"],
                 nb=case["nb"])
    elif kind == "grad":
        a, b, c, (d, gx) = _system(n, g, dt, 2)
        s.update(a=a.requires_grad_(), b=b.requires_grad_(), c=c.requires_grad_(),
                 d=d.requires_grad_(), gx=gx, axis="xyz".index(case["axes"]))
    else:
        s.update(u0=_sine_fields(dims, 1, rng, dt).requires_grad_(),
                 kappa=_kappa(*dims, rng).to(dt).requires_grad_(),
                 target=_sine_fields(dims, 1, rng, dt),
                 lam=case["lam"], steps=case["steps"], every=case["every"])
    return s


# ---- one pass ---------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "mesh":
        if s["u"] is None:      # each direction overwrites its right-hand side
            return [trid.solve(s["a"], s["b"], s["c"], d, s["dims"], k, workspace=s["ws"])
                    for k, d in zip(s["axes"], s["d"])]
        for k, d in zip(s["axes"], s["d"]):   # each direction adds into one field
            trid.solve(s["a"], s["b"], s["c"], d, s["dims"], k, u=s["u"], workspace=s["ws"])
        return s["u"]
    if kind == "varlen":
        return trid.solve_varlen(s["a"], s["b"], s["c"], s["d"], s["offsets"], s["max_len"],
                                 workspace=s["ws"])
    if kind == "adi":
        return trid.adi_step(s["u"], s["dims"], s["lam"], s["steps"], s["ws"])
    if kind == "adi_batch":
        return trid.adi_step_batched(s["u"], s["nb"], s["dims"], s["lam"], s["steps"])
    if kind == "grad":
        leaves = (s["a"], s["b"], s["c"], s["d"])
        x = tridiag_solve(*leaves, s["dims"], s["axis"])
        return (x.detach(),) + torch.autograd.grad(x, leaves, s["gx"])
    uT = adi2d(s["u0"], s["kappa"], s["dims"], s["lam"], s["steps"], s["every"])
    loss = torch.mean((uT - s["target"]) ** 2)
    gu, gk = torch.autograd.grad(loss, (s["u0"], s["kappa"]))
    return {"uT": uT.detach(), "g_u0": gu, "g_kappa": gk}


# ---- what a pass cannot do without ------------------------------------------
def work(case):
    """Solves: a, b, c, d read and x written (the accumulated field read too),
    Thomas' 8 operations per unknown.  ADI: the field read and written by every
    step, or by the call where one mesh fits an SM's shared memory."""
    w = ESZ[case["dtype"]]
    kind = case["kind"]
    if kind == "varlen":
        n = int(_lengths(case, None).sum())
        return {"bytes": 5 * w * n, "flops": 8 * n}
    dims = _dims(case)
    n = math.prod(dims)
    if kind == "mesh":
        k = len(case["axes"])
        return {"bytes": (6 if case["acc"] else 5) * w * n * k, "flops": 8 * n * k}
    if kind == "grad":   # forward 5 words; backward a, b, c, x, g_x read, four gradients written
        return {"bytes": 14 * w * n, "flops": 19 * n}
    ops = 1 + (2 * len(dims) + 2) + 5 * len(dims)   # stencil, line solves, update
    if kind == "adi":
        return {"bytes": 2 * w * n * case["steps"], "flops": ops * n * case["steps"]}
    if kind == "adi_batch":
        passes = 1 if n * w <= 200 * 1024 else case["steps"]
        return {"bytes": 2 * w * n * case["nb"] * passes,
                "flops": ops * n * case["nb"] * case["steps"]}
    # adi2d: u0, kappa, target, uT, two gradients, and each checkpoint written and read
    cks = -(-case["steps"] // case["every"])
    return {"bytes": (6 + 2 * cks) * w * n, "flops": (2 * 24 + 50) * n * case["steps"]}


def tolerance(case):
    """About four times the distance from the 64-bit result that was measured:
    solves and their gradients 0.5e-7 to 1.3e-7 (32 bits) and 1.9e-16 (64 bits);
    up to 100 ADI steps 3.5e-6, each step rounding the field and the constant
    operator's factors once more; the gradients through 50 steps 1.1e-6.  In
    64 bits the same multiples of the unit roundoff."""
    unit = 2.0 ** -53 if case["dtype"] == "f64" else 2.0 ** -24
    many = {"adi": 200, "adi_batch": 200, "adi2d": 80}
    return {"rel": many.get(case["kind"], 10) * unit}


# ---- the result in 64 bits --------------------------------------------------
def _thomas(a, b, c, d):
    """x of tridiagonal systems along dim 0 (64 bits, all systems at once)."""
    n = d.shape[0]
    cs, ds = torch.empty_like(d), torch.empty_like(d)
    cs[0], ds[0] = c[0] / b[0], d[0] / b[0]
    for i in range(1, n):
        m = 1.0 / torch.addcmul(b[i], a[i], cs[i - 1], value=-1.0)
        torch.mul(c[i], m, out=cs[i])
        torch.mul(torch.addcmul(d[i], a[i], ds[i - 1], value=-1.0), m, out=ds[i])
    for i in range(n - 2, -1, -1):
        ds[i].addcmul_(cs[i], ds[i + 1], value=-1.0)
    return ds


def _lines(v, dims, k):
    """A flat mesh array as [rows along axis k, systems]."""
    return v.detach().double().reshape(tuple(reversed(dims))).movedim(len(dims) - 1 - k, 0) \
        .contiguous()


def _flat(v, dims, k):
    return v.movedim(0, len(dims) - 1 - k).reshape(-1)


def _solve_exact(s, d, k):
    dims = s["dims"]
    return _flat(_thomas(*(_lines(v, dims, k) for v in (s["a"], s["b"], s["c"], d))), dims, k)


def _operator_inverse(n, lam):
    m = torch.eye(n, dtype=torch.float64, device=DEV)
    i = torch.arange(1, n - 1, device=DEV)
    m[i, i] = 1.0 + 2.0 * lam
    m[i, i - 1] = -lam
    m[i, i + 1] = -lam
    return torch.linalg.inv(m)


def _adi_exact(u, dims, nb, lam, steps):
    u = u.double().reshape([nb] + list(reversed(dims)))
    nd = len(dims)
    inv = [_operator_inverse(n, lam) for n in dims]
    core = (slice(None),) + (slice(1, -1),) * nd
    for _ in range(steps):
        d = torch.zeros_like(u)
        acc = -2.0 * nd * u[core]
        for ax in range(1, nd + 1):
            for sl in (slice(0, -2), slice(2, None)):
                acc = acc + u[core[:ax] + (sl,) + core[ax + 1:]]
        d[core] = lam * acc
        for k in range(nd):
            d = torch.matmul(d.movedim(nd - k, -1), inv[k].T).movedim(-1, nd - k)
        u = u + d
    return u.reshape(-1)


class _Line:
    """Thomas with the pivots kept, along axis 0 of numpy arrays."""

    def __init__(self, a, b, c):
        self.a, self.m, self.cs = a, np.empty_like(b), np.empty_like(b)
        prev = 0.0
        for i in range(b.shape[0]):
            self.m[i] = 1.0 / (b[i] - a[i] * prev)
            prev = self.cs[i] = c[i] * self.m[i]

    def __call__(self, d):
        x = d * self.m
        q = self.a * self.m
        for i in range(1, x.shape[0]):
            x[i] -= q[i] * x[i - 1]
        for i in range(x.shape[0] - 2, -1, -1):
            x[i] -= self.cs[i] * x[i + 1]
        return x


def _axis_operator(kap, lam):
    """a, b, c along axis 0: faces are node means, the end rows identities."""
    face = 0.5 * (kap[:-1] + kap[1:])
    a, c, b = np.zeros_like(kap), np.zeros_like(kap), np.ones_like(kap)
    a[1:-1], c[1:-1] = -lam * face[:-1], -lam * face[1:]
    b[1:-1] = 1.0 - a[1:-1] - c[1:-1]
    return a, b, c


def _transposed(a, b, c):
    at, ct = np.zeros_like(a), np.zeros_like(a)
    at[1:], ct[:-1] = c[:-1], a[1:]
    return at, b, ct


def _adi2d_exact(s):
    nx, ny = s["dims"]
    u, kap, tgt = (s[k].detach().double().cpu().numpy().reshape(ny, nx)
                   for k in ("u0", "kappa", "target"))
    # axis 0 of every array is the line: index 0 = y lines [ny, nx], 1 = x lines [nx, ny]
    op = [_axis_operator(kap, s["lam"]), _axis_operator(np.ascontiguousarray(kap.T), s["lam"])]
    fwd, rev = [_Line(*o) for o in op], [_Line(*_transposed(*o)) for o in op]
    turn = lambda v: np.ascontiguousarray(v.T)   # noqa: E731

    def inside(v):
        w = np.zeros_like(v)
        w[1:-1, 1:-1] = v[1:-1, 1:-1]
        return w

    def stencil(o, v):
        a, _, c = o
        d = np.zeros_like(v)
        d[1:-1] = a[1:-1] * (v[1:-1] - v[:-2]) - c[1:-1] * (v[2:] - v[1:-1])
        return d

    states = []
    for _ in range(s["steps"]):
        d = inside(stencil(op[0], u) + stencil(op[1], turn(u)).T)
        w = fwd[1](turn(d))
        dl = fwd[0](turn(w))
        states.append((u, w, dl))
        u = u + dl
    uT = u
    g = 2.0 * (uT - tgt) / uT.size
    acc = [[np.zeros_like(o[0]) for _ in range(3)] for o in op]

    def coef(k, gd, x, v, gi):
        """The gradients of axis k's a, b, c: of the solve (x its solution) and,
        with gi the explicit part's gradient, of the stencil on v."""
        ga, gb, gc = acc[k]
        ga[1:-1] += gi[1:-1] * (v[1:-1] - v[:-2]) - gd[1:-1] * x[:-2]
        gb[1:-1] -= gd[1:-1] * x[1:-1]
        gc[1:-1] += gi[1:-1] * (v[1:-1] - v[2:]) - gd[1:-1] * x[2:]

    def stencil_t(o, gi):
        a, _, c = o
        r = np.zeros_like(gi)
        r[1:-1] += (a[1:-1] + c[1:-1]) * gi[1:-1]
        r[:-2] -= a[1:-1] * gi[1:-1]
        r[2:] -= c[1:-1] * gi[1:-1]
        return r

    for u, w, dl in reversed(states):
        gw = rev[0](g)
        gd = rev[1](turn(gw))
        gi = inside(gd)
        coef(0, gw, dl, u, turn(gi))
        coef(1, gd, w, turn(u), gi)
        g = g + stencil_t(op[0], turn(gi)) + stencil_t(op[1], gi).T
    gk = 0.0
    for k in (0, 1):
        ga, gb, gc = acc[k]
        face = s["lam"] * ((gb - ga)[1:-1]), s["lam"] * ((gb - gc)[1:-1])
        gf = np.zeros((ga.shape[0] - 1, ga.shape[1]))
        gf[:-1] += face[0]
        gf[1:] += face[1]
        node = np.zeros_like(ga)
        node[:-1] += 0.5 * gf
        node[1:] += 0.5 * gf
        gk = gk + (node if k == 0 else node.T)
    return {"uT": uT.reshape(-1), "g_u0": g.reshape(-1), "g_kappa": np.ascontiguousarray(gk)
            .reshape(-1)}


def exact(case, seed):
    s = prepare(case, seed)
    kind = s["kind"]
    if kind == "mesh":
        xs = [_solve_exact(s, d, k) for k, d in zip(s["axes"], s["d"])]
        return xs if s["u"] is None else s["u"].double() + sum(xs)
    if kind == "varlen":
        off = s["offsets"]
        lens = off[1:] - off[:-1]
        row = torch.arange(int(lens.max()), device=DEV)[:, None]
        at = torch.where(row < lens, off[:-1] + row, -1)     # [rows, systems], -1 = padding
        pick = [torch.where(at >= 0, v.double()[at], fill)
                for v, fill in ((s["a"], 0.0), (s["b"], 1.0), (s["c"], 0.0), (s["d"], 0.0))]
        pick[0][0] = 0.0
        pick[2][lens - 1, torch.arange(len(lens), device=DEV)] = 0.0
        x = _thomas(*pick)
        out = torch.empty(s["d"].numel(), dtype=torch.float64, device=DEV)
        out[at[at >= 0]] = x[at >= 0]
        return out
    if kind in ("adi", "adi_batch"):
        return _adi_exact(s["u"], s["dims"], s.get("nb", 1), s["lam"], s["steps"])
    if kind == "adi2d":
        return _adi2d_exact(s)
    dims, k = s["dims"], s["axis"]
    a, b, c, d, gx = (_lines(s[v], dims, k) for v in ("a", "b", "c", "d", "gx"))
    x = _thomas(a, b, c, d)
    at, ct = torch.zeros_like(a), torch.zeros_like(a)
    at[1:], ct[:-1] = c[:-1], a[1:]
    gd = _thomas(at, b, ct, gx)
    ga, gb, gc = torch.zeros_like(a), -gd * x, torch.zeros_like(a)
    ga[1:] = -gd[1:] * x[:-1]
    gc[:-1] = -gd[:-1] * x[1:]
    return tuple(_flat(v, dims, k) for v in (x, ga, gb, gc, gd))
