"""What the framework is timed on: whole calls of its public classes, from one
request of a few thousand points to the benchmark's 512^3 field, with inputs
and results on the device.

A case is a dict of plain values; "kind" says which class it calls:

  heat        Heat: upload, `steps` explicit steps, read; `arith` is the handle's
              arithmetic (f64, f32, fixed64)
  paper       Heat with HS_VARKAPPA, the paper's variable-coefficient problem
  cg          CG on the 7-point Laplacian: `op` matrix_free or csr, `mixed` for
              FP32 Krylov vectors inside FP64 refinement
  heat_batch  HeatBatch: many uneven grids, FP64 and FP32 in turn, one launch
  cg_batch    CGBatch: many systems solved together

The grids of a batch follow from the case (its `pick`), the values of every
input from the seed given to prepare().
"""
import math
import random

import numpy as np
import torch

import paper_2608_11882_gb300 as hc

KAPPA_MAX = 0.95
PAPER_R = 1.0 / (12.0 * KAPPA_MAX)   # dt = h^2 / (12 kappa_max)


def listed():
    return [
        # the smallest call: one short FP32 request as the server admits them
        # (edges from 32 up, odd, steps from 10 up); launches and latency
        dict(name="heat_request_f32", kind="heat", nx=45, ny=37, nz=61, r=0.11, steps=60, arith="f32", field="uniform"),
        # the parity configuration: 64^3, r = 0.1, 100 FP64 steps
        dict(name="heat_64_f64", kind="heat", nx=64, ny=64, nz=64, r=0.1, steps=100, arith="f64", field="modes"),
        # an ordinary request: uneven edges, odd nx and ny, FP64
        dict(name="heat_ragged_f64", kind="heat", nx=191, ny=101, nz=150, r=0.14, steps=200, arith="f64",
             field="uniform"),
        # the benchmark's field and arithmetic, 100 of its 1000 steps
        dict(name="heat_512_f64", kind="heat", nx=512, ny=512, nz=512, r=0.15, steps=100, arith="f64", field="modes"),
        # the same field in single precision
        dict(name="heat_512_f32", kind="heat", nx=512, ny=512, nz=512, r=0.15, steps=200, arith="f32", field="modes"),
        # the paper's own problem at its N = 512 (510^3 interior points), FP64
        dict(name="paper_510_f64", kind="paper", nx=510, ny=510, nz=510, steps=40, dtype="f64"),
        # a small solve, as batches and the server's stream hold them
        dict(name="cg_64", kind="cg", nx=64, ny=64, nz=64, op="matrix_free", mixed=False, rtol=1e-8),
        # the benchmark's solve, matrix-free, CSR and mixed precision
        dict(name="cg_256", kind="cg", nx=256, ny=256, nz=256, op="matrix_free", mixed=False, rtol=1e-8),
        dict(name="cg_256_csr", kind="cg", nx=256, ny=256, nz=256, op="csr", mixed=False, rtol=1e-8),
        # the tighter tolerance of the precision workload
        dict(name="cg_256_mixed", kind="cg", nx=256, ny=256, nz=256, op="matrix_free", mixed=True, rtol=1e-10),
        # the batching workload: 256 uneven grids, edges 16 to 128, 50 to 500 steps
        dict(name="heat_batch_256", kind="heat_batch", grids=256, lo=16, hi=128, steps_lo=50, steps_hi=500, pick=3),
        # 64 systems with edges 32 to 128
        dict(name="cg_batch_64", kind="cg_batch", systems=64, lo=32, hi=128, pick=4, rtol=1e-8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["heat", "heat", "heat", "paper", "cg", "cg", "heat_batch", "cg_batch"])
    if kind == "heat":
        nx, ny, nz = (_log_int(rng, 16, 640) for _ in range(3))
        most = 512 ** 3 * 100 // (nx * ny * nz)   # no more updates than the largest listed field
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, r=round(rng.uniform(0.05, 0.16), 4),
                    steps=_log_int(rng, 10, max(10, min(500, most))), arith=rng.choice(["f64", "f64", "f32", "fixed64"]),
                    field=rng.choice(["modes", "uniform"]))
    if kind == "paper":
        nx = _log_int(rng, 48, 510)
        ny, nz = (nx, nx) if rng.random() < 0.7 else (_log_int(rng, 48, 510), _log_int(rng, 48, 510))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=rng.randint(10, 40), dtype=rng.choice(["f64", "f32"]))
    if kind == "cg":
        nx, ny, nz = (_log_int(rng, 32, 256) for _ in range(3))
        op, mixed = rng.choice([("matrix_free", False), ("matrix_free", False), ("csr", False), ("matrix_free", True)])
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, op=op, mixed=mixed, rtol=1e-10 if mixed else 1e-8)
    if kind == "heat_batch":
        return dict(kind=kind, grids=_log_int(rng, 8, 256), lo=16, hi=128, steps_lo=50, steps_hi=500,
                    pick=rng.randrange(1 << 20))
    return dict(kind=kind, systems=_log_int(rng, 4, 64), lo=32, hi=128, pick=rng.randrange(1 << 20), rtol=1e-8)


def _batch_specs(case):
    """The grids of a batch: edges log-uniform per axis, and for heat r in
    [0.05, 0.16], the step count and the arithmetic of each."""
    rng = random.Random(case["pick"])
    out = []
    for g in range(case.get("grids") or case["systems"]):
        shape = tuple(_log_int(rng, case["lo"], case["hi"]) for _ in range(3))   # (nz, ny, nx)
        if case["kind"] == "heat_batch":
            out.append((shape, rng.uniform(0.05, 0.16), rng.randint(case["steps_lo"], case["steps_hi"]),
                        "f32" if g % 2 else "f64"))
        else:
            out.append(shape)
    return out


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, gen, dtype=torch.float64):
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen).mul_(2.0).sub_(1.0).to(dtype)


def _sines(k, n):
    return torch.sin(k * math.pi * torch.arange(1, n + 1, dtype=torch.float64, device="cuda") / (n + 1))


def _field(case, seed, dtype):
    """Initial field: the benchmark's 8 sine modes plus 1e-3 noise, or a
    request's U[-1, 1]."""
    gen = _gen(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    if case.get("field") == "uniform":
        return _uniform(shape, gen, dtype)
    rng = random.Random(seed)
    u = _uniform(shape, gen).mul_(1e-3)
    for _ in range(8):
        a = rng.uniform(0.5, 1.0)
        sz, sy, sx = (_sines(rng.randint(1, 16), n) for n in shape)
        u += (a * sz)[:, None, None] * (sy[:, None] * sx[None, :])
    return u.to(dtype)


def _paper_field(case, seed, dtype):
    """The paper's initial field, one sine mode, with 1% noise."""
    shape = (case["nz"], case["ny"], case["nx"])
    sz, sy, sx = (_sines(1, n) for n in shape)
    return (sz[:, None, None] * (sy[:, None] * sx[None, :]) + 0.01 * _uniform(shape, _gen(seed))).to(dtype)


def _rhs(n, gen):
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)


def _csr(nx, ny, nz):
    """The 7-point Dirichlet Laplacian as int32 CSR, columns ascending."""
    n = nx * ny * nz
    row = torch.arange(n, dtype=torch.int32, device="cuda")
    i, j, k = row % nx, row // nx % ny, row // (nx * ny)
    offs = [-nx * ny, -nx, -1, 0, 1, nx, nx * ny]
    have = torch.stack([k > 0, j > 0, i > 0, row >= 0, i < nx - 1, j < ny - 1, k < nz - 1], dim=1)
    col = (row[:, None] + torch.tensor(offs, dtype=torch.int32, device="cuda"))[have]
    val = torch.tensor([-1.0, -1.0, -1.0, 6.0, -1.0, -1.0, -1.0], dtype=torch.float64, device="cuda").repeat(n, 1)[have]
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rowptr[1:] = torch.cumsum(have.sum(dim=1), 0)
    return rowptr, col, val


_ARITH = {"f64": ("f64", 0), "f32": ("f32", 0), "fixed64": ("f64", "HS_FIXED64")}


def _dtype(name):
    return torch.float32 if name == "f32" else torch.float64


def prepare(case, seed):
    kind = case["kind"]
    if kind == "heat":
        dtype, flags = _ARITH[case["arith"]]
        u0 = _field(case, seed, _dtype(dtype))
        h = hc.Heat(case["nx"], case["ny"], case["nz"], case["r"], dtype=dtype,
                    flags=getattr(hc, flags) if flags else 0)
        return {"kind": kind, "heat": h, "steps": case["steps"], "u0": u0, "out": torch.empty_like(u0)}
    if kind == "paper":
        u0 = _paper_field(case, seed, _dtype(case["dtype"]))
        h = hc.Heat(case["nx"], case["ny"], case["nz"], PAPER_R, dtype=case["dtype"], flags=hc.HS_VARKAPPA)
        return {"kind": "heat", "heat": h, "steps": case["steps"], "u0": u0, "out": torch.empty_like(u0)}
    if kind == "cg":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        op = hc.Operator.csr(*_csr(nx, ny, nz)) if case["op"] == "csr" else hc.Operator.stencil(nx, ny, nz)
        return {"kind": kind, "cg": hc.CG(op, mixed=case["mixed"]), "b": _rhs(nx * ny * nz, _gen(seed)),
                "rtol": case["rtol"]}
    gen = _gen(seed)
    specs = _batch_specs(case)
    if kind == "heat_batch":
        # the results of all grids of a type land in one buffer, grid after grid
        flat = {d: torch.empty(sum(math.prod(s[0]) for s in specs if s[3] == d), dtype=_dtype(d), device="cuda")
                for d in ("f64", "f32")}
        at = {"f64": 0, "f32": 0}
        heats, u0s, outs = [], [], []
        for shape, r, _, d in specs:
            n = math.prod(shape)
            heats.append(hc.Heat(shape[2], shape[1], shape[0], r, dtype=d, tdepth=1))
            u0s.append(_uniform(shape, gen, _dtype(d)))
            outs.append(flat[d][at[d]:at[d] + n])
            at[d] += n
        return {"kind": kind, "batch": hc.HeatBatch(heats, [s[2] for s in specs]), "heats": heats, "u0": u0s,
                "views": outs, "out": flat}
    return {"kind": kind, "batch": hc.CGBatch([hc.Operator.stencil(s[2], s[1], s[0]) for s in specs]),
            "b": [_rhs(math.prod(s), gen) for s in specs], "sizes": [math.prod(s) for s in specs],
            "rtol": case["rtol"]}


def run(state):
    kind = state["kind"]
    if kind == "heat":
        h = state["heat"]
        h.upload(state["u0"])
        h.step(state["steps"])
        return h.read(state["out"])
    if kind == "cg":
        x, _ = state["cg"].run(state["b"], rtol=state["rtol"])
        return x
    if kind == "heat_batch":
        for h, u in zip(state["heats"], state["u0"]):
            h.upload(u)
        state["batch"].run()
        state["batch"].wait()
        for h, o in zip(state["heats"], state["views"]):
            h.read(o)
        return state["out"]
    flat = torch.zeros(sum(state["sizes"]), dtype=torch.float64, device="cuda")
    state["batch"].run(state["b"], list(flat.split(state["sizes"])), rtol=state["rtol"])
    return flat


def _iterations(shape, rtol):
    """About how many iterations CG takes on the Laplacian of a grid for a
    N(0, 1) right-hand side (174 at 48^3, 851 at 256^3 to 1e-8)."""
    edge = math.sqrt(3.0 / sum(1.0 / (n * n) for n in shape))
    return 4.35 * edge ** 0.953 * (1.0 + 0.1 * (math.log10(1e-8 / rtol)))


def work(case):
    """Bytes and operations of one pass, each step or iteration reading what it
    needs once and writing what it forms once."""
    kind = case["kind"]
    if kind in ("heat", "paper"):
        f32 = (case.get("arith") or case["dtype"]) == "f32"
        pts, e = case["nx"] * case["ny"] * case["nz"], 4 if f32 else 8
        per = 2 * e if kind == "heat" else 4 * e    # the paper's update reads kappa and the source too
        flops = 9 if kind == "heat" else 29
        return {"bytes": pts * (4 * e + per * case["steps"]), "flops": pts * flops * case["steps"]}
    if kind == "heat_batch":
        specs = _batch_specs(case)
        return {"bytes": sum(math.prod(s) * (4 if d == "f32" else 8) * (4 + 2 * n) for s, _, n, d in specs),
                "flops": sum(math.prod(s) * 9 * n for s, _, n, _ in specs)}
    shapes = _batch_specs(case) if kind == "cg_batch" else [(case["nz"], case["ny"], case["nx"])]
    nbytes = flops = 0.0
    for s in shapes:
        n, its = math.prod(s), _iterations(s, case["rtol"])
        # SpMV: read p, write q; update: read x, r, p, q, write x, r; direction: read r, p, write p
        per = 88 if not case.get("mixed") else 44
        if case.get("op") == "csr":
            per += 7 * 12 + 4
        nbytes += n * per * its
        flops += n * 20 * its
    return {"bytes": nbytes, "flops": flops}


# ---- the same results in 64 bits, without the framework ------------------------------------

def _pad(u):
    return torch.nn.functional.pad(u.double(), (1, 1, 1, 1, 1, 1))


def _neighbours(p):
    c = p[1:-1, 1:-1, 1:-1]
    return c, (p[1:-1, 1:-1, :-2], p[1:-1, 1:-1, 2:], p[1:-1, :-2, 1:-1], p[1:-1, 2:, 1:-1], p[:-2, 1:-1, 1:-1],
               p[2:, 1:-1, 1:-1])


def _heat_exact(u0, r, steps):
    p = _pad(u0)
    for _ in range(steps):
        c, (xm, xp, ym, yp, zm, zp) = _neighbours(p)
        s = xm + xp
        s += ym
        s += yp
        s += zm
        s += zp
        s.sub_(c, alpha=6.0).mul_(r)
        c += s
    return p[1:-1, 1:-1, 1:-1].contiguous()


def _paper_exact(u0, steps):
    shape = u0.shape
    h = [1.0 / (n + 1) for n in shape]
    dt = PAPER_R * min(h) ** 2
    grid = [torch.arange(0, n + 2, dtype=torch.float64, device="cuda") / (n + 1) * math.pi for n in shape]
    s, c = [torch.sin(g) for g in grid], [torch.cos(g) for g in grid]
    kap = 0.5 + 0.45 * s[0][:, None, None] * s[1][None, :, None] * s[2][None, None, :]
    src = dt * (1.0 + (c[0][:, None, None] * c[1][None, :, None] * c[2][None, None, :])[1:-1, 1:-1, 1:-1])
    beta = [dt / (2.0 * v * v) for v in h]
    kc, kn = _neighbours(kap)
    p = _pad(u0)
    for _ in range(steps):
        u, un = _neighbours(p)
        new = u + src
        for n in range(6):
            b = beta[2 - n // 2]
            new += (b * (kn[n] + kc)) * (un[n] - u)
        p[1:-1, 1:-1, 1:-1] = new
    return p[1:-1, 1:-1, 1:-1].contiguous()


def _poisson_exact(b, shape):
    """The solution of the 7-point system by sine transforms along each axis."""
    mats, lam = [], []
    for n in shape:
        i = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
        mats.append(math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi * torch.outer(i, i) / (n + 1)))
        lam.append(4.0 * torch.sin(i * math.pi / (2 * (n + 1))) ** 2)

    def transform(v):
        v = v @ mats[2]
        v = mats[1] @ v
        return (mats[0] @ v.reshape(shape[0], -1)).reshape(shape)

    v = transform(b.reshape(shape))
    v /= lam[0][:, None, None] + lam[1][None, :, None] + lam[2][None, None, :]
    return transform(v).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "heat":
        return _heat_exact(_field(case, seed, _dtype(case["arith"])), case["r"], case["steps"])
    if kind == "paper":
        return _paper_exact(_paper_field(case, seed, _dtype(case["dtype"])), case["steps"])
    gen = _gen(seed)
    if kind == "cg":
        shape = (case["nz"], case["ny"], case["nx"])
        return _poisson_exact(_rhs(math.prod(shape), gen), shape)
    if kind == "heat_batch":
        parts = {"f64": [], "f32": []}
        for shape, r, steps, d in _batch_specs(case):
            parts[d].append(_heat_exact(_uniform(shape, gen, _dtype(d)), r, steps).reshape(-1))
        return {d: torch.cat(v) if v else torch.empty(0, dtype=torch.float64, device="cuda") for d, v in parts.items()}
    return torch.cat([_poisson_exact(_rhs(math.prod(s), gen), s) for s in _batch_specs(case)])
