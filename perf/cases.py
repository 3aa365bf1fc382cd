"""The work whose speed is measured, case by case, through the public entry points.

A case is one call (or one short sequence of calls) of a user's program on
synthetic Darcy systems: the two-point flux matrix of ``-div(k grad u) = f``
on a box of cells with homogeneous Dirichlet data, ``k`` a lognormal Gaussian
random field or a background of 1 crossed by channels, cut into regular
blocks of cells.  Kinds:

``solve``   ``AmsSolver.solve`` with a solver that is kept: one matrix, 1 to
            32 right-hand sides, in the mixed precisions and in FP64.
``batch``   ``AmsBatchedSolver.solve``: systems of uneven size in one call.
``train``   ``ams_solve`` forward and backward: misfit at observation cells,
            gradients of the matrix values and of the right-hand side.
``new``     a matrix that changes from call to call: the solver is built,
            solves once and goes.
``krylov``  ``apply_preconditioner`` and ``spmv`` as a user's own Krylov
            method calls them.

Right-hand sides are the unit source (``h^d``) or N(0, 1); every solve stops
at a relative residual of 1e-8.
"""

import math

import numpy as np
import torch

from paper_2606_04864_gb300 import AmsBatchedSolver, AmsSolver
from paper_2606_04864_gb300.autograd import ams_solve

RTOL = 1e-8


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one solve of a small 2-D system, where launches and latency count
        dict(name="solve2d_64_r1", kind="solve", shape="64x64", bs=8, m=4, field="grf", std=2.0, nrhs=1,
             precision="fp32_bf16"),
        # one large 2-D system of high contrast, one source: a reservoir pressure solve (its residual stalls on
        # plateaus, where the last bit of any rounding decides between two iteration counts: u alone comes back)
        dict(name="solve2d_1024_channels_r1", kind="solve", shape="1024x1024", bs=32, m=8, field="channels", kmax=1e4,
             nrhs=1, precision="fp32_bf16"),
        # the largest: many sources on one large 3-D system
        dict(name="solve3d_128_r32", kind="solve", shape="128x128x128", bs=8, m=6, field="grf", std=3.0, nrhs=32,
             precision="fp32_bf16"),
        # a few sources on a box with unequal sides, FP32 basis
        dict(name="solve3d_96x80x72_r3_fp32", kind="solve", shape="96x80x72", bs=8, m=6, field="grf", std=2.0, nrhs=3,
             precision="fp32"),
        # all in FP64, sides that the blocks do not divide, a number of sources between two strides
        dict(name="solve3d_50_r5_fp64", kind="solve", shape="50x50x50", bs=8, m=6, field="grf", std=2.0, nrhs=5,
             precision="fp64"),
        # the multiplicative cycle with its damping estimated
        dict(name="solve3d_77_r8_cycle", kind="solve", shape="77x77x77", bs=8, m=6, field="grf", std=2.0, nrhs=8,
             precision="fp32_bf16", cycle=True),
        # an ensemble of uneven 2-D and 3-D systems in one call
        dict(name="batch_uneven_r8", kind="batch", shape="131x131,200x200,317x317,450x450,33x33x33,47x47x47,64x64x64,"
             "90x90x90", bs=8, m=6, field="grf", std=2.5, nrhs=8, precision="fp32_bf16"),
        # one training step of an inverse problem: forward, misfit, adjoint, gradients
        dict(name="train3d_96_r1", kind="train", shape="96x96x96", bs=8, m=6, field="grf", std=2.0, nrhs=1,
             precision="fp32_bf16"),
        # a matrix that changes with every call (a time step, a sample): setup and solve
        dict(name="new2d_512_r1", kind="new", shape="512x512", bs=32, m=8, field="grf", std=2.0, nrhs=1,
             precision="fp32_bf16"),
        dict(name="new3d_64_r8", kind="new", shape="64x64x64", bs=8, m=6, field="grf", std=2.5, nrhs=8,
             precision="fp32_bf16"),
        # a user's own Krylov method on a block of vectors: one preconditioner application, one product
        dict(name="krylov3d_96_r16", kind="krylov", shape="96x96x96", bs=8, m=6, field="grf", std=2.0, nrhs=16,
             precision="fp32_bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side2(rng, lo, hi):
    """A 2-D side and the block side that goes with it (the coarse space stays in the range of the listed cases)."""
    side = _log(rng, lo, hi)
    return side, rng.choice([8, 16] if side <= 256 else [16, 32] if side <= 640 else [32])


def draw(rng):
    kind = rng.choice(["solve2", "solve3", "solve3", "batch", "train", "new2", "new3", "krylov"])
    case = dict(kind=kind.rstrip("23"), m=rng.randint(4, 8), field="grf", std=round(rng.uniform(1.5, 3.0), 2),
                nrhs=_log(rng, 1, 32), precision=rng.choice(["fp32_bf16", "fp32_bf16", "fp32"]), bs=8)
    if kind in ("solve2", "new2"):
        side, case["bs"] = _side2(rng, 64, 1024 if kind == "solve2" else 600)
        case["shape"] = "%dx%d" % (max(64, side - rng.randint(0, 40)), side)
        case["nrhs"] = _log(rng, 1, 8)
        case["std"] = round(rng.uniform(1.5, 2.2), 2)
    elif kind == "batch":
        twos = ["%dx%d" % ((_log(rng, 128, 400),) * 2) for _ in range(rng.randint(1, 3))]
        threes = ["%dx%dx%d" % ((_log(rng, 32, 84),) * 3) for _ in range(rng.randint(1, 3))]
        case["shape"] = ",".join(twos + threes)
        case["nrhs"] = _log(rng, 2, 16)
        case["precision"] = "fp32_bf16"
    else:
        side = _log(rng, 24, 64 if kind == "new3" else 110)
        case["shape"] = "%dx%dx%d" % (max(24, side - rng.randint(0, 12)), side, max(24, side - rng.randint(0, 12)))
        case["m"] = rng.randint(4, 6)
        if kind == "train":
            case["nrhs"] = rng.choice([1, 1, 2, 4])
        elif kind == "solve3":
            if side <= 56 and rng.random() < 0.4:
                case["precision"] = "fp64"
            elif rng.random() < 0.2:
                case["cycle"] = True
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _shape(text):
    return tuple(int(s) for s in text.split("x"))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _logk(case, shape, seed):
    """log-permeability: white noise under a Gaussian filter of 4 (2-D) or 6 (3-D) cells, or channels."""
    g = _gen(seed)
    if case["field"] == "channels":
        rng = np.random.default_rng(seed)
        k = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for _ in range(200):
            width, length = int(rng.integers(2, 5)), int(rng.integers(64, 513))
            y, x = int(rng.integers(0, shape[0])), int(rng.integers(0, shape[1]))
            dy, dx = (width, length) if rng.integers(0, 2) else (length, width)
            k[y:y + dy, x:x + dx] = math.log(case["kmax"])
        return k
    sigma = 4.0 if len(shape) == 2 else 6.0
    noise = torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")
    spec = torch.fft.fftn(noise)
    for a, s in enumerate(shape):
        w = 2.0 * math.pi * torch.fft.fftfreq(s, dtype=torch.float64, device="cuda")
        spec = spec * torch.exp(-0.5 * (sigma * w) ** 2).reshape([-1 if b == a else 1 for b in range(len(shape))])
    f = torch.fft.ifftn(spec).real
    f = f - f.mean()
    return f * (case["std"] / f.std(unbiased=False))


def _stencil(logk):
    """The matrix by slots in ascending column order: (values (slots, n), present (slots, n), column offsets)."""
    shape, d = logk.shape, logk.dim()
    fac = (1.0 / max(shape)) ** (d - 2)
    k = torch.exp(logk)
    diag = torch.zeros_like(k)
    low, high, offs = [], [], []
    stride = 1
    strides = [0] * d
    for a in range(d - 1, -1, -1):
        strides[a] = stride
        stride *= shape[a]
    for a in range(d):
        lo, hi = k.narrow(a, 0, shape[a] - 1), k.narrow(a, 1, shape[a] - 1)
        t = fac * 2.0 * lo * hi / (lo + hi)
        up, dn = torch.zeros_like(k), torch.zeros_like(k)      # to the next cell, to the one before
        up.narrow(a, 0, shape[a] - 1).copy_(t)
        dn.narrow(a, 1, shape[a] - 1).copy_(t)
        diag += up + dn
        for e in (0, shape[a] - 1):
            diag.narrow(a, e, 1).add_(fac * 2.0 * k.narrow(a, e, 1))
        low.append(-dn.reshape(-1))
        high.append(-up.reshape(-1))
        offs.append(strides[a])
    vals = torch.stack(low + [diag.reshape(-1)] + high[::-1])
    here = vals != 0
    return vals, here, [-o for o in offs] + [0] + offs[::-1]


def _csr(logk):
    vals, here, offs = _stencil(logk)
    n = vals.shape[1]
    cols = torch.arange(n, device="cuda").unsqueeze(0) + torch.tensor(offs, device="cuda").unsqueeze(1)
    keep = here.t()
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(here.sum(0), 0)
    return rowptr, cols.t()[keep].to(torch.int32).contiguous(), vals.t()[keep].contiguous()


def _blocks(shape, bs):
    """Regular blocks of bs cells a side, the last along an axis partial."""
    nb = [-(-s // bs) for s in shape]
    part = torch.zeros(shape, dtype=torch.int64, device="cuda")
    for a, s in enumerate(shape):
        i = torch.arange(s, device="cuda") // bs
        part = part * nb[a] + i.reshape([-1 if b == a else 1 for b in range(len(shape))])
    return part.reshape(-1).to(torch.int32), math.prod(nb)


def _rhs(case, shape, seed):
    n, r = math.prod(shape), case["nrhs"]
    if r == 1:
        f = torch.full((1, n), (1.0 / max(shape)) ** len(shape), dtype=torch.float64, device="cuda")
        return f
    return torch.randn((r, n), generator=_gen(seed + 7919), dtype=torch.float64, device="cuda")


def _options(case):
    return dict(precision=case["precision"], device=True)


def _system(case, shape, seed):
    rowptr, colind, vals = _csr(_logk(case, shape, seed))
    part, nparts = _blocks(shape, case["bs"])
    return rowptr, colind, vals, part, nparts, case["m"]


def prepare(case, seed):
    shapes = [_shape(t) for t in case["shape"].split(",")]
    if case["kind"] == "batch":
        systems = [_system(case, s, seed + 101 * k) for k, s in enumerate(shapes)]
        solver = AmsBatchedSolver(systems, **_options(case))
        f = solver.pack([_rhs(case, s, seed + 101 * k) if case["nrhs"] > 1 else _rhs(case, s, 0)
                         for k, s in enumerate(shapes)])
        return dict(case=case, solver=solver, f=f)
    shape = shapes[0]
    system = _system(case, shape, seed)
    state = dict(case=case, f=_rhs(case, shape, seed))
    if case["kind"] == "new":
        return dict(state, system=system)
    options = dict(two_grid_omega=-1.0) if case.get("cycle") else {}
    state["solver"] = AmsSolver(*system, **_options(case), **options)
    if case["kind"] == "krylov":
        state["x"] = torch.randn(state["f"].shape, generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
    if case["kind"] == "train":
        n = math.prod(shape)
        state["vals"] = system[2].clone().requires_grad_(True)
        state["f"].requires_grad_(True)
        state["obs"] = torch.randperm(n, generator=_gen(seed + 2), device="cuda")[:min(4096, n // 8)].sort().values
        # data: what a field of the same kind gives at the observation cells, here its size only
        state["data"] = torch.randn((case["nrhs"], state["obs"].numel()), generator=_gen(seed + 3), dtype=torch.float64,
                                    device="cuda")
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case, f = state["case"], state["f"]
    if case["kind"] == "batch":
        u, iters, _ = state["solver"].solve(f, case["nrhs"], RTOL)
        return {"u": u, "iters": iters}
    if case["kind"] == "new":
        solver = AmsSolver(*state["system"], **_options(case))
        u, iters, _ = solver.solve(f, RTOL)
        solver.close()
        return {"u": u, "iters": iters}
    if case["kind"] == "krylov":
        # in the mixed precisions z holds FP32 values: the program keeps it so
        return {"z": state["solver"].apply_preconditioner(f).float(), "q": state["solver"].spmv(state["x"])}
    if case["kind"] == "train":
        u = ams_solve(state["vals"], f, state["solver"], RTOL)
        loss = 0.5 * (u[:, state["obs"]] - state["data"]).square().sum()
        dvals, df = torch.autograd.grad(loss, (state["vals"], f))
        return {"u": u.detach(), "dvals": dvals, "df": df}
    u, iters, _ = state["solver"].solve(f, RTOL)
    return {"u": u} if case["field"] == "channels" else {"u": u, "iters": iters}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _sizes(case, shape):
    """(n, nnz, subdomains, N_c, entries of the local factors, entries of the coarse factor), the factors with
    nested-dissection fill: entries a row of a block's factor by its side, and of the coarse one by its size."""
    n, d = math.prod(shape), len(shape)
    nnz = n + 2 * sum(n // s * (s - 1) for s in shape)
    nsub = math.prod(-(-s // case["bs"]) for s in shape)
    nc = nsub * case["m"]
    local = n * (32.5 if d == 3 else {8: 7.0, 16: 11.0, 32: 15.7}[case["bs"]])
    coarse = min(nc * (nc + 1) / 2, 19.3 * nc ** (4 / 3) if d == 3 else 9.4 * nc * math.log2(max(2, nc)))
    return n, nnz, nsub, nc, local, coarse


def work(case):
    """A solve: its iterations (about as many as the range takes) times one iteration's operands, each read once and each
    result written once, since they pass any cache between two iterations.  Setup: the matrix in, the factors out, band
    Cholesky and ten steps of the local eigenproblems."""
    bytes_, flops, r = 0.0, 0.0, case["nrhs"]
    tf = 8 if case["precision"] == "fp64" else 4
    tp = {"fp64": 8, "fp32": 4, "fp32_bf16": 2}[case["precision"]]
    for shape in (_shape(t) for t in case["shape"].split(",")):
        n, nnz, nsub, nc, local, coarse = _sizes(case, shape)
        iters = 110 if case["field"] == "channels" else 33
        if case.get("cycle"):
            iters = 17
        precond = tf * (local + coarse) + tp * n * case["m"] + 16 * n * r
        step = 12 * nnz + 4 * n + precond + 48 * n * r
        mult = 2 * r * (2 * local + 2 * coarse + 2 * n * case["m"])
        if case["kind"] == "krylov":
            bytes_ += precond + 12 * nnz + 4 * n + 16 * n * r
            flops += mult + 2 * nnz * r
            continue
        solves = 2 if case["kind"] == "train" else 1
        bytes_ += solves * (iters * step + 16 * n * r) + (24 * nnz if solves == 2 else 0)
        flops += solves * iters * (mult + 2 * nnz * r + 16 * n * r)
        if case["kind"] == "new":
            band = case["bs"] ** (len(shape) - 1)
            bytes_ += 12 * nnz + 4 * (local + coarse) + 2 * n * case["m"]
            flops += 2 * n * band * band + 10 * 4 * n * band * 2 * case["m"]
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, by plain torch
# ---------------------------------------------------------------------------

def _apply(st, x):
    """A x for x (r, n), by the stencil's slots."""
    vals, _, offs = st
    y = torch.zeros_like(x)
    n = x.shape[1]
    for v, o in zip(vals, offs):
        if o >= 0:
            y[:, :n - o] += v[:n - o] * x[:, o:]
        else:
            y[:, -o:] += v[-o:] * x[:, :o]
    return y


def _cg(st, f, most=20000):
    """A^{-1} f by CG with the diagonal as its preconditioner, and one correction from the true residual; None where it
    takes too long."""
    d = st[0][len(st[2]) // 2]
    u = torch.zeros_like(f)
    for tol in (1e-13, 1e-4):
        b = f - _apply(st, u)
        x, r = torch.zeros_like(b), b.clone()
        z = r / d
        p, rho, stop = z.clone(), (r * z).sum(1), tol * b.norm(dim=1)
        for it in range(most):
            if it % 50 == 0 and bool((r.norm(dim=1) <= stop).all()):
                break
            q = _apply(st, p)
            pq = (p * q).sum(1)
            a = torch.where(pq > 0, rho / pq, torch.zeros_like(pq)).unsqueeze(1)
            x += a * p
            r -= a * q
            z = r / d
            new = (r * z).sum(1)
            p = z + torch.where(rho > 0, new / rho, torch.zeros_like(rho)).unsqueeze(1) * p
            rho = new
        else:
            return None
        u = u + x
    return u


def exact(case, seed):
    shapes = [_shape(t) for t in case["shape"].split(",")]
    if case["kind"] != "krylov" and sum(math.prod(s) for s in shapes) * case["nrhs"] > 12e6:
        return None
    if case["kind"] == "batch":
        out = []
        for k, s in enumerate(shapes):
            u = _cg(_stencil(_logk(case, s, seed + 101 * k)), _rhs(case, s, seed + 101 * k if case["nrhs"] > 1 else 0))
            if u is None:
                return None
            out.append(u.reshape(-1))
        return {"u": torch.cat(out), "iters": None}
    shape = shapes[0]
    st = _stencil(_logk(case, shape, seed))
    if case["kind"] == "krylov":
        x = torch.randn((case["nrhs"], math.prod(shape)), generator=_gen(seed + 1), dtype=torch.float64, device="cuda")
        return {"z": None, "q": _apply(st, x)}
    u = _cg(st, _rhs(case, shape, seed))
    if u is None:
        return None
    if case["kind"] != "train":
        return {"u": u, "iters": None}
    n = math.prod(shape)
    obs = torch.randperm(n, generator=_gen(seed + 2), device="cuda")[:min(4096, n // 8)].sort().values
    data = torch.randn((case["nrhs"], obs.numel()), generator=_gen(seed + 3), dtype=torch.float64, device="cuda")
    g = torch.zeros_like(u)
    g[:, obs] = u[:, obs] - data
    lam = _cg(st, g)
    if lam is None:
        return None
    vals, here, offs = st
    dv = torch.zeros_like(vals)
    for k, o in enumerate(offs):
        lo, hi = max(0, -o), n - max(0, o)
        dv[k, lo:hi] = -(lam[:, lo:hi] * u[:, lo + o:hi + o]).sum(0)
    return {"u": u, "dvals": dv.t()[here.t()], "df": lam}
