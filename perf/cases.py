"""Timed cases: what a user of the library has it do, through its Python entry points.

Every case is a dict of plain values whose "kind" names the call:

  cg        pk.cg_solve, plain pipelined CG to 1e-8 from x0 = 0, Laplacian of a 2D or 3D grid
  heat      pk.cg_solve from the previous time step: one implicit heat step, variable
            coefficients (a handful of iterations: setup, launches and the status read count)
  mixed     the same step in mixed precision (FP32 inside FP64 refinement) to 1e-10
  pcg       Jacobi-preconditioned CG on a 3D linear-elasticity matrix (3 x 3 blocks, up to 45
            nonzeros per row) with a mass term, as one step of implicit dynamics solves it
  bicgstab  pipelined BiCGStab on upwind convection-diffusion
  gmres     pipelined GMRES(m) on the same matrices
  circuit   right-Jacobi BiCGStab on a matrix of power-law row lengths (3 to 256)
  batched   pk.batched_solve: independent shifted 2D Laplacians of uneven size
  conv      one 16-channel 3x3x3 layer of the learned start: forward, backward-data, weight
            gradient
  train     one training sample of the learned start: input, forward, loss, backward, Adam

Systems are manufactured: x* is drawn, b = A x*, so the exact answer of a solve is x*.
"""
import functools
import math

import numpy as np
import torch

from paper_1410_4054_gb300 import pk
from paper_1410_4054_gb300 import workloads as W
from paper_1410_4054_gb300.warmstart import CH, LAYERS, ConvNet

DEV = "cuda"
F64 = torch.float64
BF16 = torch.bfloat16


def listed():
    return [
        # the smallest call: latency of one solve that fits a few SMs
        dict(name="cg_2d_64", kind="cg", nz=1, ny=64, nx=64),
        # a million unknowns, the working set about as large as L2
        dict(name="cg_3d_100", kind="cg", nz=100, ny=100, nx=100),
        # the largest: four million unknowns, bound by memory and FP64 throughput
        dict(name="cg_3d_160", kind="cg", nz=160, ny=160, nx=160),
        # one time step of a transient simulation, started from the last one
        dict(name="heat_step_64", kind="heat", nz=64, ny=64, nx=64),
        # a larger time step in mixed precision; no side is a power of two
        dict(name="heat_mixed_130", kind="mixed", nz=130, ny=131, nx=127),
        # blocks of 3 unknowns, 45 per row: grouped rows, many more gathers per row
        dict(name="pcg_elasticity_23", kind="pcg", k=23),
        # nonsymmetric systems of a quarter million unknowns
        dict(name="bicgstab_64", kind="bicgstab", nz=64, ny=64, nx=64),
        dict(name="gmres30_64", kind="gmres", nz=64, ny=64, nx=64, restart=30),
        # irregular rows, columns spread over the whole vector
        dict(name="circuit_1e5", kind="circuit", n=100_000),
        # many uneven systems at once
        dict(name="batched_512", kind="batched", nsys=512),
        # the learned start's layer, and a whole training sample
        dict(name="conv_layer_64", kind="conv", nz=64, ny=64, nx=64),
        dict(name="train_sample_64", kind="train", nz=64, ny=64, nx=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    return dict(nz=_log(rng, lo, hi), ny=_log(rng, lo, hi), nx=_log(rng, lo, hi))


def draw(rng):
    kind = rng.choice(["cg", "cg", "heat", "mixed", "pcg", "bicgstab", "gmres", "circuit", "batched", "conv", "train"])
    if kind == "cg":
        if rng.random() < 0.4:
            return dict(kind=kind, nz=1, ny=_log(rng, 48, 800), nx=_log(rng, 48, 800))
        return dict(kind=kind, **_box(rng, 12, 150))
    if kind == "heat":
        return dict(kind=kind, **_box(rng, 16, 120))
    if kind == "mixed":
        return dict(kind=kind, **_box(rng, 24, 140))
    if kind == "pcg":
        return dict(kind=kind, k=rng.randint(5, 23))
    if kind == "bicgstab":
        return dict(kind=kind, **_box(rng, 16, 110))
    if kind == "gmres":
        return dict(kind=kind, **_box(rng, 16, 90), restart=rng.choice([10, 20, 30, 50]))
    if kind == "circuit":
        return dict(kind=kind, n=_log(rng, 5_000, 150_000))
    if kind == "batched":
        return dict(kind=kind, nsys=_log(rng, 24, 400))
    return dict(kind=kind, **_box(rng, 12, 72))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _grid_csr(diag, lower, upper):
    """CSR arrays on the GPU of a grid operator: diag [nz, ny, nx]; lower[a] / upper[a] the
    coefficient of the neighbour at index -1 / +1 along axis a (numbers or fields); neighbours
    outside the grid are dropped, an axis of one cell has none."""
    shape = diag.shape
    n = diag.numel()
    stride = (shape[1] * shape[2], shape[2], 1)
    own = torch.arange(n, device=DEV).view(shape)
    axes = [a for a in range(3) if shape[a] > 1]
    cols, vals, keep = [], [], []

    def put(a, step, v):
        inside = torch.ones(shape, dtype=torch.bool, device=DEV)
        if step:
            inside.select(a, 0 if step < 0 else shape[a] - 1).zero_()
        cols.append((own + (step * stride[a] if step else 0)).reshape(-1))
        vals.append((v if torch.is_tensor(v) else torch.full(shape, float(v), dtype=F64, device=DEV)).reshape(-1))
        keep.append(inside.reshape(-1))

    for a in axes:
        put(a, -1, lower[a])
    put(0, 0, diag)
    for a in reversed(axes):
        put(a, 1, upper[a])
    k = torch.stack(keep, 1)
    rp = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rp[1:] = k.sum(1).cumsum(0)
    return rp, torch.stack(cols, 1)[k].to(torch.int32), torch.stack(vals, 1)[k].contiguous()


def _laplacian(c):
    d = 4.0 if c["nz"] == 1 else 6.0
    return _grid_csr(torch.full(_dims(c), d, dtype=F64, device=DEV), (-1.0,) * 3, (-1.0,) * 3)


def _convdiff(c):
    """First-order upwind, velocity (1, 1, 1), cell Peclet number 0.5."""
    return _grid_csr(torch.full(_dims(c), 9.0, dtype=F64, device=DEV), (-2.0,) * 3, (-1.0,) * 3)


def _dims(c):
    return (c["nz"], c["ny"], c["nx"])


def _heat(c, seed):
    """I + dt L with a smoothed lognormal conductivity (harmonic means on the faces, Dirichlet
    boundary), dt such that the least dominant row has a dominance ratio of 1.5."""
    shape = _dims(c)
    kap = torch.exp(torch.randn(shape, generator=_gen(seed), dtype=F64, device=DEV))
    kap = torch.nn.functional.avg_pool3d(kap[None, None], 5, 1, 2, count_include_pad=False)[0, 0]
    diag = torch.zeros(shape, dtype=F64, device=DEV)
    low, upp = [], []
    for a in range(3):
        m = shape[a]
        ka, kb = kap.narrow(a, 0, m - 1), kap.narrow(a, 1, m - 1)
        kf = 2.0 * ka * kb / (ka + kb)
        lo, up = torch.zeros_like(kap), torch.zeros_like(kap)
        lo.narrow(a, 1, m - 1).copy_(kf)
        up.narrow(a, 0, m - 1).copy_(kf)
        diag += lo + up
        diag.select(a, 0).add_(kap.select(a, 0))
        diag.select(a, m - 1).add_(kap.select(a, m - 1))
        low.append(lo)
        upp.append(up)
    dt = 2.0 / float(diag.max())
    return _grid_csr(1.0 + dt * diag, [-dt * v for v in low], [-dt * v for v in upp])


def _field(c, t, seed):
    """The temperature at time t: a warm spot moving on a circle over a broad background."""
    shape = _dims(c)
    z, y, x = (torch.arange(m, dtype=F64, device=DEV) / m for m in shape)
    ph = 2.0 * math.pi * (t + (seed % 97)) / 300.0
    d = ((z[:, None, None] - 0.5) ** 2 + (y[None, :, None] - 0.5 - 0.25 * math.sin(ph)) ** 2
         + (x[None, None, :] - 0.5 - 0.25 * math.cos(ph)) ** 2)
    return (3.0 * torch.exp(-d / 0.008) + (1.0 + 0.002 * t) * torch.exp(-d / 0.15)).reshape(-1)


@functools.lru_cache(maxsize=2)
def _elasticity(k):
    a = W.fe_elasticity_3d(k)
    rows = np.repeat(np.arange(a.n), np.diff(a.row_ptr))
    on = rows == a.col
    val = a.val.copy()
    val[on] += 0.01 * a.val[on].max()  # mass term
    return a.row_ptr, a.col, val


@functools.lru_cache(maxsize=2)
def _circuit(n):
    a = W.power_law(n)
    return a.row_ptr, a.col, a.val


def _to_gpu(arrays):
    return tuple(torch.from_numpy(np.ascontiguousarray(v)).to(DEV) for v in arrays)


def _times(csr, x):
    """A x in plain torch."""
    rp, ci, va = csr
    return torch.segment_reduce(va * x[ci.long()], "sum", offsets=rp.long(), initial=0.0)


def _uniform(n, seed):
    return 2.0 * torch.rand(n, generator=_gen(seed), dtype=F64, device=DEV) - 1.0


def _rectangles(nsys, seed):
    """Sides log-uniform in [32, 256], shifts uniform in [0.01, 1]: sizes by nsys alone, so that
    every seed is the same amount of work."""
    r = np.random.default_rng(nsys)
    sides = np.rint(np.exp(r.uniform(math.log(32), math.log(256), size=(nsys, 2)))).astype(int)
    return sides, np.random.default_rng([nsys, seed]).permutation(np.linspace(0.01, 1.0, nsys))


def _system(c, seed):
    """(CSR arrays, x*, x0 or None for zero) of a single-system case."""
    kind = c["kind"]
    if kind in ("heat", "mixed"):
        return _heat(c, seed), _field(c, 2, seed), _field(c, 1, seed)
    csr = {"cg": lambda: _laplacian(c), "bicgstab": lambda: _convdiff(c), "gmres": lambda: _convdiff(c),
           "pcg": lambda: _to_gpu(_elasticity(c["k"])), "circuit": lambda: _to_gpu(_circuit(c["n"]))}[kind]()
    return csr, _uniform(csr[0].numel() - 1, seed), None


def _layer_inputs(c, seed):
    g = _gen(seed)
    v = _dims(c) + (CH,)
    randn = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    return dict(x=torch.relu(randn(*v)).to(BF16), w=(randn(27, CH, CH) * math.sqrt(2.0 / (27 * CH))).to(BF16),
                b=0.1 * randn(CH), g=(0.01 * randn(*v)).to(BF16))


# ------------------------------------------------------------------ the calls

SOLVE = {
    "cg": (pk.cg_solve, dict(tol=1e-8, maxit=50_000)),
    "heat": (pk.cg_solve, dict(tol=1e-8, maxit=10_000)),
    "mixed": (pk.cg_solve, dict(tol=1e-10, maxit=10_000, precision="mixed")),
    "pcg": (pk.cg_solve, dict(tol=1e-8, maxit=50_000, precond="jacobi")),
    "bicgstab": (pk.bicgstab_solve, dict(tol=1e-8, maxit=20_000)),
    "gmres": (pk.gmres_solve, dict(tol=1e-8, maxit=20_000)),
    "circuit": (pk.bicgstab_solve, dict(tol=1e-8, maxit=20_000, precond="jacobi")),
}


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(kind=kind)
    if kind in SOLVE:
        csr, xs, x0 = _system(c, seed)
        s["A"] = pk.CSRMatrix(*csr)
        s["b"] = _times(csr, xs)
        s["x0"] = x0
        s["x"] = torch.zeros_like(xs)
        s["kw"] = dict(SOLVE[kind][1], **({"restart": c["restart"]} if kind == "gmres" else {}))
    elif kind == "batched":
        sides, shifts = _rectangles(c["nsys"], seed)
        n = [int(a * b) for a, b in sides]
        s["x"] = torch.zeros(sum(n), dtype=F64, device=DEV)
        s["xs"] = list(s["x"].split(n))
        want = _uniform(sum(n), seed).split(n)
        s["A"], s["b"] = [], []
        for k, (side, shift) in enumerate(zip(sides, shifts)):
            d = torch.full((1, int(side[0]), int(side[1])), 4.0 + float(shift), dtype=F64, device=DEV)
            csr = _grid_csr(d, (-1.0,) * 3, (-1.0,) * 3)
            s["A"].append(pk.CSRMatrix(*csr))
            s["b"].append(_times(csr, want[k]))
    elif kind == "conv":
        s.update(_layer_inputs(c, seed), dims=_dims(c))
        s["y"], s["dx"] = torch.zeros_like(s["x"]), torch.zeros_like(s["x"])
        s["wf"] = torch.zeros_like(s["w"])
        pk.conv3d_flip(s["w"], s["wf"])
        s["dw"], s["db"] = torch.zeros(27, CH, CH, device=DEV), torch.zeros(CH, device=DEV)
        s["scratch"] = torch.zeros(pk.conv3d_wgrad_scratch_floats(s["dims"]), device=DEV)
    else:
        csr = _heat(c, seed)
        s["A"] = pk.CSRMatrix(*csr)
        s["xm2"], s["xm1"], s["xt"] = (_field(c, t, seed) for t in range(3))
        s["b"] = _times(csr, s["xt"])
        s["net"] = ConvNet(_dims(c), device=DEV, seed=seed % 1000)
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind in SOLVE:
        if s["x0"] is None:
            s["x"].zero_()
        else:
            s["x"].copy_(s["x0"])
        info = SOLVE[kind][0](s["A"], s["b"], s["x"], **s["kw"])
        return dict(x=s["x"]) if kind == "mixed" else dict(x=s["x"], iters=info["iters"], status=info["status"])
    if kind == "batched":
        s["x"].zero_()
        infos = pk.batched_solve(s["A"], s["b"], s["xs"], tol=1e-10, maxit=20_000)
        return dict(x=s["x"], status=np.array([i["status"] for i in infos]))
    if kind == "conv":
        pk.conv3d_fwd(s["x"], s["w"], s["b"], s["y"], s["dims"], relu=True)
        pk.conv3d_fwd(s["g"], s["wf"], None, s["dx"], s["dims"], relu=False, mask=s["x"])
        pk.conv3d_wgrad(s["x"], s["g"], s["scratch"], s["dw"], s["db"], s["dims"])
        return dict(y=s["y"], dx=s["dx"], dw=s["dw"], db=s["db"])
    net = s["net"]
    net.train_sample(s["A"], s["xm1"], s["xm2"], s["b"], s["xt"])
    return dict(out=net.out, loss=net.loss, dW=net.dW, db=net.db, W=net.W32, bias=net.b32)


# ------------------------------------------------------------------ what a pass needs

def _iterations(c):
    """About how many iterations (GMRES: steps) the case takes."""
    kind = c["kind"]
    if kind in ("cg", "bicgstab", "gmres"):
        side = max(c["ny"], c["nx"], c["nz"])
        if kind == "cg":
            return (2.5 if c["nz"] == 1 else 2.5 - side / 1600.0 + (0.8 if side < 40 else 0.3)) * side
        return (2.2 if kind == "bicgstab" else 4.2) * side
    return {"heat": 8, "mixed": 14, "pcg": 4 * c.get("k", 0), "circuit": 14}[kind]


def _entries(c):
    """(rows, nonzeros)."""
    if c["kind"] == "pcg":
        n = 3 * c["k"] * (c["k"] + 1) ** 2
        return n, 40 * n
    if c["kind"] == "circuit":
        return c["n"], 12 * c["n"]
    nz, ny, nx = _dims(c)
    n = nz * ny * nx
    return n, n + 2 * (3 * n - nz * ny - nz * nx - ny * nx) - (0 if nz > 1 else 2 * (n - ny * nx))


def work(case):
    c, kind = case, case["kind"]
    if kind in SOLVE:
        n, nnz = _entries(c)
        it = _iterations(c)
        f = 4 if kind == "mixed" else 8
        once = 12 * nnz + 4 * n + 24 * n
        # FP64 operations and bytes of one iteration: product, inner products, vector updates
        if kind in ("bicgstab", "circuit"):
            flops, per = 4 * nnz + 24 * n, 2 * (4 + f) * nnz + 160 * n
        elif kind == "gmres":
            flops, per = 2 * nnz + 2 * n * (c["restart"] + 2), (4 + f) * nnz + 8 * n * (c["restart"] + 5)
        else:
            flops, per = 2 * nnz + 12 * n, (4 + f) * nnz + 9.5 * f * n
        # a system that fits the 129 MB L2 with its vectors need not be read again
        fits = (4 + f) * nnz + 6 * f * n < 100e6 and kind != "gmres"
        return dict(bytes=once if fits else once + it * per, flops=it * flops)
    if kind == "batched":
        sides, _ = _rectangles(c["nsys"], 0)
        n = float((sides[:, 0] * sides[:, 1]).sum())
        return dict(bytes=(12 * 5 + 4 + 24) * n, flops=60 * 22 * n)
    n = float(np.prod(_dims(c)))
    layer = 2.0 * n * 27 * CH * CH
    if kind == "conv":
        return dict(bytes=2 * CH * n * 5, flops=3 * layer)
    return dict(bytes=(12 * 7 + 4 + 32) * n + 4 * n * 2, flops=2.0 * 27 * n * sum(3 * a * b for a, b in LAYERS))


# ------------------------------------------------------------------ in 64 bits

def _conv64(x, w, b=None):
    """[D, H, W, ci] * [27, co, ci] in float64."""
    k = w.double().view(3, 3, 3, CH, CH).permute(3, 4, 0, 1, 2)
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    D, H, Wd = x.shape[:3]
    y = torch.zeros(D, H, Wd, CH, dtype=F64, device=x.device)
    for t in range(27):
        z, r, q = t // 9, (t // 3) % 3, t % 3
        y += xp[z:z + D, r:r + H, q:q + Wd] @ k[:, :, z, r, q].T
    return y if b is None else y + b.double()


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in SOLVE:
        xs = _system(c, seed)[1]
        return dict(x=xs) if kind == "mixed" else dict(x=xs, iters=None, status=None)
    if kind == "batched":
        sides, _ = _rectangles(c["nsys"], seed)
        return dict(x=_uniform(int((sides[:, 0] * sides[:, 1]).sum()), seed), status=None)
    if kind == "conv":
        s = _layer_inputs(c, seed)
        y = torch.relu(_conv64(s["x"], s["w"], s["b"]))
        flipped = s["w"].flip(0).transpose(1, 2)
        dx = _conv64(s["g"], flipped) * (s["x"] > 0)
        D, H, Wd = _dims(c)
        xp = torch.nn.functional.pad(s["x"].double(), (0, 0, 1, 1, 1, 1, 1, 1))
        g = s["g"].double().reshape(-1, CH)
        dw = torch.stack([g.T @ xp[t // 9:t // 9 + D, (t // 3) % 3:(t // 3) % 3 + H, t % 3:t % 3 + Wd].reshape(-1, CH)
                          for t in range(27)])
        return dict(y=y, dx=dx, dw=dw, db=g.sum(0))
    return None
