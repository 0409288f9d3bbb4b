"""The work that this library is used for, as cases that can be timed.

A case is a dict of plain values: what is called (`kind`), on which matrix
sequence (`family`, `nx`, `maps`), with which pattern level, precision and
refinement.  `prepare` makes a case's inputs on the GPU from a seed, `run` is
one pass through the public entry points, `work` the bytes and operations that
a pass cannot do without, `exact` the same outputs by plain torch in 64 bits.

Kinds
  maps     patterns of a sequence, then all its maps (the whole construction)
  step     one new matrix of a sequence: its pattern, its map, the map's
           residual and its product with a vector
  rebuild  the maps of a sequence of fixed sparsity from a captured plan
  train    independent pairs: maps and their adjoint in batched calls
  grad     one map through torch.autograd: the build, ||A M - A_0||_F^2 +
           ||M v||^2, and the gradients
  study    sparsified sources, the patterns of those, and the maps on them
  solve    GMRES on the systems of a sequence with its maps, a fixed number
           of steps

Families (the matrices' sizes and structures are those of `workloads.py`)
  fd5      5-point Laplacian plus a drifting diagonal
  cd5      5-point nonlinear convection-diffusion Jacobians
  q1       9-point bilinear finite elements, log-normal coefficient
  upwind   7-point upwind convection-diffusion in 3-D
  p1       linear finite elements on a jittered mesh whose edges flip: every
           matrix has its own structure
  band     about 85 random entries per column, nonsymmetric
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_17656_gb300 import autograd, sam

DEV = "cuda"


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # the smallest call: two matrices of 1024 rows, plain FP64, level 1;
        # launches and synchronisations are all it costs
        dict(name="fd5 32^2 l1 fp64", kind="maps", family="fd5", nx=32, maps=2, level=1, precision="fp64", steps=0),
        # one step of a time integration or Newton loop on a small grid: the
        # next Jacobian's pattern and map, checked and applied once
        dict(name="cd5 64^2 l2 step", kind="step", family="cd5", nx=64, maps=1, level=2, precision="fp32r", steps=1),
        # a comparison of pattern choices: 66 sparsified Jacobians, their
        # level-2 patterns, and the maps with automatic refinement
        dict(name="cd5 64^2 x66 study", kind="study", family="cd5", nx=64, maps=66, level=2, precision="fp32r", steps=-1,
             tau=0.8),
        # the benchmark's own workload: level-2 patterns and ten maps
        dict(name="q1 256^2 x10 l2", kind="maps", family="q1", nx=256, maps=10, level=2, precision="fp32r", steps=1),
        # the same construction in plain FP64, a user's reference
        dict(name="q1 256^2 x2 l2 fp64", kind="maps", family="q1", nx=256, maps=2, level=2, precision="fp64", steps=0),
        # level-3 patterns: 81 x 49 column problems
        dict(name="q1 256^2 x2 l3", kind="maps", family="q1", nx=256, maps=2, level=3, precision="fp32r", steps=1),
        # sensitivities of one level-2 map through autograd
        dict(name="q1 256^2 l2 grad", kind="grad", family="q1", nx=256, maps=1, level=2, precision="fp32r", steps=1),
        # training: 32 independent pairs, level 1, two refinement steps,
        # forward and adjoint
        dict(name="q1 512^2 x32 l1 train", kind="train", family="q1", nx=512, maps=32, level=1, precision="fp32r", steps=2),
        # a long 3-D sequence of fixed sparsity replayed from a plan
        dict(name="upwind 64^3 x20 l2 plan", kind="rebuild", family="upwind", nx=64, maps=20, level=2, precision="fp32r",
             steps=1),
        # a mesh whose structure changes: patterns and uneven columns of
        # sixteen different structures in one batch (odd order, 513^2)
        dict(name="p1 513^2 x16 l2", kind="maps", family="p1", nx=513, maps=16, level=2, precision="fp32r", steps=1),
        # dense rows (weather-model density): up to 201 x 96 column problems
        dict(name="band 7700 x2 l1", kind="maps", family="band", nx=7700, maps=2, level=1, precision="fp32r", steps=1),
        # the maps in use: nine systems, 60 steps of GMRES(30)
        dict(name="q1 256^2 x9 gmres", kind="solve", family="q1", nx=256, maps=9, level=2, precision="fp32r", steps=1,
             restart=30, iters=60),
    ]


# |J|, |I| and stored entries per column of an interior column, by family and
# level (p1, band: mean)
_COLS = {
    ("fd5", 1): (5, 13, 25), ("fd5", 2): (13, 25, 65), ("cd5", 1): (5, 13, 25), ("cd5", 2): (13, 25, 65),
    ("q1", 1): (9, 25, 81), ("q1", 2): (25, 49, 225), ("q1", 3): (49, 81, 441),
    ("upwind", 1): (7, 25, 49), ("upwind", 2): (25, 63, 175), ("p1", 1): (7, 19, 49), ("p1", 2): (19, 38, 135),
    ("band", 1): (86, 195, 7300),
}
_ROW = {"fd5": 5, "cd5": 5, "q1": 9, "upwind": 7, "p1": 7, "band": 86}


def _order(case):
    f, nx = case["family"], case["nx"]
    return nx if f == "band" else nx**3 if f == "upwind" else nx * nx


def _flops(case):
    J, I, nB = _COLS[(case["family"], case["level"])]
    cols = case["maps"] * _order(case)
    steps = 2 if case["steps"] < 0 else case["steps"]
    # normal equations, their factor, and per step the residual, B^T r and two
    # triangular solves: fewer operations than any orthogonal factorisation
    solve = I * J * J + J**3 / 3 + 2 * nB + 2 * J * J
    per = solve + steps * (4 * nB + 2 * J * J)
    if case["kind"] in ("train", "grad"):
        per += solve + 2 * J * J + 9 * nB
    if case["kind"] == "solve":
        per = case["iters"] * (2 * (_ROW[case["family"]] + 2 * J) + 4 * case["restart"] / 2 + 3)
    return per * cols


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["maps", "maps", "maps", "step", "rebuild", "train", "grad", "study", "solve"])
    case = {"kind": kind, "precision": "fp32r", "steps": rng.choice([1, 1, 2, -1])}
    if kind == "maps":
        case["family"] = rng.choice(["fd5", "q1", "upwind", "p1", "band"])
    elif kind == "study":
        case.update(family="cd5", tau=rng.choice([0.7, 0.8, 0.9]))
    elif kind == "solve":
        case.update(family="q1", restart=rng.choice([20, 30, 40]), iters=rng.randrange(30, 70), steps=1)
    elif kind == "step":
        case["family"] = rng.choice(["cd5", "q1", "upwind", "p1"])
    else:
        case["family"] = rng.choice(["q1", "upwind", "p1"] if kind != "rebuild" else ["q1", "upwind"])
    f = case["family"]
    case["level"] = 1 if f == "band" else 2 if kind in ("solve", "study") else rng.choice([1, 2, 2])
    if kind == "maps" and f == "q1" and rng.random() < 0.3:
        case["level"] = 3
    if kind == "maps" and f != "band" and case["level"] < 3 and rng.random() < 0.2:
        case.update(precision="fp64", steps=0)
    if kind in ("step", "grad"):
        case["maps"] = 1
    else:
        case["maps"] = {"study": log(8, 66), "solve": rng.randrange(1, 10), "train": log(2, 32)}.get(kind) or log(2, 20)
    if kind == "train":
        case["level"] = 1
    # columns of the whole batch, held to what the largest listed case costs
    most = 8.0e6 if case["level"] == 1 else 4.0e6
    if case["level"] == 3:
        most = 1.3e5
    if f == "band":
        most = 1.5e4
    if case["precision"] == "fp64":
        most /= 10
    if kind == "solve":
        most = 6.0e5
    if kind == "study":
        most = 3.0e5
    # (60 steps solve a small system to its last digit: nothing to compare)
    n = log(1.0e4 if kind == "solve" else 900, max(1000, min(2.7e5, most / case["maps"])))
    case["nx"] = n if f == "band" else max(8, int(round(n ** (1 / 3)))) if f == "upwind" else max(24, int(round(n**0.5)))
    return case


def work(case):
    J, I, nB = _COLS[(case["family"], case["level"])]
    n, K, row = _order(case), case["maps"], _ROW[case["family"]]
    src = 12 * n * row + 4 * n  # one matrix: structure and values
    mp = 12 * n * J + 4 * n     # one map
    kind = case["kind"]
    byts = {
        "maps": (K + 1) * src + K * (mp + 12 * n),
        "step": 2 * src + mp + 28 * n,
        "rebuild": (K + 1) * 8 * n * row + K * (8 * n * J + 8 * n),
        "train": 2 * K * src + K * (mp + 8 * n * J) + 2 * K * 8 * n * row,
        "grad": 2 * src + mp + 16 * n * row + 16 * n,
        "study": (K + 1) * src + K * (mp + 12 * n),
        "solve": K * (src + mp) + mp + K * 16 * n + case.get("iters", 0) * K * 8 * n,
    }[kind]
    return {"bytes": float(byts), "flops": float(_flops(case))}


# ------------------------------------------------------------------ matrices
# A sequence is made as a list of (indptr, indices, values) in CSR, columns
# ascending; the values of every entry are sums in a fixed order.


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _field(m, g, ell=0.1):
    """A smooth random field on m x m cells of the unit square, mean 0, variance 1."""
    k = torch.fft.fftfreq(2 * m, d=1.0 / m, device=DEV, dtype=torch.float64)
    w = torch.randn((2 * m, 2 * m), generator=g, device=DEV, dtype=torch.float64)
    amp = torch.exp(-math.pi**2 * ell**2 * (k[:, None] ** 2 + k[None, :] ** 2))
    f = torch.fft.ifft2(torch.fft.fft2(w) * amp).real[:m, :m]
    return (f - f.mean()) / f.std()


def _stencil(offsets, values, present):
    """CSR from per-row slots: slot s of row i holds column i + offsets[s]
    (ascending offsets) where present[:, s]."""
    n = values.shape[0]
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = present.sum(1).cumsum(0)
    col = torch.arange(n, device=DEV)[:, None] + torch.tensor(offsets, device=DEV)[None, :]
    return ptr.to(torch.int32), col[present].to(torch.int32), values[present].contiguous()


def _grid2(nx, offs):
    """present[i, s] for the neighbours (dy, dx) of an nx x nx grid."""
    y, x = torch.meshgrid(torch.arange(nx, device=DEV), torch.arange(nx, device=DEV), indexing="ij")
    return torch.stack([((y + dy >= 0) & (y + dy < nx) & (x + dx >= 0) & (x + dx < nx)).reshape(-1) for dy, dx in offs], 1)


_OFF5 = [(-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)]
_OFF9 = [(dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]


def _fd5(nx, K, g):
    pres = _grid2(nx, _OFF5)
    base = torch.tensor([-1.0, -1.0, 4.0, -1.0, -1.0], device=DEV, dtype=torch.float64).repeat(nx * nx, 1)
    mats = []
    for k in range(K):
        v = base.clone()
        if k:
            v[:, 2] += _uniform(g, nx * nx, 0.0, 0.5)
        mats.append(_stencil([dy * nx + dx for dy, dx in _OFF5], v, pres))
    return mats


def _cd5(nx, K, g):
    """Jacobian-like: -div(k(u) grad) + convection, u drifting along the sequence."""
    pres = _grid2(nx, _OFF5)
    h = 1.0 / (nx + 1)
    u0, du = 0.3 * _field(nx + 2, g), 0.05 * _field(nx + 2, g)
    mats = []
    for k in range(K):
        u = u0 + du * k / max(K - 1, 1)
        c = 0.1 + u * u
        mid = c[1:-1, 1:-1]
        face = {(0, 1): c[1:-1, 2:], (0, -1): c[1:-1, :-2], (1, 0): c[2:, 1:-1], (-1, 0): c[:-2, 1:-1]}
        val = {o: -(mid + f) / (2 * h * h) + (o[0] + o[1]) / (2 * h) for o, f in face.items()}
        val[(0, 0)] = sum((mid + f) / (2 * h * h) for f in face.values())
        mats.append(_stencil([dy * nx + dx for dy, dx in _OFF5], torch.stack([val[o].reshape(-1) for o in _OFF5], 1), pres))
    return mats


def _q1_values(kap):
    a, b, c, d = kap[:-1, :-1], kap[:-1, 1:], kap[1:, :-1], kap[1:, 1:]  # the cells around each node
    v = {(-1, -1): -2 * a, (-1, 0): -(a + b), (-1, 1): -2 * b, (0, -1): -(a + c), (0, 0): 4 * (a + b + c + d),
         (0, 1): -(b + d), (1, -1): -2 * c, (1, 0): -(c + d), (1, 1): -2 * d}
    return torch.stack([v[o].reshape(-1) / 6.0 for o in _OFF9], 1)


def _q1(nx, K, g, drift=0.05):
    pres = _grid2(nx, _OFF9)
    off = [dy * nx + dx for dy, dx in _OFF9]
    kap = torch.exp(_field(nx + 1, g))
    mats = [_stencil(off, _q1_values(kap), pres)]
    for k in range(1, K):
        mats.append(_stencil(off, _q1_values(kap * torch.exp(drift * k * _field(nx + 1, g))), pres))
    return mats


def _upwind(nx, K, g):
    offs = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)]
    z, y, x = torch.meshgrid(*[torch.arange(nx, device=DEV)] * 3, indexing="ij")
    pres = torch.stack([((z + a >= 0) & (z + a < nx) & (y + b >= 0) & (y + b < nx) & (x + c >= 0) & (x + c < nx)).reshape(-1)
                        for a, b, c in offs], 1)
    h = 1.0 / (nx + 1)
    turn = float(_uniform(g, 1, 0.0, 2 * math.pi))
    mats = []
    for k in range(K):
        pe = 10.0 + 90.0 * k / max(K - 1, 1)
        th = turn + math.radians(5.0 * k)
        w = (math.cos(th) - 0.5 * math.sin(th), math.sin(th) + 0.5 * math.cos(th), 0.25)  # x, y, z
        row = []
        for o in offs:
            d = [i for i in range(3) if o[i]]
            if not d:
                row.append(6.0 + pe * h * sum(abs(t) for t in w))
            else:
                wd, s = w[2 - d[0]], o[d[0]]
                row.append(-1.0 - pe * h * (max(wd, 0.0) if s < 0 else max(-wd, 0.0)))
        # (a small reaction term that varies in space: no two columns are alike)
        v = torch.tensor(row, device=DEV, dtype=torch.float64).repeat(nx**3, 1)
        v[:, 3] += _uniform(g, nx**3, 0.0, 0.1)
        mats.append(_stencil([a * nx * nx + b * nx + c for a, b, c in offs], v, pres))
    return mats


def _p1(nv, K, g):
    nc, h = nv - 1, 1.0 / (nv - 1)
    t = torch.arange(nv, device=DEV, dtype=torch.float64) * h
    px = t[None, :] + _uniform(g, (nv, nv), -0.3 * h, 0.3 * h)
    py = t[:, None] + _uniform(g, (nv, nv), -0.3 * h, 0.3 * h)
    corner = [(0, 0), (0, 1), (1, 0), (1, 1)]  # (dy, dx)

    def local(tri, c):
        """3 x 3 element matrices of the triangle over the given corners of every cell."""
        P = [(px[a:a + nc, b:b + nc], py[a:a + nc, b:b + nc]) for a, b in (corner[q] for q in tri)]
        det = (P[1][0] - P[0][0]) * (P[2][1] - P[0][1]) - (P[1][1] - P[0][1]) * (P[2][0] - P[0][0])
        area = 0.5 * det.abs()
        gx = [(P[(q + 1) % 3][1] - P[(q + 2) % 3][1]) / det for q in range(3)]
        gy = [(P[(q + 2) % 3][0] - P[(q + 1) % 3][0]) / det for q in range(3)]
        return {(tri[a], tri[b]): area * (gx[a] * gx[b] + gy[a] * gy[b]) + c * area / 12.0 * (2.0 if a == b else 1.0)
                for a in range(3) for b in range(3)}

    gm = _gen(4000)  # the mesh's edges are one mesh's at every seed; positions and values are the seed's
    flip = _uniform(gm, (nc, nc)) < 0.5
    pos = {o: s for s, o in enumerate(_OFF9)}
    inside = _grid2(nv, _OFF9)
    mats = []
    for k in range(K):
        if k:
            flip = flip ^ (_uniform(gm, (nc, nc)) < 0.01)
        c = 0.1 * 100.0 ** (k / max(K - 1, 1))
        val = torch.zeros((9, nv, nv), device=DEV, dtype=torch.float64)
        has = torch.zeros((9, nv, nv), device=DEV, dtype=torch.bool)
        # corners 0 (0,0), 1 (0,1), 2 (1,0), 3 (1,1); the diagonal is 0-3, or 1-2 where flipped
        for tri, on in (((0, 1, 3), ~flip), ((0, 3, 2), ~flip), ((0, 1, 2), flip), ((1, 3, 2), flip)):
            for (a, b), e in local(tri, c).items():
                (ay, ax), (by, bx) = corner[a], corner[b]
                s = pos[(by - ay, bx - ax)]
                val[s, ay:ay + nc, ax:ax + nc] += torch.where(on, e, 0.0)
                has[s, ay:ay + nc, ax:ax + nc] |= on
        mats.append(_stencil([dy * nv + dx for dy, dx in _OFF9], val.reshape(9, -1).T.contiguous(),
                             has.reshape(9, -1).T & inside))
    return mats


def _band(n, K, g, half=50, keep=0.85):
    off = torch.arange(-half, half + 1, device=DEV)
    col = torch.arange(n, device=DEV)[:, None] + off[None, :]
    # one structure at every seed
    pres = (col >= 0) & (col < n) & ((_uniform(_gen(7000), (n, 2 * half + 1)) < keep) | (off == 0))
    base = _uniform(g, (n, 2 * half + 1), -1.0, 1.0)
    mats = []
    for k in range(K):
        v = base * (1.0 + 0.05 * k * _uniform(g, (n, 2 * half + 1), -1.0, 1.0))
        v = torch.where(pres, v, 0.0)
        v[:, half] = 0.0
        v[:, half] = v.abs().sum(1) + 1.0
        mats.append(_stencil(off.tolist(), v, pres))
    return mats


_MAKE = {"fd5": _fd5, "cd5": _cd5, "q1": _q1, "upwind": _upwind, "p1": _p1, "band": _band}


def _inputs(case, seed):
    """The CSR matrices of a case, the index of each map's source and of its target, and its random vectors."""
    g = _gen(seed)
    f, nx, K, kind = case["family"], case["nx"], case["maps"], case["kind"]
    if kind == "train":  # independent (A_0, A_1) pairs
        pairs = [_MAKE[f](nx, 2, g) for _ in range(K)]
        mats, src, tgt = [m for p in pairs for m in p], list(range(1, 2 * K, 2)), list(range(0, 2 * K, 2))
    elif kind in ("step", "grad"):
        mats, src, tgt = _MAKE[f](nx, 2, g), [1], [0]
    elif kind == "solve":
        mats, src, tgt = _MAKE[f](nx, K + 1, g), list(range(1, K + 1)), [0]
    else:
        mats, src, tgt = _MAKE[f](nx, K, g), list(range(K)), [0]
    n = mats[0][0].numel() - 1
    vec = torch.randn(K * n, generator=g, device=DEV, dtype=torch.float64)
    return mats, src, tgt, vec, g


# ------------------------------------------------------------- prepare and run


def _steps(case):
    return "auto" if case["steps"] < 0 else case["steps"]


def prepare(case, seed):
    mats, src, tgt, vec, g = _inputs(case, seed)
    csr = [sam.Csr(*m) for m in mats]
    n, K = csr[0].n, case["maps"]
    st = {"case": case, "h": sam.Handle(), "A": [csr[i] for i in src], "Z": [csr[i] for i in tgt], "n": n, "K": K, "vec": vec}
    st["stat"] = torch.empty(K * n, dtype=torch.int32, device=DEV)
    st["res2"] = torch.empty(K * n, dtype=torch.float64, device=DEV)
    h, kind, steps = st["h"], case["kind"], _steps(case)
    if kind == "rebuild":
        ps = h.sam_pattern_build_batched(st["A"], case["level"])
        st["plan"] = h.sam_plan_create(st["A"], st["Z"][0], ps, case["precision"], steps, want_status=True, want_res2=True)
        h.sam_sync()
        del ps
    elif kind == "study":
        # arrays with room for the patterns of the whole matrices
        st["ci"] = torch.zeros(K * n * 13, dtype=torch.int32, device=DEV)
        st["v"] = torch.zeros(K * n * 13, dtype=torch.float64, device=DEV)
    elif kind == "train":
        # the patterns of a training set are fixed, the loss's gradient comes from outside
        st["ps"] = h.sam_pattern_build_batched(st["A"], case["level"])
        st["dm"] = torch.randn(sum(p.nnz for p in st["ps"]), generator=g, device=DEV, dtype=torch.float64)
    elif kind == "grad":
        a, z = st["A"][0], st["Z"][0]
        st["ps"] = h.sam_pattern_build(a, case["level"])
        st["map"] = autograd.SamMap(h, (a.indptr, a.indices), (z.indptr, z.indices), st["ps"], case["precision"], steps)
    elif kind == "solve":
        # the maps and P_0, a sparse approximate inverse of A_0
        A0 = st["Z"][0]
        eye = sam.Csr(torch.arange(n + 1, dtype=torch.int32, device=DEV), torch.arange(n, dtype=torch.int32, device=DEV),
                      torch.ones(n, dtype=torch.float64, device=DEV))
        p0 = h.sam_pattern_build(A0, case["level"])
        st["P"] = sam.Csr(*h.sam_build(A0, eye, p0, "fp64", 0))
        ps = h.sam_pattern_build_batched(st["A"], case["level"])
        offs, rp, ci, v, _ = h.sam_build_batched(st["A"], A0, ps, "fp64", 0)
        h.sam_sync()
        st["M"] = [sam.Csr(rp[k * (n + 1):(k + 1) * (n + 1)], ci[offs[k]:offs[k + 1]], v[offs[k]:offs[k + 1]]) for k in range(K)]
    return st


def run(state):
    s, c, h = state, state["case"], state["h"]
    kind, prec, steps, level = c["kind"], c["precision"], _steps(c), c["level"]
    A, Z = s["A"], s["Z"]
    if kind in ("maps", "study"):
        src = h.sam_sparsify_batched(A, "tau", c["tau"]) if kind == "study" else A
        ps = h.sam_pattern_build_batched(src, level)
        offs, rp, ci, v, _ = h.sam_build_batched(A, Z[0], ps, prec, steps, M_col_idx=s.get("ci"), M_val=s.get("v"),
                                               col_status=s["stat"], res2=s["res2"])
        return {"offsets": offs, "indptr": rp, "indices": ci, "values": v, "status": s["stat"], "res2": s["res2"]}
    if kind == "step":
        p = h.sam_pattern_build(A[0], level)
        rp, ci, v = h.sam_build(A[0], Z[0], p, prec, steps)
        M = sam.Csr(rp, ci, v)
        fro, rel = h.sam_residual(A[0], M, Z[0])
        return {"indptr": rp, "indices": ci, "values": v, "fro": fro, "rel": rel, "y": h.sam_apply(M, s["vec"])}
    if kind == "rebuild":
        p = s["plan"]
        p.execute()
        return {"values": p.M_val, "status": p.col_status, "res2": p.res2, "fro2": p.fro2}
    if kind == "train":
        offs, rp, ci, v, _ = h.sam_build_batched(A, Z, s["ps"], prec, steps, col_status=s["stat"], res2=s["res2"])
        da, dz = h.sam_build_backward_batched(A, Z, s["ps"], v, s["dm"], prec, steps, 1.0, offsets=offs)
        return {"indptr": rp, "indices": ci, "values": v, "status": s["stat"], "res2": s["res2"], "dA": da, "dZ": dz}
    if kind == "grad":
        a = A[0].data.detach().requires_grad_()
        z = Z[0].data.detach().requires_grad_()
        f = s["map"]
        m = f(a, z)
        y = f.matvec(m, s["vec"])
        loss = f.residual_sq(a, z, m) + (y * y).sum()
        loss.backward()
        return {"values": m.detach(), "y": y.detach(), "loss": loss.detach(), "dA": a.grad, "dZ": z.grad}
    hist = torch.empty(s["K"] * c["iters"], dtype=torch.float64, device=DEV)
    x, its, rel = h.sam_gmres_batched(A, s["vec"], Ms=s["M"], P_0=s["P"], restart=c["restart"], maxiter=c["iters"],
                                      rtol=1e-12, history=hist)
    return {"x": x, "steps": its, "relres": rel, "history": hist}


# ---------------------------------------------------------- the same in 64 bits
# Plain torch, dense column problems: normal equations by Cholesky with
# refinement, FP64 throughout.


def _csc(n, m):
    """(colptr, rows, positions in the CSR) of a CSR matrix."""
    rp, ci = m[0].long(), m[1].long()
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    perm = torch.argsort(ci * n + row)
    cp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    cp[1:] = torch.bincount(ci, minlength=n).cumsum(0)
    return cp, row[perm], perm


def _expand(owner, cp, col):
    """For every (owner, column) pair, the entries of that column: owner's index per entry, and the entry."""
    cnt = cp[col + 1] - cp[col]
    rep = torch.repeat_interleave(torch.arange(col.numel(), device=DEV), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    e = cp[col][rep] + torch.arange(rep.numel(), device=DEV) - first[rep]
    return rep, e


def _pattern(n, m, level):
    """CSC (colptr, rows) of the level-L neighbourhoods of a CSR matrix's graph."""
    cp, ri, _ = _csc(n, m)
    key = torch.arange(n, device=DEV) * (n + 1)  # column * n + row: the diagonal
    for _ in range(level):
        rep, e = _expand(None, cp, key % n)
        key = torch.unique(torch.cat([key, (key // n)[rep] * n + ri[e]]))
    jp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    jp[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return jp, key % n


class _Columns:
    """The column problems of one structure (source, target, pattern), dense and in chunks."""

    def __init__(self, n, src, tgt, pat):
        self.n = n
        self.jp, self.jr = pat
        self.cp, self.ri, self.perm = _csc(n, src)
        self.zp, self.zr, self.zperm = _csc(n, tgt)
        jcol = torch.repeat_interleave(torch.arange(n, device=DEV), self.jp[1:] - self.jp[:-1])
        self.rep, self.ent = _expand(None, self.cp, self.jr)
        self.tcol = jcol[self.rep]
        self.tloc = (torch.arange(self.jr.numel(), device=DEV) - self.jp[jcol])[self.rep]
        key = self.tcol * n + self.ri[self.ent]
        uniq, inv = torch.unique(key, return_inverse=True)
        ip = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        ip[1:] = torch.bincount(uniq // n, minlength=n).cumsum(0)
        self.trow = inv - ip[self.tcol]
        zcol = torch.repeat_interleave(torch.arange(n, device=DEV), self.zp[1:] - self.zp[:-1])
        zkey = zcol * n + self.zr
        at = torch.searchsorted(uniq, zkey).clamp(max=uniq.numel() - 1)
        self.zin = uniq[at] == zkey
        self.zcol, self.zloc = zcol, at - ip[zcol]
        self.ni, self.nj = int((ip[1:] - ip[:-1]).max()), int((self.jp[1:] - self.jp[:-1]).max())
        self.tptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        self.tptr[1:] = torch.bincount(self.tcol, minlength=n).cumsum(0)
        # map entry p (CSC) -> CSR order
        order = torch.argsort(self.jr * n + jcol)
        self.order, self.jcol = order, jcol
        self.ci = jcol[order].to(torch.int32)
        self.chunk = max(1, min(n, int(1.5e9 // (8 * self.ni * self.nj))))

    def csr_ptr(self):
        p = torch.zeros(self.n + 1, dtype=torch.int64, device=DEV)
        p[1:] = torch.bincount(self.jr, minlength=self.n).cumsum(0)
        return p

    def solve(self, av, zv, dm=None, w=0.0, no_dm=False):
        """Map values (CSR order) and squared residuals; with dm (CSR order) or w also the gradients."""
        n, adj = self.n, dm is not None
        av, zc = av[self.perm], zv[self.zperm]
        m_out = torch.empty(self.jr.numel(), device=DEV, dtype=torch.float64)
        res2 = torch.empty(n, device=DEV, dtype=torch.float64)
        out2 = torch.zeros(n, device=DEV, dtype=torch.float64)
        out2.index_add_(0, self.zcol[~self.zin], zc[~self.zin] ** 2)
        if adj:
            dm_c = torch.empty_like(m_out)
            dm_c[self.order] = dm
            da = torch.zeros(av.numel(), device=DEV, dtype=torch.float64)
            dz = torch.where(self.zin, 0.0, 2 * w * zc)
        for j0 in range(0, n, self.chunk):
            j1 = min(n, j0 + self.chunk)
            t = slice(int(self.tptr[j0]), int(self.tptr[j1]))
            p = slice(int(self.jp[j0]), int(self.jp[j1]))
            z = slice(int(self.zp[j0]), int(self.zp[j1]))
            B = torch.zeros((j1 - j0, self.ni, self.nj), device=DEV, dtype=torch.float64)
            tc, tr, tl = self.tcol[t] - j0, self.trow[t], self.tloc[t]
            B[tc, tr, tl] = av[self.ent[t]]
            c = torch.zeros((j1 - j0, self.ni, 1), device=DEV, dtype=torch.float64)
            zin, zcol, zloc = self.zin[z], self.zcol[z] - j0, self.zloc[z]
            c[zcol[zin], zloc[zin], 0] = zc[z][zin]
            Bt = B.transpose(1, 2)
            G = Bt @ B
            nj = (self.jp[j0 + 1:j1 + 1] - self.jp[j0:j1])
            pad = torch.arange(self.nj, device=DEV)[None, :] >= nj[:, None]
            G += torch.diag_embed(pad.to(torch.float64))
            L = torch.linalg.cholesky(G)
            del G
            m = torch.cholesky_solve(Bt @ c, L)
            for _ in range(3):
                m = m + torch.cholesky_solve(Bt @ (c - B @ m), L)
            r = c - B @ m
            loc = torch.arange(p.start, p.stop, device=DEV) - self.jp[self.jcol[p]]
            pc = self.jcol[p] - j0
            m_out[p] = m[pc, loc, 0]
            res2[j0:j1] = (r * r).sum((1, 2))
            if adj:
                gvec = torch.zeros_like(m)
                gvec[pc, loc, 0] = dm_c[p]
                lam = torch.cholesky_solve(gvec, L)
                for _ in range(3):
                    lam = lam + torch.cholesky_solve(gvec - Bt @ (B @ lam), L)
                bl = B @ lam
                d = r[tc, tr, 0] * lam[tc, tl, 0] - bl[tc, tr, 0] * m[tc, tl, 0] - 2 * w * r[tc, tr, 0] * m[tc, tl, 0]
                da.index_add_(0, self.ent[t], d)
                dzc = (bl + 2 * w * r)[zcol, zloc.clamp(0, self.ni - 1), 0]
                dz[z] = torch.where(zin, dzc, dz[z])
            del B, L
        out = {"values": m_out[self.order], "res2": res2 + out2}
        if adj:
            out["dA"], out["dZ"] = torch.empty_like(da), torch.empty_like(dz)
            out["dA"][self.perm], out["dZ"][self.zperm] = da, dz
        return out


def _sparsified(n, m, tau):
    """The entries above (1 - tau) of their column's largest magnitude, and the diagonal."""
    rp, ci, v = m[0].long(), m[1].long(), m[2].abs()
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    top = torch.zeros(n, device=DEV, dtype=torch.float64).scatter_reduce_(0, ci, v, "amax")
    keep = (row == ci) | (v > (1.0 - tau) * top[ci])
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.bincount(row[keep], minlength=n).cumsum(0)
    return ptr, ci[keep], m[2][keep]


def _times(n, ptr, ci, v, x):
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (ptr[1:] - ptr[:-1]).long())
    return torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, row, v * x[ci.long()])


def _gmres(n, apply, b, restart, iters):
    """Restarted GMRES of a right-preconditioned operator: (x = update of z, history)."""
    x, hist = torch.zeros_like(b), []
    bn = float(b.norm())
    mul, pre = apply
    while len(hist) < iters:
        r = b - mul(x)
        beta = float(r.norm())
        V = torch.zeros((restart + 1, n), device=DEV, dtype=torch.float64)
        V[0] = r / beta
        H = np.zeros((restart + 1, restart))
        k = 0
        while k < restart and len(hist) < iters:
            w = mul(pre(V[k]))
            for _ in range(2):
                hk = V[:k + 1] @ w
                w = w - hk @ V[:k + 1]
                H[:k + 1, k] += hk.cpu().numpy()
            H[k + 1, k] = float(w.norm())
            V[k + 1] = w / H[k + 1, k]
            k += 1
            e1 = np.zeros(k + 1)
            e1[0] = beta
            y, *_ = np.linalg.lstsq(H[:k + 1, :k], e1, rcond=None)
            hist.append(float(np.linalg.norm(e1 - H[:k + 1, :k] @ y)) / bn)
        x = x + pre(torch.from_numpy(y).to(DEV) @ V[:k])
    return x, hist


def exact(case, seed):
    mats, src, tgt, vec, g = _inputs(case, seed)
    kind, K, level = case["kind"], case["maps"], case["level"]
    n = mats[0][0].numel() - 1
    cat = lambda parts, key: torch.cat([p[key] for p in parts])  # noqa: E731

    cols = None

    def columns(a, z, pattern_of=None):
        nonlocal cols
        own = case["family"] == "p1" or pattern_of is not None
        if cols is None or own:
            cols = _Columns(n, a, z, _pattern(n, pattern_of or a, level))
        return cols

    parts = []
    if kind in ("maps", "study", "rebuild"):
        z = mats[tgt[0]]
        for i in src:
            sp = _sparsified(n, mats[i], case["tau"]) if kind == "study" else None
            parts.append(columns(mats[i], z, sp).solve(mats[i][2], z[2]))
        out = {"values": cat(parts, "values"), "status": None, "res2": cat(parts, "res2")}
        if kind == "rebuild":
            return {**out, "fro2": torch.stack([p["res2"].sum() for p in parts])}
        if kind == "study":
            v = torch.zeros(K * n * 13, device=DEV, dtype=torch.float64)
            v[:out["values"].numel()] = out["values"]
            out["values"] = v
        return {**out, "offsets": None, "indptr": None, "indices": None}
    if kind == "step":
        a, z = mats[src[0]], mats[tgt[0]]
        C = columns(a, z)
        p = C.solve(a[2], z[2])
        fro = math.sqrt(float(p["res2"].sum()))
        return {"indptr": None, "indices": None, "values": p["values"], "fro": fro, "rel": fro / float(z[2].norm()),
                "y": _times(n, C.csr_ptr(), C.ci, p["values"], vec)}
    if kind == "train":
        dm, at = None, 0
        for k in range(K):
            a, z = mats[src[k]], mats[tgt[k]]
            C = columns(a, z)
            if dm is None:  # drawn for all maps at once, as prepare() does
                tot = sum(_pattern(n, mats[i], level)[1].numel() for i in src) if case["family"] == "p1" else K * C.jr.numel()
                dm = torch.randn(tot, generator=g, device=DEV, dtype=torch.float64)
            m = C.jr.numel()
            parts.append(C.solve(a[2], z[2], dm[at:at + m], 1.0))
            at += m
        return {"indptr": None, "indices": None, "status": None, **{k: cat(parts, k) for k in ("values", "res2", "dA", "dZ")}}
    if kind == "grad":
        a, z = mats[src[0]], mats[tgt[0]]
        C = columns(a, z)
        m = C.solve(a[2], z[2])
        ptr = C.csr_ptr()
        y = _times(n, ptr, C.ci, m["values"], vec)
        row = torch.repeat_interleave(torch.arange(n, device=DEV), ptr[1:] - ptr[:-1])
        p = C.solve(a[2], z[2], 2 * y[row] * vec[C.ci.long()], 1.0)
        return {"values": m["values"], "y": y, "loss": p["res2"].sum() + (y * y).sum(), "dA": p["dA"], "dZ": p["dZ"]}
    # solve
    A0 = mats[tgt[0]]
    C = columns(mats[src[0]], A0)
    i = torch.arange(n, device=DEV)
    eye = (torch.arange(n + 1, dtype=torch.int32, device=DEV), i.to(torch.int32), torch.ones(n, device=DEV, dtype=torch.float64))
    CP = _Columns(n, A0, eye, _pattern(n, A0, level))
    pv = CP.solve(A0[2], eye[2])["values"]

    def matrix(ptr, ci, v):
        return torch.sparse_csr_tensor(ptr.long(), ci.long(), v, size=(n, n))

    P = matrix(CP.csr_ptr(), CP.ci, pv)
    xs, hs = [], []
    for k in range(K):
        a = mats[src[k]]
        M = matrix(C.csr_ptr(), C.ci, C.solve(a[2], A0[2])["values"])
        A = matrix(*a)
        x, hist = _gmres(n, (lambda q: A @ q, lambda q: M @ (P @ q)), vec[k * n:(k + 1) * n], case["restart"], case["iters"])
        xs.append(x)
        hs += [hist]
    return {"x": torch.cat(xs), "steps": None, "relres": np.array([q[-1] for q in hs]),
            "history": torch.tensor(hs, dtype=torch.float64).reshape(-1)}
