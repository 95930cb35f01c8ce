"""The work users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values.  Its "op" names the public call, "shape" the structure of the
operands, and the rest their sizes, the value type and the workspace policy:

  spgemm  C(i,j)   = A(i,k) B(k,j)      Context.spgemm        uniform rows, power law, stencil
  ttm     C(i,j,l) = A(i,j,k) B(k,l)    Context.ttm           uniform coordinates
  outer   C(i,j)   = A(k,i) B(k,j)      Context.spgemm_outer  live rows of equal length
  spttm, spttm_i, spmttkrp              Context.scatter_coo   uniform coordinates

Every call runs the symbolic pass (sizes, row pointer) and the numeric pass (coordinates, values)
and returns the whole result, newly allocated, as a program that multiplies sparse operands gets it.
The operands are made on the GPU.  The case fixes which entries a structure has up to a relabelling;
the seed draws the relabelling (a rotation of an index, which keeps every size of the result, so that
results of two seeds can be laid side by side) and all values.  Values are uniform in [-1, 1] ([0.5,
1.5] for the stencil, as a discretised operator has them).
"""
import math
import zlib

import numpy as np
import torch

from paper_2404_04541_b200 import api
from paper_2404_04541_b200 import binding

DEVICE = "cuda"
I32, I64 = torch.int32, torch.int64


def listed():
    return [
        # The smallest call: a small sparse product inside a larger program, where launches and host
        # work are all there is (2048 x 2048, 8 entries per row: the first benchmark configuration).
        dict(name="uniform_2048_f64", op="spgemm", shape="uniform", m=2048, k=2048, n=2048, da=8, db=8, f64=True, policy="auto"),
        # An ordinary rectangular product with odd extents in single precision: about 140 products a row.
        dict(name="uniform_odd_f32", op="spgemm", shape="uniform", m=30011, k=25013, n=20011, da=11, db=13, f64=False, policy="auto"),
        # A mid-size graph squared (paths of length two) in single precision: skewed rows that fit the caches.
        dict(name="powerlaw_16381_f32", op="spgemm", shape="powerlaw", n=16381, degree=16, f64=False, policy="auto"),
        # The largest: the power-law graph of the benchmark, 2^18 vertices of average degree 16, squared:
        # 2.9e9 products, 1.3e9 outputs.
        dict(name="powerlaw_2^18_f64", op="spgemm", shape="powerlaw", n=1 << 18, degree=16, f64=True, policy="auto"),
        # The benchmark's discretised operator squared, as a multigrid set-up does: 27-point stencil on 64^3.
        dict(name="stencil_64_f64", op="spgemm", shape="stencil", nx=64, ny=64, nz=64, f64=True, policy="auto"),
        # The same on a ragged grid in single precision, with the paper's sparse workspace asked for by name.
        dict(name="stencil_odd_ism_f32", op="spgemm", shape="stencil", nx=41, ny=37, nz=53, f64=False, policy="ism"),
        # Rows spread over 2^26 columns (the benchmark's wide configuration): every row is short, B is 2.7 GB.
        dict(name="wide_2^26_f32", op="spgemm", shape="uniform", m=1 << 16, k=1 << 26, n=1 << 26, da=4, db=4, f64=False, policy="auto"),
        # The benchmark's hyper-sparse 3-tensor times a matrix: most fibres hold one entry.
        dict(name="ttm_4096_f64", op="ttm", i=4096, j=4096, k=4096, nnz=1 << 21, n=4096, db=8, f64=True, policy="auto"),
        # A denser tensor with odd extents in single precision: fibres of about nine entries, 110 products each.
        dict(name="ttm_odd_f32", op="ttm", i=311, j=523, k=1201, nnz=1500007, n=3001, db=12, f64=False, policy="auto"),
        # The paper's second-order sweep at its middle: 10^4 x 10^4 outputs from 100 live coordinates.
        dict(name="outer_10000_f64", op="outer", i=10000, k=10000, n=10000, live=100, da=1000, db=1000, f64=True, policy="auto"),
        # The outer-product form over an output too wide for a dense workspace: A^T B of two tall matrices.
        dict(name="outer_wide_f32", op="outer", i=200003, k=50021, n=180001, live=50021, da=14, db=17, f64=False, policy="auto"),
        # A higher-order scatter with a coordinate-form result: the outermost mode of a 3-tensor contracted
        # with a matrix that is 1 % dense.
        dict(name="spttm_f64", op="spttm", i=512, j=1024, k=2048, nnz=1 << 20, n=4096, db=41, f64=True, policy="auto"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: smaller than the largest listed one, odd sizes among them."""
    f64 = rng.random() < 0.5
    kind = rng.choice(("uniform", "uniform", "powerlaw", "powerlaw", "stencil", "stencil", "ttm", "ttm", "outer", "coo"))
    if kind == "uniform":
        da, db = _log(rng, 2, 40), _log(rng, 2, 40)
        m = _log(rng, 500, min(400000, 60e6 / (da * db)))
        k = max(db, _log(rng, max(500, m / 4), m * 4))
        n = max(db, _log(rng, 1000, 1 << 24))
        return dict(op="spgemm", shape="uniform", m=m, k=k, n=n, da=da, db=db, f64=f64, policy="auto")
    if kind == "powerlaw":
        return dict(op="spgemm", shape="powerlaw", n=_log(rng, 1500, 200000), degree=rng.randint(4, 16), f64=f64, policy="auto")
    if kind == "stencil":
        side = _log(rng, 8, 72)
        nx, ny, nz = (max(4, int(side * rng.uniform(0.7, 1.3))) for _ in range(3))
        policy = rng.choice(("auto", "auto", "auto", "ism", "hash"))
        if policy != "auto":
            nx, ny, nz = min(nx, 45), min(ny, 45), min(nz, 45)
        return dict(op="spgemm", shape="stencil", nx=nx, ny=ny, nz=nz, f64=f64, policy=policy)
    if kind == "ttm":
        i, j, k = _log(rng, 100, 5000), _log(rng, 100, 5000), _log(rng, 100, 5000)
        nnz = min(_log(rng, 20000, 2500000), i * j * k // 8)
        db = rng.randint(3, 16)
        return dict(op="ttm", i=i, j=j, k=k, nnz=nnz, n=_log(rng, 64, 8192), db=db, f64=f64, policy="auto")
    if kind == "outer":
        i, n = _log(rng, 1000, 600000), _log(rng, 1000, 600000)
        da, db = _log(rng, 4, min(1000, i // 4)), _log(rng, 4, min(1000, n // 4))
        live = _log(rng, 10, max(11, min(100000, 40e6 / (da * db))))
        return dict(op="outer", i=i, k=live * rng.randint(1, 10), n=n, live=live, da=da, db=db, f64=f64, policy="auto")
    op = rng.choice(("spttm", "spttm_i", "spmttkrp"))
    i, j, k = _log(rng, 50, 2000), _log(rng, 50, 2000), _log(rng, 50, 2000)
    n = _log(rng, 64, 4096)
    db = max(2, min(64, int(n * rng.uniform(0.01, 0.1))))
    nnz = min(_log(rng, 20000, 1000000), i * j * k // 8, int(40e6 / db))
    return dict(op=op, i=i, j=j, k=k, nnz=nnz, n=n, db=db, f64=f64, policy="auto")


# ------------------------------------------------------------------ operands
def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _structure(case):
    """The generator that fixes a case's structure: the same for every seed."""
    return _generator(zlib.crc32(repr(sorted((k, v) for k, v in case.items() if k != "name")).encode()))


def _shift(g, n):
    return int(torch.randint(0, n, (1,), generator=g, device=DEVICE))


def _uniform(g, n, lo, hi, f64):
    return torch.rand(n, generator=g, device=DEVICE, dtype=torch.float64 if f64 else torch.float32) * (hi - lo) + lo


def _pos_of(counts):
    pos = torch.zeros(counts.numel() + 1, dtype=I64, device=DEVICE)
    torch.cumsum(counts, 0, out=pos[1:])
    return pos


def _distinct_rows(g, rows, width, d):
    """[rows, d] int32: d distinct uniformly drawn columns per row, ascending."""
    crd = torch.randint(0, width, (rows, d), generator=g, device=DEVICE, dtype=I32).sort(dim=1).values
    for turn in range(1000):
        bad = (crd[:, 1:] == crd[:, :-1]).any(dim=1).nonzero().flatten()
        if bad.numel() == 0:
            break
        if turn < 20 and d * d < 4 * width:
            redo = torch.randint(0, width, (bad.numel(), d), generator=g, device=DEVICE, dtype=I32)
        else:                                   # d is not small next to the width: the first d of a random order
            bad = bad[: max(1, (1 << 28) // width)]
            redo = torch.rand(bad.numel(), width, generator=g, device=DEVICE).argsort(dim=1)[:, :d].to(I32)
        crd[bad] = redo.sort(dim=1).values
    return crd


def _uniform_rows(fixed, g, rows, width, d, f64, rotate=False):
    """d entries in every row; `rotate`: the rows are rotated by a drawn number."""
    crd = _distinct_rows(fixed, rows, width, d)
    if rotate:
        crd = crd.roll(_shift(g, rows), 0)
    pos = torch.arange(rows + 1, dtype=I64, device=DEVICE) * d
    return api.DeviceCSR(rows, width, pos, crd.reshape(-1), _uniform(g, rows * d, -1.0, 1.0, f64))


def _live_rows(fixed, g, rows, width, live, d, f64, rotate=False):
    """`live` of the rows, spread evenly over them, hold d distinct uniform columns each, the others
    are empty; `rotate`: the columns are rotated by a drawn number."""
    counts = torch.zeros(rows, dtype=I64, device=DEVICE)
    counts[torch.arange(live, device=DEVICE) * rows // live] = d
    crd = _distinct_rows(fixed, live, width, d)
    if rotate:
        crd = ((crd.long() + _shift(g, width)) % width).to(I32).sort(dim=1).values
    return api.DeviceCSR(rows, width, _pos_of(counts), crd.reshape(-1), _uniform(g, live * d, -1.0, 1.0, f64))


def _powerlaw(fixed, g, n, degree, f64):
    """R-MAT with quadrant probabilities (0.57, 0.19, 0.19, 0.05), duplicates removed, cut to n x n; the
    vertices are rotated by up to a sixty-fourth of their number, so the hubs stay near the front."""
    levels = max(1, (n - 1).bit_length())
    edges = degree << levels
    rows = torch.zeros(edges, dtype=I64, device=DEVICE)
    cols = torch.zeros(edges, dtype=I64, device=DEVICE)
    for _ in range(levels):
        r = torch.rand(edges, generator=fixed, device=DEVICE)
        rows = (rows << 1) | (r >= 0.76)
        cols = (cols << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    keep = (rows < n) & (cols < n)
    by = _shift(g, max(1, n // 64))
    key = torch.unique((((rows[keep] + by) % n) << levels) | ((cols[keep] + by) % n))
    pos = _pos_of(torch.bincount(key >> levels, minlength=n))
    return api.DeviceCSR(n, n, pos, (key & ((1 << levels) - 1)).to(I32), _uniform(g, key.numel(), -1.0, 1.0, f64))


def _stencil(g, nx, ny, nz, f64):
    """27-point stencil: row x + nx (y + ny z), neighbours that lie inside the grid."""
    x = torch.arange(nx, device=DEVICE).view(1, 1, nx, 1)
    y = torch.arange(ny, device=DEVICE).view(1, ny, 1, 1)
    z = torch.arange(nz, device=DEVICE).view(nz, 1, 1, 1)
    o = torch.arange(27, device=DEVICE)
    px, py, pz = x + o % 3 - 1, y + o // 3 % 3 - 1, z + o // 9 - 1
    inside = ((px >= 0) & (px < nx) & (py >= 0) & (py < ny) & (pz >= 0) & (pz < nz)).reshape(-1, 27)
    col = (px + nx * (py + ny * pz)).reshape(-1, 27)
    crd = col[inside].to(I32)
    return api.DeviceCSR(nx * ny * nz, nx * ny * nz, _pos_of(inside.sum(dim=1)), crd, _uniform(g, crd.numel(), 0.5, 1.5, f64))


def _tensor(fixed, g, dims, nnz, f64, rotate):
    """nnz distinct uniform coordinates in CSF; mode `rotate` (never the first) is rotated by a drawn number."""
    total = dims[0] * dims[1] * dims[2]
    lin = torch.unique(torch.randint(0, total, (nnz + nnz // 4 + 64,), generator=fixed, device=DEVICE, dtype=I64))
    while lin.numel() < nnz:
        lin = torch.unique(torch.cat([lin, torch.randint(0, total, (nnz,), generator=fixed, device=DEVICE, dtype=I64)]))
    lin = lin[torch.randperm(lin.numel(), generator=fixed, device=DEVICE)[:nnz]]
    step = 1 if rotate == 2 else dims[2]
    was = lin // step % dims[rotate]
    lin = (lin + ((was + _shift(g, dims[rotate])) % dims[rotate] - was) * step).sort().values
    fibre, crd2 = lin // dims[2], (lin % dims[2]).to(I32)
    fibres, len2 = torch.unique_consecutive(fibre, return_counts=True)
    slices, len1 = torch.unique_consecutive(fibres // dims[1], return_counts=True)
    pos0 = torch.tensor([0, slices.numel()], dtype=I64, device=DEVICE)
    return api.DeviceCSF3(dims, pos0, slices.to(I32), _pos_of(len1), (fibres % dims[1]).to(I32), _pos_of(len2), crd2,
                          _uniform(g, nnz, -1.0, 1.0, f64))


_EXPR = {"spgemm": api.EXPR_SPGEMM, "ttm": api.EXPR_TTM, "outer": api.EXPR_OUTER, "spttm": api.EXPR_SPTTM,
         "spttm_i": api.EXPR_SPTTM_I, "spmttkrp": api.EXPR_SPMTTKRP}


def prepare(case, seed):
    """Operands, and the library handle and plan a program keeps (the scatters take no plan)."""
    fixed, g = _structure(case), _generator(seed)
    op, f64 = case["op"], case["f64"]
    D = None
    if op == "spgemm":
        if case["shape"] == "uniform":
            A = _uniform_rows(fixed, g, case["m"], case["k"], case["da"], f64, rotate=True)
            B = _uniform_rows(fixed, g, case["k"], case["n"], case["db"], f64)
        elif case["shape"] == "powerlaw":
            A = B = _powerlaw(fixed, g, case["n"], case["degree"], f64)
        else:
            A = B = _stencil(g, case["nx"], case["ny"], case["nz"], f64)
    elif op == "outer":
        A = _live_rows(fixed, g, case["k"], case["i"], case["live"], case["da"], f64, rotate=True)
        B = _live_rows(fixed, g, case["k"], case["n"], case["live"], case["db"], f64)
    else:
        A = _tensor(fixed, g, (case["i"], case["j"], case["k"]), case["nnz"], f64, rotate=1 if op == "ttm" else 2)
        picked = {"ttm": "k", "spttm": "i", "spttm_i": "j", "spmttkrp": "i"}[op]
        B = _uniform_rows(fixed, g, case[picked], case["n"], case["db"], f64)
        if op == "spmttkrp":
            D = _uniform_rows(fixed, g, case["j"], case["n"], case["db"], f64)
    ctx = api.Context(DEVICE)
    plan = None
    if op in ("spgemm", "ttm", "outer"):
        fmt = binding.SPWS_CSF3 if op == "ttm" else binding.SPWS_CSR
        plan = ctx.plan(_EXPR[op], (fmt, fmt, binding.SPWS_CSR), np.float64 if f64 else np.float32, case["policy"])
    return dict(op=op, policy=case["policy"], ctx=ctx, plan=plan, A=A, B=B, D=D)


def run(state):
    ctx, plan, A, B = state["ctx"], state["plan"], state["A"], state["B"]
    if state["op"] == "spgemm":
        C, _ = ctx.spgemm(A, B, plan=plan)
        return C.pos, C.crd, C.val
    if state["op"] == "outer":
        C, _ = ctx.spgemm_outer(A, B, plan=plan)
        return C.pos, C.crd, C.val
    if state["op"] == "ttm":
        C, _ = ctx.ttm(A, B, plan=plan)
        return C.pos0, C.crd0, C.pos1, C.crd1, C.pos2, C.crd2, C.val
    crd, val, _ = ctx.scatter_coo(_EXPR[state["op"]], A, B, state["D"], policy=state["policy"])
    return crd, val


# ------------------------------------------------------------------ what a pass cannot do without
def _nbytes(*tensors):
    return sum(t.numel() * t.element_size() for t in tensors)


def _rows_read(M, picks):
    """Bytes of the distinct rows of M that `picks` names: their bounds, coordinates and values."""
    rows = torch.unique(picks.long())
    entries = int((M.pos[rows + 1] - M.pos[rows]).sum())
    return 16 * rows.numel() + entries * (4 + M.val.element_size())


def work(case):
    """Bytes: the first operand once, the rows of the others that it picks once, the result once.
    Operations: a multiplication and an addition per product (one multiplication more for the
    scatter with three operands).  Counted on the operands of seed 0."""
    s = prepare(case, 0)
    A, B, D, op = s["A"], s["B"], s["D"], s["op"]
    lens = (B.pos[1:] - B.pos[:-1])
    out = run(s)
    if op in ("spgemm", "outer"):
        nbytes = _nbytes(A.pos, A.crd, A.val)
        if op == "spgemm":
            products = int(lens[A.crd.long()].sum())
            nbytes += _rows_read(B, A.crd) if B is not A else 0
        else:
            live = A.pos[1:] - A.pos[:-1]
            products = int((live * lens).sum())
            nbytes += _rows_read(B, live.nonzero().flatten())
    else:
        nbytes = _nbytes(A.pos0, A.crd0, A.pos1, A.crd1, A.pos2, A.crd2, A.val)
        fibre_of = torch.repeat_interleave(A.pos2[1:] - A.pos2[:-1])
        slice_of = torch.repeat_interleave(A.pos1[1:] - A.pos1[:-1])
        picks = A.crd2 if op == "ttm" else A.crd1[fibre_of] if op == "spttm_i" else A.crd0[slice_of[fibre_of]]
        products = int(lens[picks.long()].sum())
        nbytes += _rows_read(B, picks)
        if D is not None:
            nbytes += _rows_read(D, A.crd1)
    return {"bytes": nbytes + _nbytes(*out), "flops": (3 if op == "spmttkrp" else 2) * products}


def tolerance(case):
    """Structure is exact; values are sums of rounded products whose order may differ.  About four
    times what was measured: float against double operands, and double in another order of the sums.
    The hubs of a power-law graph add thousands of products of mixed signs into one output."""
    if case.get("shape") == "powerlaw":
        return {"rel": 8e-16, "max": 1.2e-13} if case["f64"] else {"rel": 3.2e-7, "max": 1.1e-4}
    return {"rel": 4e-16, "max": 4e-15} if case["f64"] else {"rel": 2.4e-7, "max": 1.4e-6}
