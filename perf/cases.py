"""The work a user of this library has it do, as cases that can be timed: products y <- alpha A x + beta y through a kept handle,
the run-time mode from triplets to the first product, a handle built from an unordered edge list, the selector, conjugate
gradients and a batch of small products.  Matrices are the five structures of the benchmark (27-point stencil, random rows, R-MAT,
banded, block-diagonal), generated on the GPU from the seed; sizes are the benchmark's, the selector's training range (10^3 to
2.1 10^6 rows) and the batch's (10^3 to 2 10^5 rows)."""
import math

import numpy as np
import torch

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import selector as S

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}
FORMATS = {"csr": dict(format=B.FMT_CSR), "csr_split": dict(format=B.FMT_CSR, threads_per_row=B.TPR_SPLIT),
           "ell": dict(format=B.FMT_ELL), "coo": dict(format=B.FMT_COO), "hyb": dict(format=B.FMT_HYB),
           "bsr": dict(format=B.FMT_BSR), "sell": dict(format=B.FMT_SELL)}
REGULAR = ("lap2d", "stencil27", "banded", "blockdiag")  # structures that the padded formats accept at every size
MOST_NNZ = 50_000_000                                     # of a drawn matrix


# ------------------------------------------------------------------ cases
def listed():
    return [
        # The smallest call: the 5-point Laplacian on a 64 x 64 grid in a default handle, as inside somebody's inner loop.
        dict(name="run_lap2d_64_csr_f64", kind="run", family="lap2d", n=4096, par=0.0, dtype="f64", fmt="csr", residual=False),
        # PDE operators, the largest product: a 27-point stencil on 128^3 in the format that the selector picks.
        dict(name="run_stencil27_128_f64", kind="run", family="stencil27", n=2097152, par=0.0, dtype="f64", fmt="selected", residual=False),
        # Random sparse rows (uniform columns, about 16 a row) in the selected format, single precision.
        dict(name="run_poisson16_2p20_f32", kind="run", family="poisson", n=1048576, par=16.0, dtype="f32", fmt="selected", residual=False),
        # A power-law graph in a handle made without a configuration: what a caller gets who never selects.
        dict(name="run_rmat20_csr_f64", kind="run", family="rmat", n=1048576, par=0.57, dtype="f64", fmt="csr", residual=False),
        # A wide band with bf16 values (fp32 vectors) in the selected format.
        dict(name="run_banded_2p20_bf16", kind="run", family="banded", n=1048576, par=32.0, dtype="bf16", fmt="selected", residual=False),
        # The residual b - A x of an odd-sized system left in triplet form (COO), single precision.
        dict(name="run_poisson23_odd_coo_f32", kind="run", family="poisson", n=300007, par=23.0, dtype="f32", fmt="coo", residual=True),
        # The run-time mode as the README shows it: ordered triplets -> handle -> selection -> conversion -> product.
        dict(name="pipeline_stencil27_101_f64", kind="pipeline", family="stencil27", n=1030301, par=0.0, dtype="f64"),
        # A graph as it is collected: an edge list in no order with repeated edges, turned into a handle and multiplied once.
        dict(name="create_edges_rmat19_f32", kind="create", family="rmat", n=524288, par=0.57, dtype="f32"),
        # Selection alone on a kept handle: features of the matrix and the classifier.
        dict(name="select_poisson16_2p20_f64", kind="select", family="poisson", n=1048576, par=16.0, dtype="f64"),
        # A small solve, where the latency of an iteration counts: 200 iterations on the 64 x 64 Laplacian.
        dict(name="cg_lap2d_64_f64", kind="cg", family="lap2d", n=4096, par=0.0, dtype="f64", iterations=200),
        # A large solve in the selected format: 40 iterations on the 27-point Laplacian, 128^3.
        dict(name="cg_stencil27_128_f64", kind="cg", family="stencil27", n=2097152, par=0.0, dtype="f64", iterations=40),
        # Many uneven matrices in one launch, each in its selected format.
        dict(name="batch_96_f32", kind="batch", count=96, low=1000, high=200000, dtype="f32"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_matrix(rng, families, lo, hi):
    family = rng.choice(families)
    par, per_row = 0.0, 5.0
    if family == "stencil27":
        per_row = 27.0
    elif family == "poisson":
        par = per_row = round(rng.uniform(2.0, 64.0), 2)
    elif family == "rmat":
        par, per_row = round(rng.uniform(0.45, 0.65), 3), 16.0
    elif family == "banded":
        par = float(rng.randint(1, 64))
        per_row = 2 * par + 1
    elif family == "blockdiag":
        par = per_row = float(rng.choice((2, 4, 8)))
    return dict(family=family, n=int(min(_log(rng, lo, hi), MOST_NNZ / per_row)), par=par)


def draw(rng):
    kind = rng.choices(("run", "pipeline", "create", "select", "cg", "batch"), (60, 9, 8, 8, 9, 6))[0]
    dtype = rng.choice(("f64", "f32", "bf16"))
    if kind == "cg":
        return dict(kind=kind, **_draw_matrix(rng, ("lap2d", "stencil27"), 1e3, 1.9e6), dtype=rng.choice(("f64", "f32")),
                    iterations=rng.randint(5, 40))
    if kind == "batch":
        low = int(_log(rng, 1e3, 1e4))
        return dict(kind=kind, count=rng.randint(16, 96), low=low, high=int(_log(rng, 4 * low, 2e5)), dtype=dtype)
    c = dict(kind=kind, **_draw_matrix(rng, REGULAR + ("poisson", "rmat"), 1e3, 2.1e6), dtype=dtype)
    if kind in ("pipeline", "create", "select"):
        c["n"] = min(c["n"], 600000)
    if kind == "run":
        formats = ("csr", "csr_split", "coo", "hyb", "sell") + (("ell", "bsr") if c["family"] in REGULAR else ())
        c["fmt"] = "selected" if rng.random() < 0.5 else rng.choice(formats)
        c["residual"] = rng.random() < 0.3
    return c


# --------------------------------------------------------------- matrices
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _side(case):
    """Grid side of a Laplacian, scale of an R-MAT matrix."""
    if case["family"] == "lap2d":
        return max(2, round(math.sqrt(case["n"])))
    if case["family"] == "stencil27":
        return max(2, round(case["n"] ** (1.0 / 3.0)))
    return max(3, round(math.log2(case["n"])))


def _offsets(n, offsets, keep):
    """Rows and columns of the entries (i, i + offset), where keep(i, k) says that offset k exists in row i."""
    i = torch.arange(n, device="cuda", dtype=torch.int32)
    off = torch.tensor(offsets, device="cuda", dtype=torch.int32)
    valid = torch.stack([keep(i, k) for k in range(len(offsets))], 1)
    cols = (i[:, None] + off[None, :])[valid]
    return torch.repeat_interleave(i, valid.sum(1)), cols


def _edges(case, g):
    """R-MAT edges in the order they are drawn, repeats among them."""
    scale, a = _side(case), case["par"]
    b = 0.19 if a == 0.57 else (1.0 - a) / 2.0 * 0.95
    count = 16 << scale
    r = torch.zeros(count, device="cuda", dtype=torch.int32)
    c = torch.zeros_like(r)
    for _ in range(scale):
        u = torch.rand(count, device="cuda", generator=g)
        r = 2 * r + (u >= a + b)
        c = 2 * c + (((u >= a) & (u < a + b)) | (u >= a + 2 * b))
    return r, c


def _matrix(case, seed):
    """(m, rows, cols, vals, generator): square, ordered by (row, column), no repeats; values N(0, 1) in the case's type."""
    g = _generator(seed)
    family, n = case["family"], case["n"]
    if family == "lap2d":
        s = _side(case)
        n = s * s
        rows, cols = _offsets(n, (-s, -1, 0, 1, s), lambda i, k: (i >= s, i % s > 0, i >= 0, i % s < s - 1, i < n - s)[k])
    elif family == "stencil27":
        s = _side(case)
        n = s * s * s
        d = [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]

        def keep(i, k):
            z, y, x = d[k]
            at = (i // (s * s) + z, i // s % s + y, i % s + x)
            return (at[0] >= 0) & (at[0] < s) & (at[1] >= 0) & (at[1] < s) & (at[2] >= 0) & (at[2] < s)
        rows, cols = _offsets(n, [z * s * s + y * s + x for z, y, x in d], keep)
    elif family == "banded":
        w = int(case["par"])
        rows, cols = _offsets(n, range(-w, w + 1), lambda i, k: (i + (k - w) >= 0) & (i + (k - w) < n))
    elif family == "blockdiag":
        r = int(case["par"])
        n = max(r, n // r * r)
        rows = torch.arange(n, device="cuda", dtype=torch.int32).repeat_interleave(r)
        cols = (rows // r) * r + torch.arange(r, device="cuda", dtype=torch.int32).repeat(n)
    else:
        if family == "poisson":
            lens = torch.poisson(torch.full((n,), case["par"], device="cuda"), generator=g).to(torch.int64)
            rows = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
            cols = torch.randint(n, rows.shape, device="cuda", generator=g)
        else:
            rows, cols = _edges(case, g)
            n = 1 << _side(case)
        key = torch.unique(rows.to(torch.int64) * n + cols)
        rows, cols = (key // n).to(torch.int32), (key % n).to(torch.int32)
    vals = torch.randn(rows.shape, device="cuda", dtype=torch.float64, generator=g).to(DTYPES[case["dtype"]])
    return n, rows.contiguous(), cols.contiguous(), vals, g


def _laplace(case):
    """The constant-coefficient operator of the grid: centre (number of neighbours), others -1."""
    n, rows, cols, vals, _ = _matrix(case, 0)
    centre = 4.0 if case["family"] == "lap2d" else 26.0
    return n, rows, cols, torch.where(rows == cols, centre, -1.0).to(vals.dtype)


def _vector(n, dtype, g):
    v = 2.0 * torch.rand(n, device="cuda", dtype=torch.float64, generator=g) - 1.0
    return v if dtype == "f64" else v.float()


def _edge_list(case, seed):
    g = _generator(seed)
    if case["family"] == "rmat":
        rows, cols = _edges(case, g)
        n = 1 << _side(case)
    else:  # the other structures in no order, a sixteenth of the entries given twice
        n, rows, cols, _, g = _matrix(case, seed)
        at = torch.cat([torch.arange(rows.numel(), device="cuda"), torch.arange(0, rows.numel(), 16, device="cuda")])
        at = at[torch.randperm(at.numel(), device="cuda", generator=g)]
        rows, cols = rows[at], cols[at]
    vals = torch.randn(rows.shape, device="cuda", dtype=torch.float64, generator=g).to(DTYPES[case["dtype"]])
    return n, rows, cols, vals, g


def _structure(case, seed):
    """A matrix to be looked at: the regular structures with a thirty-second of their entries absent."""
    n, rows, cols, vals, g = _matrix(case, seed)
    if case["family"] in REGULAR:
        kept = torch.rand(rows.shape, device="cuda", generator=g) < 31 / 32
        rows, cols, vals = rows[kept], cols[kept], vals[kept]
    return n, rows, cols, vals, g


def _members(case, seed):
    """The matrices of a batch (sizes spread over their logarithm, structures in turn) and the seed of each one's values."""
    rng = np.random.default_rng((case["count"], case["low"], case["high"]))
    for i in range(case["count"]):
        family = ("stencil27", "poisson", "rmat", "banded", "blockdiag")[i % 5]
        par = {"stencil27": 0.0, "poisson": round(float(rng.uniform(2, 64)), 2), "rmat": round(float(rng.uniform(0.45, 0.65)), 3),
               "banded": float(rng.integers(1, 65)), "blockdiag": float(rng.choice([2, 4, 8]))}[family]
        n = int(math.exp(rng.uniform(math.log(case["low"]), math.log(case["high"]))))
        yield dict(family=family, n=n, par=par, dtype=case["dtype"]), seed * 1000 + i


_INPUT = {"create": _edge_list, "select": _structure}


# ------------------------------------------------------------ prepare, run
_selector = []


def _load_selector():
    if not _selector:
        _selector.append(S.load_default_selector())


class _State:
    """What a user's program keeps; handles and plans go with it."""

    def __init__(self, **kw):
        self.handles, self.batch = [], None
        self.__dict__.update(kw)

    def __del__(self):
        if self.batch:
            B.spmv_batch_destroy(self.batch)
        for h in self.handles:
            B.spmv_destroy(h)


def _handle(n, rows, cols, vals, fmt):
    if fmt != "selected":
        return B.spmv_create(n, n, rows, cols, vals, None if fmt == "csr" else B.make_config(**FORMATS[fmt]))
    h = B.spmv_create(n, n, rows, cols, vals)
    cfg, _ = B.spmv_select(h)
    B.spmv_set_config(h, cfg)
    return h


def prepare(case, seed):
    _load_selector()
    kind, dtype = case["kind"], case["dtype"]
    if kind == "batch":
        hs, xs, ns = [], [], []
        for c, s in _members(case, seed):
            n, rows, cols, vals, g = _matrix(c, s)
            hs.append(_handle(n, rows, cols, vals, "selected"))
            xs.append(_vector(n, dtype, g))
            ns.append(n)
        y = torch.empty(sum(ns), device="cuda", dtype=xs[0].dtype)
        b = B.spmv_batch_create(hs, [1.0] * len(hs), xs, [0.0] * len(hs), list(torch.split(y, ns)))
        return _State(kind=kind, handles=hs, batch=b, xs=xs, y=y)
    if kind == "cg":
        n, rows, cols, vals = _laplace(case)
        b = _vector(n, dtype, _generator(seed))
        return _State(kind=kind, handles=[_handle(n, rows, cols, vals, "selected")], b=b, x=torch.zeros_like(b),
                      rho=torch.zeros(case["iterations"] + 1, device="cuda", dtype=torch.float64), iterations=case["iterations"])
    n, rows, cols, vals, g = _INPUT.get(kind, _matrix)(case, seed)
    x = _vector(n, dtype, g)
    if kind in ("pipeline", "create"):
        return _State(kind=kind, n=n, rows=rows, cols=cols, vals=vals, x=x, y=torch.empty_like(x))
    if kind == "select":
        return _State(kind=kind, handles=[B.spmv_create(n, n, rows, cols, vals)])
    b = _vector(n, dtype, g) if case["residual"] else None
    return _State(kind=kind, handles=[_handle(n, rows, cols, vals, case["fmt"])], x=x, b=b, y=torch.empty_like(x))


def run(state):
    if state.kind == "run":
        if state.b is None:
            B.spmv_run(state.handles[0], 1.0, state.x, 0.0, state.y)
        else:
            state.y.copy_(state.b)
            B.spmv_run(state.handles[0], -1.0, state.x, 1.0, state.y)
        return state.y
    if state.kind == "batch":
        B.spmv_batch_launch(state.batch)
        return state.y
    if state.kind == "cg":
        state.x.zero_()
        r = B.spmv_cg(state.handles[0], state.b, state.x, 0.0, state.iterations, state.rho)
        return {"x": state.x, "rho": state.rho, "iterations": r.iterations}
    if state.kind == "select":
        cfg, features = B.spmv_select(state.handles[0])
        return {"config": [int(v) for v in cfg.as_dict().values()], "features": features}
    h = B.spmv_create(state.n, state.n, state.rows, state.cols, state.vals)
    out = {}
    if state.kind == "pipeline":
        cfg, _ = B.spmv_select(h)
        B.spmv_set_config(h, cfg)
        out["format"] = int(cfg.format)
    B.spmv_run(h, 1.0, state.x, 0.0, state.y)
    out["nnz"] = int(B.spmv_get_info(h).nnz)
    B.spmv_destroy(h)
    return {"y": state.y, **out}


# -------------------------------------------------------------- work, exact
def _sizes(case):
    """(rows, stored entries), the entries as expected where they are random."""
    family, n, par = case["family"], case["n"], case["par"]
    if family == "lap2d":
        s = _side(case)
        return s * s, 5 * s * s - 4 * s
    if family == "stencil27":
        s = _side(case)
        return s ** 3, (3 * s - 2) ** 3
    if family == "banded":
        w = int(min(par, n - 1))
        return n, n * (2 * w + 1) - w * (w + 1)
    if family == "blockdiag":
        r = int(par)
        n = max(r, n // r * r)
        return n, n * r
    return (n, int(n * par)) if family == "poisson" else (1 << _side(case), 16 << _side(case))


def work(case):
    vb = VALUE_BYTES[case["dtype"]]
    xb = 8 if case["dtype"] == "f64" else 4
    kind = case["kind"]
    members = [c for c, _ in _members(case, 0)] if kind == "batch" else [case]
    total = {"bytes": 0, "flops": 0}
    for c in members:
        m, nnz = _sizes(c)
        matrix = nnz * (vb + 4) + 4 * (m + 1)
        if kind in ("run", "batch"):  # matrix and x read, y written, the right-hand side read
            total["bytes"] += matrix + (3 if c.get("residual") else 2) * xb * m
            total["flops"] += 2 * nnz
        elif kind in ("pipeline", "create"):  # triplets and x read, y written
            total["bytes"] += nnz * (vb + 8) + 2 * xb * m
            total["flops"] += 2 * nnz
        elif kind == "select":  # the structure read
            total["bytes"] += 4 * nnz + 4 * (m + 1)
        else:  # an iteration reads the matrix and reads and writes x, r and p
            total["bytes"] += c["iterations"] * (matrix + 6 * xb * m)
            total["flops"] += c["iterations"] * (2 * nnz + 10 * m)
    return total


def _product(n, rows, cols, vals, x):
    y = torch.zeros(n, device="cuda", dtype=torch.float64)
    step = 1 << 24
    for k in range(0, rows.numel(), step):
        y.index_add_(0, rows[k:k + step], vals[k:k + step].double() * x.double()[cols[k:k + step]])
    return y


def _features(n, rows, cols):
    """The 20 sparsity features by their definitions, from the triplets of a square matrix."""
    r, c, nnz = rows.to(torch.int64), cols.to(torch.int64), rows.numel()
    lens = torch.sort(torch.bincount(r, minlength=n)).values
    count = torch.bincount(lens)
    mean, longest = nnz / n, int(lens[-1])
    var = float(((lens.double() - mean) ** 2).mean())
    place = torch.arange(1, n + 1, device="cuda", dtype=torch.int64)
    gini = float((lens * (2 * place - n - 1)).sum()) / (n * nnz)
    far = (r - c).abs()
    at_least = n - torch.cumsum(count, 0) + count
    k = torch.arange(longest + 1, device="cuda")
    wide = k[(k >= 1) & (at_least >= 4096) & (3 * at_least >= n)]
    width = int(wide.max()) if wide.numel() else 0

    def fill(b):
        return nnz / (b * b * torch.unique((r // b) * (n // b + 1) + c // b).numel())
    return [n, nnz, nnz / n / n, mean, var, math.sqrt(var), int(lens[0]), longest, int(lens[(n - 1) // 2]), int(torch.argmax(count)),
            nnz / (n * longest), gini, math.sqrt(var) / mean, float((lens == 0).sum()) / n, int(far.max()), float(far.sum()) / nnz,
            float((far == 0).sum()) / nnz, fill(4), fill(2), float((lens - width).clamp(min=0).sum()) / nnz]


def _grid_operator(case):
    """The Laplacian of _laplace() on a flat vector, by shifts of the grid."""
    s = _side(case)

    def lap2d(v):
        p = torch.nn.functional.pad(v.view(s, s), (1, 1, 1, 1))
        return (4.0 * p[1:-1, 1:-1] - p[:-2, 1:-1] - p[2:, 1:-1] - p[1:-1, :-2] - p[1:-1, 2:]).reshape(-1)

    def stencil27(v):
        p = torch.nn.functional.pad(v.view(s, s, s), (1,) * 6)
        p = p[:-2] + p[1:-1] + p[2:]
        p = p[:, :-2] + p[:, 1:-1] + p[:, 2:]
        p = p[:, :, :-2] + p[:, :, 1:-1] + p[:, :, 2:]
        return 27.0 * v - p.reshape(-1)
    return lap2d if case["family"] == "lap2d" else stencil27


def exact(case, seed):
    kind, dtype = case["kind"], case["dtype"]
    if kind == "batch":
        ys = []
        for c, s in _members(case, seed):
            n, rows, cols, vals, g = _matrix(c, s)
            ys.append(_product(n, rows, cols, vals, _vector(n, dtype, g)))
        return torch.cat(ys)
    if kind == "cg":
        apply = _grid_operator(case)
        side = _side(case)
        n = side * side if case["family"] == "lap2d" else side ** 3
        r = _vector(n, dtype, _generator(seed)).double()
        x, p = torch.zeros_like(r), r.clone()
        rho = [r @ r]
        for _ in range(case["iterations"]):
            q = apply(p)
            alpha = rho[-1] / (p @ q)
            x = x + alpha * p
            r = r - alpha * q
            rho.append(r @ r)
            p = r + (rho[-1] / rho[-2]) * p
        return {"x": x, "rho": torch.stack(rho), "iterations": None}
    n, rows, cols, vals, g = _INPUT.get(kind, _matrix)(case, seed)
    if kind == "select":
        return {"config": None, "features": np.array(_features(n, rows, cols), dtype=np.float64)}
    y = _product(n, rows, cols, vals, _vector(n, dtype, g))
    if kind == "run":
        return _vector(n, dtype, g).double() - y if case["residual"] else y
    return {"y": y, "nnz": None, "format": None}
