"""ELL and HYB handles held by diagonals of row slices (2^20 entries and more,
with fp64 values 160 MB of columns and values, rows that share their column offsets), against the oracle (gpu_util.TOL) and
bit for bit against CSR with one lane per row, which adds a row's entries in
the same order; matrices just outside the rule keep the column layout."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import TOL, create, oracle_for, rel_err, run

pytestmark = pytest.mark.gpu
VS = {B.SPMV_F64: 8, B.SPMV_F32: 4, B.SPMV_BF16: 2}
VTS = list(VS)


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _band(m, n, w, keep=1.0, seed=0):
    """Band of half-width w in an m x n matrix, a fraction of its entries kept."""
    rng = np.random.default_rng(seed)
    i = np.arange(m)[:, None]
    j = i + np.arange(-w, w + 1)[None, :]
    ok = (j >= 0) & (j < n) & (rng.random(j.shape) < keep)
    rows = np.broadcast_to(i, j.shape)[ok]
    return matgen.Coo(m, n, rows, j[ok], rng.standard_normal(rows.size))


# f: times the rows (fp64 needs more of them)
MATS = {
    "stencil": lambda f: matgen.stencil_3d(36 if f == 1 else 85, 27, np.random.default_rng(1)),  # 46,656 or 614,125 rows
    "band": lambda f: _band(33333 * f, 33333 * f, 16),
    "tall": lambda f: _band(40001 * f, 30000 * f, 20),                   # the last rows are empty
    "wide": lambda f: _band(34001 * f, 50000 * f, 17),
    "holes": lambda f: _band(33333 * f, 33333 * f, 16, keep=0.98, seed=2),
    "wide_band": lambda f: _band(8200 * f, 8200 * f, 70),                # 141 diagonals, over 4 rounds of 32
}
SCALE = {B.SPMV_F64: 13, B.SPMV_F32: 1, B.SPMV_BF16: 1}


def _is_dia(h, vt):
    info = B.spmv_get_info(h)
    return info.format_bytes < info.nnz * (VS[vt] + 1.5)


@pytest.mark.parametrize("vt", VTS)
@pytest.mark.parametrize("name", list(MATS))
def test_diagonals(oracle, name, vt):
    coo = MATS[name](SCALE[vt])
    assert coo.nnz >= 1 << 20
    x = matgen.dense_vector(coo.n, 3)
    y0 = matgen.dense_vector(coo.m, 4)
    h = create(coo, vt, B.make_config(format=B.FMT_CSR, threads_per_row=1))
    try:
        for beta in (0.0, 0.5):
            B.spmv_set_config(h, B.make_config(format=B.FMT_CSR, threads_per_row=1))
            want = run(h, vt, x, 1.25, beta, y0, m=coo.m)
            assert rel_err(want, oracle_for(oracle, coo, vt, x, 1.25, beta, y0)) <= TOL[vt]
            for kw in (dict(), dict(unroll=1, regcap=32), dict(unroll=2, threads_per_block=32), dict(unroll=8, regcap=48)):
                B.spmv_set_config(h, B.make_config(format=B.FMT_ELL, **kw))
                got = run(h, vt, x, 1.25, beta, y0, m=coo.m)
                assert np.array_equal(got, want), (name, kw)
        if name in ("stencil", "band", "wide_band"):
            assert _is_dia(h, vt)
    finally:
        B.spmv_destroy(h)


@pytest.mark.parametrize("vt", VTS)
def test_hyb_part_and_exports(oracle, vt):
    import torch
    coo = _band(33333 * SCALE[vt], 33333 * SCALE[vt], 16)
    x = matgen.dense_vector(coo.n, 5)
    for width in (1, 20, 33):
        h = create(coo, vt, B.make_config(format=B.FMT_HYB, hyb_ell_width=width))
        try:
            got = run(h, vt, x, m=coo.m)
            info = B.spmv_get_info(h)
            pitch = B.spmv_export_bytes(h, B.ARR_ELL_PITCH)
            col = torch.empty(width * pitch, dtype=torch.int32, device="cuda")
            B.spmv_export(h, B.ARR_ELL_COLIDX, col)
            assert B.spmv_export_bytes(h, B.ARR_ELL_VALS) == VS[vt] * width * pitch
        finally:
            B.spmv_destroy(h)
        assert info.ell_width == width and info.hyb_coo_nnz == coo.nnz - np.minimum(np.bincount(coo.rows), width).sum()
        assert rel_err(got, oracle_for(oracle, coo, vt, x)) <= TOL[vt]
        col = col.cpu().numpy().reshape(width, pitch)[:, :coo.m]
        start = np.searchsorted(coo.rows, np.arange(coo.m))
        assert np.array_equal(col[0], coo.cols[start])
        assert np.array_equal(col[-1][50:-50], coo.cols[(start + width - 1)[50:-50]])


def test_rows_without_an_entry_never_see_its_x():
    """x is infinite in one column: only the rows that hold an entry there may show it."""
    coo = _band(33333, 33333, 16, keep=0.98, seed=7)
    for vt in (B.SPMV_F32, B.SPMV_BF16):
        x = matgen.dense_vector(coo.n, 6)
        x[20000] = np.inf
        h = create(coo, vt, B.make_config(format=B.FMT_ELL))
        try:
            assert _is_dia(h, vt)
            got = run(h, vt, x, m=coo.m)
        finally:
            B.spmv_destroy(h)
        touched = np.zeros(coo.m, bool)
        touched[coo.rows[coo.cols == 20000]] = True
        assert np.array_equal(~np.isfinite(got), touched)


@pytest.mark.parametrize("vt", VTS)
def test_outside_the_rule(oracle, vt):
    """Scattered columns and small matrices keep the column layout."""
    small = _band(33333, 33333, 16) if vt == B.SPMV_F64 else _band(3000, 3000, 16)
    for coo in (matgen.poisson_rows(70000, 16.0, np.random.default_rng(3)), small):
        x = matgen.dense_vector(coo.n, 8)
        h = create(coo, vt, B.make_config(format=B.FMT_ELL))
        try:
            info = B.spmv_get_info(h)
            pitch = B.spmv_export_bytes(h, B.ARR_ELL_PITCH)
            assert info.format_bytes >= info.ell_width * pitch * (VS[vt] + 2)
            assert rel_err(run(h, vt, x, m=coo.m), oracle_for(oracle, coo, vt, x)) <= TOL[vt]
        finally:
            B.spmv_destroy(h)


def test_batch_of_diagonals(oracle):
    import torch
    for vt in VTS:
        mats = [MATS["stencil"](SCALE[vt]), MATS["band"](SCALE[vt]), _band(500, 500, 3)]
        hs = [create(c, vt, B.make_config(format=B.FMT_ELL)) for c in mats]
        vec = torch.float64 if vt == B.SPMV_F64 else torch.float32
        x = [matgen.dense_vector(c.n, 9) for c in mats]
        xs = [torch.from_numpy(v).to(vec).cuda() for v in x]
        ys = [torch.zeros(c.m, dtype=vec, device="cuda") for c in mats]
        try:
            B.spmv_batch_run(hs, [1.0] * 3, xs, [0.0] * 3, ys)
        finally:
            for h in hs:
                B.spmv_destroy(h)
        for c, v, y in zip(mats, x, ys):
            assert rel_err(y.cpu().double().numpy(), oracle_for(oracle, c, vt, v)) <= TOL[vt]
