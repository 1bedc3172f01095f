"""ELL and HYB of regular matrices with a few irregular rows: a slice of row
slices' diagonals (32, 64 or 128 rows for fp64, fp32, bf16 values) is counted up
to 4 width + 16 distinct column offsets.  One offset more keeps the column layout, and the products
agree with the oracle (gpu_util.TOL) and bit for bit with CSR with one lane per
row on both sides of the line."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import TOL, create, oracle_for, rel_err, run

pytestmark = pytest.mark.gpu
VS = {B.SPMV_F64: 8, B.SPMV_F32: 4, B.SPMV_BF16: 2}
ROWS = {B.SPMV_F64: 32, B.SPMV_F32: 64, B.SPMV_BF16: 128}     # of a slice
# slices of a band of half-width 16: fp64 values take the diagonals from 160 MB on
SLICES = {B.SPMV_F64: 13 * 1042, B.SPMV_F32: 521, B.SPMV_BF16: 261}
W = 16
WIDTH = 2 * W + 1
MOST = 4 * WIDTH + 16


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _band_with(vt, slices, extra):
    """A band whose rows in `slices` are replaced: WIDTH entries each, `extra`
    distinct column offsets a slice in all."""
    rows, per = ROWS[vt], SLICES[vt]
    n = rows * per
    cols = np.arange(n, dtype=np.int64)[:, None] + np.arange(-W, W + 1)[None, :]
    for sl in slices:
        r = np.arange(sl * rows, (sl + 1) * rows)
        # row i of the slice takes offsets first[i] .. first[i] + WIDTH - 1 from a run of `extra`
        # offsets on either side of the diagonal that leaves every column inside the matrix
        first = np.minimum(WIDTH * np.arange(rows), extra - WIDTH)
        lowest = -(sl * rows) if sl * rows + extra + rows < n else -(sl * rows) + n - extra - rows
        cols[r] = r[:, None] + lowest + first[:, None] + np.arange(WIDTH)[None, :]
    ok = (cols >= 0) & (cols < n)
    r = np.broadcast_to(np.arange(n)[:, None], cols.shape)[ok]
    return matgen.Coo(n, n, r.astype(np.int32), cols[ok].astype(np.int32),
                      np.random.default_rng(len(slices)).standard_normal(r.size))


def _offsets(coo, vt):
    """distinct column offsets of every slice"""
    key = np.unique((coo.rows.astype(np.int64) // ROWS[vt]) * (1 << 33) + (coo.cols.astype(np.int64) - coo.rows) + (1 << 32))
    return np.bincount(key >> 33, minlength=SLICES[vt])


def _layout_is_diagonals(h, vt):
    info = B.spmv_get_info(h)
    return info.format_bytes - info.hyb_coo_nnz * (VS[vt] + 8) < (info.nnz - info.hyb_coo_nnz) * (VS[vt] + 1.5)


@pytest.mark.parametrize("fmt", ["ell", "hyb"])
@pytest.mark.parametrize("over", [0, 1, 500])
@pytest.mark.parametrize("vt", list(VS))
def test_irregular_slices(oracle, vt, over, fmt):
    last = SLICES[vt] - 1
    slices = [0, 7, 100, last - 1, last]
    extra = min(MOST + over, WIDTH * ROWS[vt])
    coo = _band_with(vt, slices, extra)
    assert coo.nnz >= 1 << 20 and (vt != B.SPMV_F64 or WIDTH * coo.m * 12 >= 160e6)
    counts = _offsets(coo, vt)
    assert all(counts[s] == extra for s in slices) and np.delete(counts, slices).max() == WIDTH
    x = matgen.dense_vector(coo.n, 3)
    h = create(coo, vt, B.make_config(format=B.FMT_CSR, threads_per_row=1))
    try:
        want = run(h, vt, x, m=coo.m)
        B.spmv_set_config(h, B.make_config(format=B.FMT_ELL) if fmt == "ell" else
                          B.make_config(format=B.FMT_HYB, hyb_ell_width=WIDTH))
        assert _layout_is_diagonals(h, vt) == (over == 0)
        got = run(h, vt, x, m=coo.m)
    finally:
        B.spmv_destroy(h)
    assert np.array_equal(got, want)
    assert rel_err(got, oracle_for(oracle, coo, vt, x)) <= TOL[vt]
