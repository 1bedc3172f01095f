"""Conversions at the edges of their tiles: sorts of 4096 and 8192 pairs a
block (each value type has its own tile), triplets checked 256 at a time,
entries merged 2048 at a time, gaps of empty rows on either side of 32, ELL
rows staged 4608 entries a warp.  The CSR arrays of an unordered list equal a
stable sort with repeats summed in triplet order, exactly."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import create, oracle_for, rel_err, run, TOL

pytestmark = pytest.mark.gpu
NP = {B.SPMV_F64: np.float64, B.SPMV_F32: np.float32}


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _csr(h):
    import torch
    out = []
    vt = B.spmv_get_info(h).value_type
    for a, dt in ((B.ARR_CSR_ROWPTR, torch.int32), (B.ARR_CSR_COLIDX, torch.int32),
                  (B.ARR_CSR_VALS, {0: torch.float64, 1: torch.float32, 2: torch.bfloat16}[vt])):
        t = torch.empty(B.spmv_export_bytes(h, a) // dt.itemsize, dtype=dt, device="cuda")
        B.spmv_export(h, a, t)
        out.append(t.cpu().double().numpy())
    return out


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_F32, B.SPMV_BF16])
@pytest.mark.parametrize("nnz", [1, 31, 255, 256, 257, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8192, 8193, 20000])
@pytest.mark.parametrize("m,n", [(1, 1), (300, 7), (5000, 70000)])
def test_unordered_triplets(m, n, nnz, vt):
    rng = np.random.default_rng(nnz)
    rows, cols = rng.integers(0, m, nnz), rng.integers(0, n, nnz)
    vals = rng.integers(-4, 5, nnz).astype(float)      # sums of few small integers: exact in every type
    if m * n < nnz // 50:                              # many repeats of one place: sums stay exact in bf16 too
        vals[:] = 0.0
        vals[::max(1, nnz // 50)] = 1.0
    coo = matgen.Coo(m, n, rows, cols, vals)
    h = create(coo, vt)
    try:
        rp, ci, va = _csr(h)
    finally:
        B.spmv_destroy(h)
    key, at = np.unique(coo.rows.astype(np.int64) * n + coo.cols, return_inverse=True)
    want = np.zeros(key.size)
    np.add.at(want, at, vals)
    assert np.array_equal(ci, key % n)
    assert np.array_equal(rp, np.searchsorted(key // n, np.arange(m + 1)))
    assert np.array_equal(va, want)


@pytest.mark.parametrize("gap", [0, 1, 31, 32, 33, 500])
def test_ordered_triplets_with_gaps(oracle, gap):
    """Row pointers written where rows open, or searched where a gap is long."""
    step = gap + 1
    rows = np.repeat(np.arange(gap, 700 * step, step), 3).astype(np.int32)
    coo = matgen.Coo(700 * step + gap, 50, rows, np.tile([1, 7, 30], 700).astype(np.int32), np.ones(2100))
    h = create(coo, B.SPMV_F64)
    try:
        rp, ci, _ = _csr(h)
        info = B.spmv_get_info(h)
        assert info.max_row == 3
    finally:
        B.spmv_destroy(h)
    assert np.array_equal(rp, np.searchsorted(coo.rows, np.arange(coo.m + 1)))
    assert np.array_equal(ci, coo.cols)


@pytest.mark.parametrize("width", [1, 31, 143, 144, 145, 400])
@pytest.mark.parametrize("fmt", [B.FMT_ELL, B.FMT_HYB, B.FMT_SELL])
def test_packs_around_the_staging(oracle, fmt, width):
    """Full rows of `width` entries (32 rows fit in the staging up to 144) and some short ones."""
    rng = np.random.default_rng(width)
    lens = [width] * 70 + [0, 1, width // 2, 0] * 8
    cols = np.concatenate([np.sort(rng.choice(900, k, replace=False)) for k in lens]).astype(np.int32)
    coo = matgen.Coo(len(lens), 900, np.repeat(np.arange(len(lens)), lens), cols, rng.standard_normal(cols.size))
    x = matgen.dense_vector(900, 2)
    for vt in (B.SPMV_F64, B.SPMV_F32, B.SPMV_BF16):
        h = create(coo, vt, B.make_config(format=fmt, **({"hyb_ell_width": max(1, width - 3)} if fmt == B.FMT_HYB else {})))
        try:
            got = run(h, vt, x, m=coo.m)
        finally:
            B.spmv_destroy(h)
        assert rel_err(got, oracle_for(oracle, coo, vt, x)) <= TOL[vt]
