"""Vector CSR with 4 to 32 lanes per row: rows that begin and end at every
offset from an 8-entry boundary, at lengths around one and several rounds of
the lanes' groups, against the oracle; integer values bit-exact.  The
tolerances are those stated for each value type (gpu_util.TOL)."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import TOL, create, oracle_for, rel_err, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


LENS = [0, 1, 2, 3, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 47, 63, 64, 65, 127, 128, 129, 191, 193, 383, 385, 511, 513]


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_F32, B.SPMV_BF16])
@pytest.mark.parametrize("unroll,regcap", [(2, 64), (4, 64), (2, 32)])
@pytest.mark.parametrize("tpr", [4, 8, 16, 32])
def test_rows_at_every_offset(oracle, tpr, unroll, regcap, vt):
    rng = np.random.default_rng(tpr)
    lens = np.concatenate([np.insert(np.array(LENS), i, 1) for i in range(8)])  # one entry more each time round
    n = 700
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    rows = np.repeat(np.arange(lens.size), lens).astype(np.int32)
    cfg = B.make_config(format=B.FMT_CSR, threads_per_row=tpr, unroll=unroll, regcap=regcap)
    for integers in (True, False):
        vals = rng.integers(-3, 4, rows.size).astype(float) if integers else rng.standard_normal(rows.size)
        coo = matgen.Coo(int(lens.size), n, rows, cols, vals)
        x = matgen.dense_vector(n, 7, integer_values=3) if integers else matgen.dense_vector(n, 7)
        y0 = matgen.dense_vector(coo.m, 4, integer_values=3) if integers else matgen.dense_vector(coo.m, 4)
        h = create(coo, vt, cfg)
        try:
            got = run(h, vt, x, -2.0, 1.0, y0)
        finally:
            B.spmv_destroy(h)
        want = oracle_for(oracle, coo, vt, x, -2.0, 1.0, y0)
        if integers:
            assert np.array_equal(got, want)
        else:
            assert rel_err(got, want) <= TOL[vt]


@pytest.mark.parametrize("tpr", [4, 8, 16, 32])
@pytest.mark.parametrize("w", [15, 16, 20, 32, 36, 64])
def test_fp64_bands_either_side_of_the_rule(oracle, w, tpr):
    """fp64 rows of consecutive columns: by groups or from their beginning,
    whichever takes fewer slots at this width (2 w + 1 entries)."""
    coo = matgen.banded(1501, w, np.random.default_rng(w))
    x, y0 = matgen.dense_vector(coo.n, 3), matgen.dense_vector(coo.m, 4)
    for unroll in (1, 2, 4):
        h = create(coo, B.SPMV_F64, B.make_config(format=B.FMT_CSR, threads_per_row=tpr, unroll=unroll, regcap=64))
        try:
            got = run(h, B.SPMV_F64, x, -1.5, 0.5, y0)
        finally:
            B.spmv_destroy(h)
        assert rel_err(got, oracle_for(oracle, coo, B.SPMV_F64, x, -1.5, 0.5, y0)) <= TOL[B.SPMV_F64]
