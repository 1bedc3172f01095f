"""Vector CSR with one or two lanes per row on uneven rows (a lane, eight lanes
or warp segments per row) at the lengths where the path changes (24, 25, 128,
129, 1024, 1025, 2048, 2049 entries), with empty rows, the ends of the matrix
and every value type, against the oracle; integer values bit-exact.  The
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


def _rows(lens, n, seed, integers=False):
    rng = np.random.default_rng(seed)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    rows = np.repeat(np.arange(len(lens)), lens).astype(np.int32)
    vals = rng.integers(-3, 4, rows.size).astype(float) if integers else rng.standard_normal(rows.size)
    return matgen.Coo(len(lens), n, rows, cols, vals)


# 32-row groups of short rows with one long row each: the longest rows average
# far above the mean, which is what selects the path
EDGES = [0, 1, 3, 24, 25, 127, 128, 129, 1023, 1024, 1025, 2048, 2049, 3100]
LENS = {
    "edges": [k for e in EDGES for k in [e] + [2] * 31],
    "edges_last_row": [2] * 31 + [900] + [0] * 31 + [129],
    "all_medium_in_a_group": [100] * 9 + [0] * 23 + [500] + [1] * 400,
    "empty_but_one": [0] * 95 + [2500] + [0] * 40,
    "one_row": [700],
}


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_F32, B.SPMV_BF16])
@pytest.mark.parametrize("tpr,regcap,tpb", [(1, 64, 256), (2, 64, 128), (1, 32, 32)])
@pytest.mark.parametrize("name", list(LENS))
def test_uneven_rows(oracle, name, tpr, regcap, tpb, vt):
    cfg = B.make_config(format=B.FMT_CSR, threads_per_row=tpr, regcap=regcap, threads_per_block=tpb)
    n = 4000
    x = matgen.dense_vector(n, 3)
    for alpha, beta in ((1.0, 0.0), (-1.5, 0.5)):
        coo = _rows(LENS[name], n, 5)
        y0 = matgen.dense_vector(coo.m, 4)
        h = create(coo, vt, cfg)
        try:
            got = run(h, vt, x, alpha, beta, y0, m=coo.m)
            again = run(h, vt, x, alpha, beta, y0, m=coo.m)
        finally:
            B.spmv_destroy(h)
        assert np.array_equal(got, again)
        assert rel_err(got, oracle_for(oracle, coo, vt, x, alpha, beta, y0)) <= TOL[vt]
    coo = _rows(LENS[name], n, 6, integers=True)
    xi = matgen.dense_vector(n, 7, integer_values=3)
    h = create(coo, vt, cfg)
    try:
        assert np.array_equal(run(h, vt, xi, m=coo.m), oracle_for(oracle, coo, vt, xi))
    finally:
        B.spmv_destroy(h)
