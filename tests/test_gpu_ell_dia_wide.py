"""Diagonals of wide bands: on either side of the width from which a slice's
columns and values no longer fit in a block's shared memory (fp64 values: 32
rows of 579 entries at 12 bytes, 224 KB with the padding) and its entries are read in place.
Values and x are small integers, whose sums are exact in every order and type: the products equal the oracle's."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import create, oracle_for, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _band(n, w):
    cols = np.arange(n, dtype=np.int64)[:, None] + np.arange(-w, w + 1)[None, :]
    ok = (cols >= 0) & (cols < n)
    rows = np.broadcast_to(np.arange(n)[:, None], cols.shape)[ok]
    return matgen.Coo(n, n, rows.astype(np.int32), cols[ok].astype(np.int32),
                      np.random.default_rng(w).integers(-8, 9, rows.size).astype(np.float64))


# (value type, bytes of a value, half-width, rows): fp64 of 160 MB of columns and values and more
CASES = [(B.SPMV_F64, 8, w, n) for w, n in ((289, 24000), (290, 24000), (293, 24001), (320, 22007), (400, 30000))] + \
        [(B.SPMV_F32, 4, 400, 5000), (B.SPMV_BF16, 2, 400, 5000)]


@pytest.mark.parametrize("fmt", ["ell", "hyb"])
@pytest.mark.parametrize("vt,vs,w,n", CASES)
def test_wide_bands(oracle, vt, vs, w, n, fmt):
    coo = _band(n, w)
    width = 2 * w + 1
    assert coo.nnz >= 1 << 20 and (vt != B.SPMV_F64 or 12 * width * n >= 160e6)
    x = np.random.default_rng(3).integers(-8, 9, n).astype(np.float64)
    h = create(coo, vt)
    try:
        B.spmv_set_config(h, B.make_config(format=B.FMT_ELL) if fmt == "ell" else
                          B.make_config(format=B.FMT_HYB, hyb_ell_width=width))
        info = B.spmv_get_info(h)
        got = run(h, vt, x, m=n)
    finally:
        B.spmv_destroy(h)
    assert info.format == (B.FMT_ELL if fmt == "ell" else B.FMT_HYB) and info.hyb_coo_nnz == 0
    assert info.format_bytes < info.nnz * (vs + 1.5)          # held by diagonals
    assert np.array_equal(got, oracle_for(oracle, coo, vt, x))
