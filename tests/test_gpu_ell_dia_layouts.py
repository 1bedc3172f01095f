"""Which ELL and HYB handles are held by diagonals: each matrix of
test_gpu_ell_dia.py whose masked slots, empty rows or m != n the diagonal kernel
is to be tested with, the HYB widths, and a batch's handles; the products of the
HYB ones against the oracle (gpu_util.TOL)."""
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import TOL, create, oracle_for, rel_err, run
from test_gpu_ell_dia import MATS, SCALE, VS, VTS, _band, _is_dia

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


@pytest.mark.parametrize("vt", VTS)
@pytest.mark.parametrize("name", list(MATS))
def test_every_matrix_is_held_by_diagonals(name, vt):
    h = create(MATS[name](SCALE[vt]), vt, B.make_config(format=B.FMT_ELL))
    try:
        assert _is_dia(h, vt)
    finally:
        B.spmv_destroy(h)


def _hyb_is_dia(h, vt):
    """the ELL part takes less than a value and two bytes a slot"""
    info = B.spmv_get_info(h)
    pitch = B.spmv_export_bytes(h, B.ARR_ELL_PITCH)
    return info.format_bytes - info.hyb_coo_nnz * (VS[vt] + 8) < info.ell_width * pitch * (VS[vt] + 1.5)


# fp64: 160 MB of columns and values take 700,000 rows at width 20
@pytest.mark.parametrize("vt,n,width,dia", [
    (B.SPMV_F64, 33333 * 13, 1, False), (B.SPMV_F64, 33333 * 13, 20, False), (B.SPMV_F64, 33333 * 13, 33, True),
    (B.SPMV_F64, 700001, 20, True), (B.SPMV_F32, 33333, 1, True), (B.SPMV_F32, 33333, 20, True), (B.SPMV_F32, 33333, 33, True),
    (B.SPMV_BF16, 33333, 1, True), (B.SPMV_BF16, 33333, 20, True), (B.SPMV_BF16, 33333, 33, True)])
def test_hyb_parts(oracle, vt, n, width, dia):
    coo = _band(n, n, 16)
    x = matgen.dense_vector(n, 5)
    h = create(coo, vt, B.make_config(format=B.FMT_HYB, hyb_ell_width=width))
    try:
        assert _hyb_is_dia(h, vt) == dia
        got = run(h, vt, x, m=n)
    finally:
        B.spmv_destroy(h)
    assert rel_err(got, oracle_for(oracle, coo, vt, x)) <= TOL[vt]


@pytest.mark.parametrize("vt", VTS)
def test_batch_handles(vt):
    for name in ("stencil", "band"):
        h = create(MATS[name](SCALE[vt]), vt, B.make_config(format=B.FMT_ELL))
        try:
            assert _is_dia(h, vt)
        finally:
            B.spmv_destroy(h)
    h = create(_band(500, 500, 3), vt, B.make_config(format=B.FMT_ELL))
    try:
        assert not _is_dia(h, vt)
    finally:
        B.spmv_destroy(h)
