"""spmv_trim: after it, device memory that handles of the library have freed is
free for others again."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import create, oracle_for, rel_err, run, TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_goes_back(oracle):
    coo = matgen.poisson_rows(300000, 4.0, np.random.default_rng(1))    # arrays of 1.2 to 15 MB
    shuffled = np.random.default_rng(2).permutation(coo.nnz)
    x = matgen.dense_vector(coo.n, 3)

    def use():
        for fmt in (B.FMT_CSR, B.FMT_COO, B.FMT_SELL, B.FMT_HYB):
            h = create(coo, B.SPMV_F64, B.make_config(format=fmt), coo.rows[shuffled], coo.cols[shuffled], coo.vals[shuffled])
            try:
                got = run(h, B.SPMV_F64, x, m=coo.m)
            finally:
                B.spmv_destroy(h)
            assert rel_err(got, oracle_for(oracle, coo, B.SPMV_F64, x)) <= TOL[B.SPMV_F64]

    use()                       # kernels loaded, torch's own cache filled
    B.spmv_trim()
    free0 = _free()
    use()
    kept = free0 - _free()
    assert kept > 8 << 20       # temporaries and small arrays stay mapped ...
    B.spmv_trim()
    assert _free() >= free0     # ... until they are given back
    use()
