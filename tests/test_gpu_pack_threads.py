"""ELL handles packed by several threads at once, with rows of different widths:
each pack asks for its own amount of shared memory, and none may take another
thread's.  Products against the oracle (gpu_util.TOL)."""
import threading

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


def _band(n, w):
    cols = np.arange(n, dtype=np.int64)[:, None] + np.arange(-w, w + 1)[None, :]
    ok = (cols >= 0) & (cols < n)
    rows = np.broadcast_to(np.arange(n)[:, None], cols.shape)[ok]
    return matgen.Coo(n, n, rows.astype(np.int32), cols[ok].astype(np.int32),
                      np.random.default_rng(w).standard_normal(rows.size))


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_BF16])
@pytest.mark.parametrize("n", [500, 12000])           # column layout, and (bf16, wide) diagonals
def test_packs_in_threads(oracle, vt, n):
    import torch
    mats = [_band(n, w) for w in (1, 8, 30, 60, 1, 8, 30, 60)]
    hs = [create(c, vt) for c in mats]
    torch.cuda.synchronize()
    failed, gate = [], threading.Barrier(len(hs))

    def work(h):
        stream = torch.cuda.Stream()
        gate.wait()
        try:
            for _ in range(150):
                for fmt in (B.FMT_ELL, B.FMT_CSR):
                    B.spmv_set_config(h, B.make_config(format=fmt), stream.cuda_stream)
            B.spmv_set_config(h, B.make_config(format=B.FMT_ELL), stream.cuda_stream)
        except B.SpmvError as e:
            failed.append(str(e))

    threads = [threading.Thread(target=work, args=(h,)) for h in hs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    try:
        assert not failed, failed[0]
        for c, h in zip(mats, hs):
            x = matgen.dense_vector(c.n, 3)
            assert rel_err(run(h, vt, x, m=c.m), oracle_for(oracle, c, vt, x)) <= TOL[vt]
    finally:
        for h in hs:
            B.spmv_destroy(h)
