"""Work units of a batch: CSR rows in steps of 32 / lanes rows at every number
of lanes, BSR block rows with one to eight blocks at once, x on and off a
16-byte boundary, ragged row counts and columns past the last whole block,
against the oracle, replayed (the item counter is reset by the launch
itself).  The tolerances are those stated for each value type
(gpu_util.TOL); integer values are bit-exact."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import TOL, create, oracle_for, rel_err, run, vec_dtype

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _rows(m, n, k, seed):
    rng = np.random.default_rng(seed)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for _ in range(m)]).astype(np.int32)
    return matgen.Coo(m, n, np.repeat(np.arange(m), k).astype(np.int32), cols, rng.integers(-3, 4, m * k).astype(float))


def _blocks(m, n, width, seed):
    """block rows of 1 .. 2 width - 1 consecutive 2 x 2 blocks, the last ones cut by m and n"""
    rng = np.random.default_rng(seed)
    rows, cols = [], []
    for b in range((m + 3) // 4):
        w = 4 * int(rng.integers(1, 2 * width))
        c0 = 4 * int(rng.integers(0, max(1, (n - w) // 4 + 2)))
        for i in range(4 * b, min(m, 4 * b + 4)):
            c = np.arange(c0, min(n, c0 + w))
            rows.append(np.full(c.size, i))
            cols.append(c)
    rows, cols = np.concatenate(rows).astype(np.int32), np.concatenate(cols).astype(np.int32)
    return matgen.Coo(m, n, rows, cols, rng.integers(-3, 4, rows.size).astype(float))


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_F32, B.SPMV_BF16])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_units_of_a_batch(oracle, shift, vt):
    import torch
    dt = vec_dtype(vt)
    mats, cfgs = [], []
    for i, k in enumerate((3, 20, 40, 80, 150, 300)):  # 1, 2, 4, 8, 16 and 32 lanes a row
        for m in (1, 31, 33, 261):
            mats.append(_rows(m, 600 + i, k, 10 * i + m))
            cfgs.append(B.make_config(format=B.FMT_CSR))
    for r in (2, 4):
        for width in (1, 8, 20, 40):
            for m, n in ((5, 403), (261, 2001), (64, 1024)):
                mats.append(_blocks(m, n, width, 7 * width + m + r))
                cfgs.append(B.make_config(format=B.FMT_BSR, bsr_block=r))
    hs, xs, ys, xh = [], [], [], []
    for i, (coo, cfg) in enumerate(zip(mats, cfgs)):
        hs.append(create(coo, vt, cfg))
        x = matgen.dense_vector(coo.n, 20 + i, integer_values=3)
        xh.append(x)
        xs.append(torch.zeros(coo.n + shift, dtype=dt, device="cuda")[shift:].copy_(torch.from_numpy(x).to(dt)))
        ys.append(torch.empty(coo.m, dtype=dt, device="cuda"))
    b = B.spmv_batch_create(hs, np.ones(len(mats)), xs, np.zeros(len(mats)), ys)
    try:
        modes = B.spmv_batch_get_plan(b, len(mats))[0].tolist()
        assert {-B.FMT_BSR, 1, 2, 4, 8, 16, 32} <= set(modes), modes
        for rep in range(3):
            for y in ys:
                y.fill_(float("nan"))
            B.spmv_batch_launch(b)
            torch.cuda.synchronize()
            for i, coo in enumerate(mats):
                assert np.array_equal(ys[i].cpu().double().numpy(), oracle_for(oracle, coo, vt, xh[i])), (rep, i, modes[i])
    finally:
        B.spmv_batch_destroy(b)
        for h in hs:
            B.spmv_destroy(h)


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_F32, B.SPMV_BF16])
@pytest.mark.parametrize("r", [2, 4])
@pytest.mark.parametrize("shift", [0, 1])
def test_bsr_reads_x_by_blocks(oracle, shift, r, vt):
    import torch
    dt = vec_dtype(vt)
    coo = _blocks(261, 2001, 20, r)
    coo = matgen.Coo(coo.m, coo.n, coo.rows, coo.cols, np.random.default_rng(r).standard_normal(coo.rows.size))
    x, y0 = matgen.dense_vector(coo.n, 3), matgen.dense_vector(coo.m, 4)
    h = create(coo, vt, B.make_config(format=B.FMT_BSR, bsr_block=r))
    try:
        xd = torch.zeros(coo.n + shift, dtype=dt, device="cuda")[shift:].copy_(torch.from_numpy(x).to(dt))
        y = torch.from_numpy(y0).to(dt).cuda()
        B.spmv_run(h, -1.5, xd, 0.5, y)
        torch.cuda.synchronize()
    finally:
        B.spmv_destroy(h)
    assert rel_err(y.cpu().double().numpy(), oracle_for(oracle, coo, vt, x, -1.5, 0.5, y0)) <= TOL[vt]
