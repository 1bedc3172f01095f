"""spmv_cg at the edges of its two forms (one thread-block cluster for small
systems, a graph for the others), against the oracle's CG: rows on either side
of the cluster's sizes, staged and unstaged rows, every format in the graph
form, and an x that is not 16-byte aligned.  Bars as in test_gpu_cg.py: after a
few iterations the iterate and the rho history agree to 1e-10 (fp64)."""
import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen
from paper_2302_05662_gb300.workload import SWEEP_VARIANTS

from gpu_util import create, rel_err

pytestmark = pytest.mark.gpu
VARIANTS = dict(SWEEP_VARIANTS)


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def band(n, w):
    """Band of half-width w: off-diagonal -1, diagonal 2 w + 1 (dominant)."""
    coo = matgen.banded(n, w, np.random.default_rng(0))
    coo.vals = np.where(coo.rows == coo.cols, 2.0 * w + 1.0, -1.0)
    return coo


def check(oracle, coo, cfg, k=4, shift=0):
    import torch
    b = matgen.dense_vector(coo.m, 31)
    x0 = matgen.dense_vector(coo.m, 32)
    h = create(coo, B.SPMV_F64, cfg)
    try:
        xt = torch.zeros(coo.m + shift, dtype=torch.float64, device="cuda")[shift:]
        xt.copy_(torch.from_numpy(x0))
        rho = torch.zeros(k + 1, dtype=torch.float64, device="cuda")
        res = B.spmv_cg(h, torch.from_numpy(b).cuda(), xt, 0.0, k, rho)
        want = oracle.cg(coo.m, coo.rows, coo.cols, coo.vals, b, x0=x0, tol=0.0, maxit=k)
        assert res.iterations == want["iterations"] and not res.breakdown
        assert rel_err(xt.cpu().numpy(), want["x"]) <= 1e-10
        np.testing.assert_allclose(rho.cpu().numpy()[:res.iterations + 1], want["rho"], rtol=1e-10)
    finally:
        B.spmv_destroy(h)


@pytest.mark.parametrize("n", [9, 255, 256, 257, 513, 4096, 4097, 8193, 32768, 32769])
def test_rows_around_the_cluster_sizes(oracle, n):
    check(oracle, matgen.laplacian_1d(n), None)


@pytest.mark.parametrize("n,w", [(700, 31), (700, 32), (4096, 31), (6000, 31), (6400, 31)])
def test_row_lengths_and_entry_limits(oracle, n, w):
    """63 and 65 entries a row; rows staged (4096) and read in place (6000); 403,000 entries."""
    check(oracle, band(n, w), B.make_config(format=B.FMT_ELL))


@pytest.mark.parametrize("fmt", [n for n, _ in SWEEP_VARIANTS])
def test_graph_form_in_every_format(oracle, fmt):
    check(oracle, matgen.laplacian_1d(33001), B.make_config(**VARIANTS[fmt]))


def test_unaligned_iterate(oracle):
    check(oracle, matgen.laplacian_1d(33001), None, shift=1)
    check(oracle, matgen.laplacian_1d(3001), None, shift=1)


@pytest.mark.parametrize("m", [1001, 40003])  # the cluster form, the graph form
def test_fp32_updates_round_product_and_sum(m):
    """fp32 vector updates round the product and the sum separately: with a
    diagonal matrix every fp32 step is one numpy rounds the same way, so x is
    equal bit by bit and the fp64 history differs by the order of its sums
    only (m terms: under m 2^-53 < 1e-11 of the sum)."""
    import torch
    rng = np.random.default_rng(m)
    d = rng.uniform(1.0, 3.0, m).astype(np.float32)
    b = rng.standard_normal(m).astype(np.float32)
    i = np.arange(m, dtype=np.int32)
    h = create(matgen.Coo(m, m, i, i, d.astype(np.float64)), B.SPMV_F32, B.make_config(format=B.FMT_ELL))
    steps = 6
    x = torch.zeros(m, device="cuda")
    hist = torch.zeros(steps + 1, dtype=torch.float64, device="cuda")
    try:
        B.spmv_cg(h, torch.from_numpy(b).cuda(), x, 0.0, steps, hist)
        torch.cuda.synchronize()
    finally:
        B.spmv_destroy(h)
    dot = lambda u, v: float(np.dot(u.astype(np.float64), v.astype(np.float64)))
    xs, r, p = np.zeros(m, np.float32), b.copy(), b.copy()
    rho = [dot(r, r)]
    for _ in range(steps):
        q = d * p
        alpha = np.float32(rho[-1] / dot(p, q))
        xs = xs + alpha * p
        r = r + (-alpha) * q
        rho.append(dot(r, r))
        p = r + np.float32(rho[-1] / rho[-2]) * p
    assert np.array_equal(x.cpu().numpy(), xs)
    assert np.allclose(hist.cpu().numpy(), rho, rtol=1e-11, atol=0.0)
