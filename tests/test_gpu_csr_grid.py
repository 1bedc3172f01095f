"""Blocks of a vector CSR product: a warp takes 32 rows whatever the lanes per
row, so no more blocks are launched than m rows divided by the block's threads
(read from the captured launch), and the products agree with the oracle
(gpu_util.TOL) from less than one wave of blocks to several."""
import ctypes

import numpy as np
import pytest

from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import TOL, create, oracle_for, rel_err, vec_dtype

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


class _KernelParams(ctypes.Structure):      # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p)] + [(n, ctypes.c_uint) for n in ("gx", "gy", "gz", "bx", "by", "bz", "smem")] + \
               [(n, ctypes.c_void_p) for n in ("params", "extra", "kern", "ctx")]


def _captured_launches(fn):
    """(blocks, threads) of the kernels fn(stream) launches, by capturing them"""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    graph, count = ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 2) == 0      # relaxed
    try:
        fn(stream.cuda_stream)
    finally:
        assert cu.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    out = []
    for node in nodes:
        kind, p = ctypes.c_int(), _KernelParams()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:                                                             # a kernel
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            out.append((p.gx, p.bx))
    assert cu.cuGraphDestroy(graph) == 0
    return out


@pytest.mark.parametrize("vt", [B.SPMV_F64, B.SPMV_F32])
@pytest.mark.parametrize("m,mean", [(31, 20.0), (33, 40.0), (5000, 16.0), (60001, 40.0), (150000, 24.0), (420000, 13.0)])
def test_blocks_of_vector_csr(oracle, vt, m, mean):
    import torch
    coo = matgen.poisson_rows(m, mean, np.random.default_rng(m)) if m > 100 else matgen.random_coo(
        m, m, int(m * mean) // 2, np.random.default_rng(m))
    x = matgen.dense_vector(coo.n, 3)
    want = oracle_for(oracle, coo, vt, x)
    xt = torch.from_numpy(x).to(vec_dtype(vt)).cuda()
    y = torch.empty(coo.m, dtype=vec_dtype(vt), device="cuda")
    h = create(coo, vt)
    try:
        for tpr in (1, 2, 4, 8, 16, 32):
            for tpb in (32, 256):
                B.spmv_set_config(h, B.make_config(format=B.FMT_CSR, threads_per_row=tpr, threads_per_block=tpb))
                y.fill_(float("nan"))
                B.spmv_run(h, 1.0, xt, 0.0, y)
                assert rel_err(y.cpu().double().numpy(), want) <= TOL[vt]
                (blocks, threads), = _captured_launches(lambda s: B.spmv_run(h, 1.0, xt, 0.0, y, s))
                assert threads == tpb and 1 <= blocks <= -(-coo.m // tpb), (tpr, tpb)
    finally:
        B.spmv_destroy(h)
