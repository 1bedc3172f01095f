"""Features on matrices that sit on the edges of the block-row kernels (4096
staged entries per 32 block rows of four rows, several
lanes a block row where rows are longer, block rows of more than 256 to 4096
entries in tiles of 2048, row lengths on either side of the shared
histogram's 4096 bins), against the oracle.  Counts are exact; the ratios are formed
from exact integers, so they agree to a few roundings (1e-12)."""
import numpy as np
import pytest

import oracle as O
from paper_2302_05662_gb300 import binding as B
from paper_2302_05662_gb300 import matgen

from gpu_util import create

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2302_05662_gb300 import build
    build.build()
    return B.load_library()


def _rows(lens, n, seed):
    """A matrix with the given row lengths and random distinct columns."""
    rng = np.random.default_rng(seed)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens] or [np.zeros(0)]).astype(np.int32)
    rows = np.repeat(np.arange(len(lens)), lens).astype(np.int32)
    return matgen.Coo(len(lens), n, rows, cols, np.ones(rows.size))


def _spans(groups, n):
    """Block rows of four rows, each (first column, entries, step)."""
    rows, cols = [], []
    for i, (first, count, step) in enumerate(r for g in groups for r in g):
        c = np.arange(first, first + count * step, step)
        c = c[c < n]
        rows.append(np.full(c.size, i))
        cols.append(c)
    rows, cols = np.concatenate(rows).astype(np.int32), np.concatenate(cols).astype(np.int32)
    return matgen.Coo(4 * len(groups), n, rows, cols, np.ones(rows.size))


CASES = {
    "staged_exactly": lambda: _rows([32] * 128, 600, 1),                 # 32 block rows of 4096 entries in all
    "staged_plus_one": lambda: _rows([32] * 127 + [33], 600, 2),
    "heavy_limit": lambda: _rows([64, 64, 64, 64, 64, 64, 64, 65] + [0] * 120, 600, 3),  # 256 and 257 entries
    "lanes_4": lambda: _rows([100] * 131, 400, 14),                      # several lanes share a block row
    "lanes_16": lambda: _rows([300] * 64, 900, 15),
    "lanes_32_heavy": lambda: _rows([900] * 38 + [1200] * 6, 1500, 16),  # on either side of 4096 a block row
    "all_heavy": lambda: _rows([1400] * 9, 1500, 17),
    "lanes_uneven_rows": lambda: _rows([1, 700, 0, 3, 400, 0, 0, 1, 2, 2, 900, 2] * 3, 1500, 18),
    "long_row_over_tiles": lambda: _rows([3, 0, 5000, 7, 2, 9], 6000, 4),
    "heavy_uneven": lambda: _rows([3000, 8, 8, 8, 1500, 1, 1, 2000, 1, 1, 1, 1], 4000, 5),
    "heavy_tiles": lambda: _rows([700, 700, 700, 700, 700, 700], 1500, 6),
    "mostly_empty_rows": lambda: matgen.random_coo(200000, 300, 60, np.random.default_rng(7)),
    "few_tiles_mostly_empty": lambda: matgen.random_coo(150000, 5000, 9000, np.random.default_rng(8)),
    "dense_blocks": lambda: matgen.block_diagonal(4100 // 4 * 4, 4, np.random.default_rng(9)),
    "band": lambda: matgen.banded(3001, 9, np.random.default_rng(10)),
    "power_law": lambda: matgen.rmat(12, 16, np.random.default_rng(11)),
    "long_lengths": lambda: _rows([4095, 4096, 4097, 9000, 1, 0], 10000, 12),  # either side of the shared histogram
    # enough rows for one lane a block row: 384 staged entries, spans of 384 and 385
    "one_lane_staged_limit": lambda: _rows([2] * 1280 + [3] * 128 + [2] * 1280 + [3] * 127 + [4] + [2] * 187200, 600, 19),
    "heavy_strides": lambda: _rows([320, 31, 32, 33, 64, 63, 65, 400, 257, 0, 0, 0, 0, 0, 0, 257, 1, 300], 700, 20),
    "heavy_clustered": lambda: _spans([[(0, 60000, 7), (30000, 9000, 1), (5, 1, 1), (59999, 1, 1)],
                                       [(2, 3000, 1), (2, 3000, 1), (1, 3000, 1), (3, 3000, 4)],
                                       [(1, 400, 3), (0, 1, 1), (600, 500, 2), (20000, 9000, 5)]], 65000),
    "single_entry": lambda: _rows([0, 0, 0, 1], 5, 13),
}


@pytest.mark.parametrize("name", list(CASES))
def test_features_at_tile_edges(name):
    coo = CASES[name]()
    h = create(coo, B.SPMV_F64)
    try:
        got = B.spmv_features(h)
    finally:
        B.spmv_destroy(h)
    want = O.features_vector(coo.m, coo.n, coo.rows, coo.cols)
    assert np.allclose(got, want, rtol=1e-12, atol=1e-15), dict(zip(O.FEATURE_NAMES, zip(got, want)))
