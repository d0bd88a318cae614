"""The radix sort of the format conversions at its edges, against numpy: entry counts around a tile
(4,096), index widths on both sides of a digit (9 bits) and of a 32-bit key, all entries in one
row or column, int64 row pointers; out-of-range and repeated entries with 64-bit keys."""

import numpy as np
import pytest
import torch

from gpu_util import gpu_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _entries(rows, cols, nnz, seed):
    rng = np.random.default_rng(seed)
    key = np.unique(rng.integers(0, rows * cols, nnz + nnz // 8 + 8) if rows * cols > 2 * nnz else np.arange(rows * cols))
    key = rng.permutation(key)[:nnz]
    return (key // cols).astype(np.int32), (key % cols).astype(np.int32), rng.random(key.size)


def _expect(rows, r, c, v):
    o = np.lexsort((c, r))
    return np.concatenate([[0], np.cumsum(np.bincount(r, minlength=rows))]), c[o], v[o]


@pytest.mark.parametrize("rows,cols", [(1, 100_000), (100_000, 1), (512, 512), (513, 511), (1 << 15, 1 << 16),
                                       (1 << 16, 1 << 16), ((1 << 18) + 1, 1 << 18), (1 << 30, 3), (3, 1 << 30)])
@pytest.mark.parametrize("nnz", [1, 4_095, 4_096, 4_097, 70_001])
def test_coo_and_transpose(rows, cols, nnz):
    import paper_2004_13907_gb300 as sp
    r, c, v = _entries(rows, cols, nnz, rows + cols + nnz)
    if rows <= 1 << 20:
        for idx64 in (False, True):
            C = sp.coo_to_csr(rows, cols, *(torch.from_numpy(x).cuda() for x in (r, c, v)), idx64=idx64)
            for got, want in zip((C.row_ptr, C.col, C.val), _expect(rows, r, c, v)):
                assert np.array_equal(got.cpu().numpy(), want)
    if max(rows, cols) <= 1 << 20:
        T = sp.csr_transpose(C)
        for got, want in zip((T.row_ptr, T.col, T.val), _expect(cols, c, r, v)):
            assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("bad", [(-1, 5), (1 << 20, 5), (7, -3), (7, 1 << 20), None])
def test_coo_refusals_with_64_bit_keys(bad):
    import paper_2004_13907_gb300 as sp
    n = 1 << 20
    r, c, v = _entries(n, n, 9_000, 3)
    if bad is None:
        r[8_000], c[8_000] = r[17], c[17]   # a repeated pair
    else:
        r[4_500], c[4_500] = bad
    with pytest.raises(sp.SpgemmError) as ei:
        sp.coo_to_csr(n, n, *(torch.from_numpy(x).cuda() for x in (r, c, v)))
    assert ei.value.name == "INVALID_CSR"
