"""Symbolic pass of the block rows (bitmap of the columns, or a hash table in wider spaces) and of the
windowed rows (six, three or one block per SM by the bitmap's size, one when a row outweighs the rest),
against the oracle: column spaces at the edges of a bitmap word and of each rule, rows of up to one
step per warp (2,048 products) and of more, one and several chunks of 256 A entries."""

import numpy as np
import pytest

import oracle
import synth
from gpu_util import gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _rows(lens, n, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=min(m, n), replace=False)) for m in lens]
    rp = np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int64)
    col = np.concatenate(cols).astype(np.int32) if cols else np.zeros(0, np.int32)
    return synth.CSR(len(lens), n, rp, col, rng.uniform(-1, 1, col.size))


def _structure(A, B, **kw):
    import paper_2004_13907_gb300 as sp
    ref = oracle.spgemm(A, B)
    rp, col, val, _, info, _ = run_gpu(A, B, sp.spgemm_opts_default(general_path=1, **kw))
    assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
    assert np.all(np.abs(val - ref.val) <= 1e-12 * ref.mag)
    return info


@pytest.mark.parametrize("n", [1_025, 2_017, 4_096, 65_537, 262_143, 262_144, 262_145])
def test_block_rows(n):
    k = 700
    # rows of 1,025 to 2,048 products: 205 to 409 entries of five, and a few entries of hundreds
    A = _rows([205, 255, 256, 257, 300, 400, 409] * 3, k, n)
    B = _rows([5] * k, n, n + 1)
    info = _structure(A, B)
    assert info["sym_class_rows"][4] == A.rows
    _structure(_rows([3, 7, 10] * 4, 40, n + 2), _rows([200] * 40, n, n + 3))


def test_block_rows_with_more_products_than_columns():
    A = _rows([50, 300, 1_000, 2_000], 2_000, 1)
    B = _rows([40] * 2_000, 1_500, 2)
    info = _structure(A, B)
    assert info["sym_class_rows"][4] == A.rows


@pytest.mark.parametrize("n", [262_144, 262_145, 524_288, 524_289, 1 << 20, (1 << 20) + 1])
def test_window_bitmaps(n):
    A = _rows([60, 300, 700] * 60, 800, n)
    _structure(A, _rows([20] * 800, n, n + 1), force_window=1)


@pytest.mark.parametrize("n", [30_000, 400_000])
def test_a_row_that_outweighs_the_rest(n):
    A = _rows([900] + [4] * 50, 900, n)
    _structure(A, _rows([700] * 900, n, n + 1), force_window=1)
