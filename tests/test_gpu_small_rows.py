"""Small products whose longest row of C is at the edges of a warp's tables (odd and even counts, the
most of 1,024 entries) in column spaces at the edges of the bitmap sizes, up to the most shared memory a
block takes; the last and first columns; rows of one step of 128 products and of more."""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


@pytest.mark.parametrize("n", [1, 33, 1_024, 1_025, 8_192, 16_384, 16_385, 32_767, 32_768])
@pytest.mark.parametrize("longest", [1, 127, 128, 129, 1_023, 1_024])
def test_longest_row(n, longest):
    rng = np.random.default_rng(n + longest)
    longest = min(longest, n)
    # row 0 of B: `longest` columns with the first and the last; the others: subsets of a few of them
    cols = np.unique(np.concatenate([[0, n - 1], rng.permutation(n)[:longest]]))
    cols = np.sort(np.concatenate([cols[:1], cols[-1:], cols[1:-1]])[:longest]) if longest > 1 else cols[-1:]
    rows = [cols] + [np.sort(rng.permutation(cols)[:rng.integers(0, min(longest, 9) + 1)]) for _ in range(39)]
    rp = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    col = np.concatenate(rows).astype(np.int32)
    B = synth.CSR(40, n, rp, col, rng.uniform(-1, 1, col.size))
    D = rng.uniform(-1, 1, (700, 40)) * (rng.random((700, 40)) < rng.choice([0.05, 0.3, 1.0], (700, 1)))
    A = synth.from_dense(D)
    rp, col, val, _, info, _ = run_gpu(A, B)
    assert_parity(A, B, rp, col, val)
    import paper_2004_13907_gb300 as sp
    cls = dict(zip(sp._native.NUM_CLASSES, info["num_class_rows"]))
    assert cls["warp1024"] == A.rows
    assert int(np.diff(rp).max()) == longest
