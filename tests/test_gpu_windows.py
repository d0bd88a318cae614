"""The numeric pass over a list of windows (FP64 rows whose bitmaps are all stored) against the
oracle: column spaces around a sub-block (1,024 columns) and a window (64 of them), up to 2^20 columns;
segments of B from single products to many whole groups of 32; rows of one and of several chunks of A
entries (256); window sizes, no split table; and the same product without stored bitmaps, which takes
the other windowed kernel."""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _opts(**kw):
    import paper_2004_13907_gb300 as sp
    return sp.spgemm_opts_default(general_path=1, force_window=1, **kw)


def _skewed(k, n, seed):
    """k rows of 0 to 3,000 entries: most short, some long and dense at the first columns."""
    rng = np.random.default_rng(seed)
    lens = np.minimum((rng.pareto(0.7, k) * 6).astype(np.int64), min(n, 3000))
    rows = []
    for m in lens:
        c = (rng.random(2 * m + 8) ** (3 if m > 200 else 1) * n).astype(np.int64)
        c = np.unique(c)
        rows.append(np.sort(rng.permutation(c)[:m]))
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    col = (np.concatenate(rows) if rows else np.zeros(0)).astype(np.int32)
    return synth.CSR(k, n, rp, col, rng.random(col.size) * 2 - 1)


@pytest.mark.parametrize("n", [1, 31, 1_000, 1_024, 1_025, 32_769, 65_536, 65_537, 70_001, 262_144, 1 << 20])
@pytest.mark.parametrize("na", [5, 128, 256, 257, 300])
def test_window_list(n, na):
    k = 400
    A = synth.uniform_random(30, k, na / k, seed=n + na)
    B = _skewed(k, n, n + 7 * na)
    rp, col, val, _, info, _ = run_gpu(A, B, _opts())
    assert sum(info["num_class_rows"][:4]) == A.rows - info["num_class_rows"][11]
    assert_parity(A, B, rp, col, val)


@pytest.mark.parametrize("kw", [dict(window_hash_fill=1), dict(window_hash_fill=1024), dict(window_split_max_mb=0),
                                dict(window_cols_max_mb=0), dict(window_cols_max_mb=1)])
def test_window_list_options(kw):
    A = synth.uniform_random(60, 500, 0.1, seed=3)
    B = _skewed(500, 150_000, 5)
    rp, col, val, *_ = run_gpu(A, B, _opts(**kw))
    assert_parity(A, B, rp, col, val)


def test_window_list_long_row_of_single_products():
    # 4,000 A entries whose B rows hold one to three columns: every group of 32 spans many segments
    rng = np.random.default_rng(11)
    A = synth.CSR(2, 4_000, np.array([0, 4_000, 4_000]), np.arange(4_000, dtype=np.int32), rng.random(4_000))
    cols = [np.sort(rng.choice(90_000, 1 + k % 3, replace=False)) for k in range(4_000)]
    rp = np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int64)
    B = synth.CSR(4_000, 90_000, rp, np.concatenate(cols).astype(np.int32), rng.random(int(rp[-1])) - 0.5)
    out = run_gpu(A, B, _opts())
    assert_parity(A, B, *out[:3])
