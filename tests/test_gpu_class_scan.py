"""Row classes and row offsets over the numbers of tiles (1,024 rows each) at which their scan changes:
one, a block's worth (1,024 tiles) and more, with rows of several classes and empty ones mixed."""

import numpy as np
import pytest

import synth
from gpu_util import gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


@pytest.mark.parametrize("m", [1, 1_024, 1_025, 1 << 20, (1 << 20) + 1, 2_100_000])
def test_product_with_a_diagonal(m):
    import paper_2004_13907_gb300 as sp
    rng = np.random.default_rng(m)
    n = 3_000
    lens = rng.choice([0, 1, 3, 9], m, p=[0.3, 0.4, 0.2, 0.1])
    lens[::max(1, m // 7)] = [40, 300, 700][m % 3]
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    first = rng.integers(0, n - lens.max(), m)
    col = (np.repeat(first - rp[:-1], lens) + np.arange(rp[-1])).astype(np.int32)
    A = synth.CSR(m, n, rp, col, rng.uniform(-1, 1, int(rp[-1])))
    D = synth.CSR(n, n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.exp2(rng.integers(-3, 4, n)))
    got_rp, got_col, got_val, *_ = run_gpu(A, D, sp.spgemm_opts_default(general_path=1))
    assert np.array_equal(got_rp, rp) and np.array_equal(got_col, col)
    assert np.array_equal(got_val, A.val * D.val[col])          # one product each, by a power of two
