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


def _lens_matrix(lens, n, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=m, replace=False)) for m in lens]
    rp = np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int64)
    col = np.concatenate(cols).astype(np.int32)
    return synth.CSR(len(lens), n, rp, col, rng.uniform(-1, 1, col.size))


@pytest.mark.parametrize("n", [40, 1_025, 32_768])
@pytest.mark.parametrize("blen", [1, 8, 11])
def test_short_rows_four_at_a_time(n, blen):
    """Groups of four rows: empty, of 32 entries and of 33 together, of 32 products and of 33 in one row
    and in two, one column by many products, and rows that take the bitmap between rows that do not."""
    rng = np.random.default_rng(n + blen)
    m = 64 * 152 + 3
    lens = rng.choice([0, 1, 2, 3, 4], m)
    lens[:4], lens[4:8], lens[8:12] = [8, 8, 8, 8], [8, 8, 8, 9], [0, 0, 0, 0]
    lens[12:16], lens[16:20] = [30, 0, 1, 1], [33, 1, 1, 1]
    A = _lens_matrix(lens, 50, n)
    B = _lens_matrix(np.full(50, blen), n, n + 1)
    B.col[B.row_ptr[7]] = B.col[B.row_ptr[8]] = 0 if blen > 1 else B.col[0]
    rp, col, val, _, info, _ = run_gpu(A, B)
    assert_parity(A, B, rp, col, val)
    import paper_2004_13907_gb300 as sp
    assert dict(zip(sp._native.NUM_CLASSES, info["num_class_rows"]))["warp1024"] == A.rows


def test_short_rows_of_a_batch():
    import paper_2004_13907_gb300 as sp
    import oracle
    import torch
    jobs = [(_lens_matrix(np.random.default_rng(j).integers(0, 6, n), n, j), _lens_matrix(np.full(n, 3), n, 50 + j))
            for j, n in enumerate([5_000, 6, 7, 2_001, 6_000, 31])]
    batch = sp.spgemm_batch([sp.DeviceCSR.from_host(A, "cuda") for A, _ in jobs],
                            [sp.DeviceCSR.from_host(B, "cuda") for _, B in jobs])
    batch.check()
    torch.cuda.synchronize()
    for j, (A, B) in enumerate(jobs):
        ref, C = oracle.spgemm(A, B), batch.result(j)
        assert np.array_equal(C.row_ptr.cpu().numpy(), ref.row_ptr) and np.array_equal(C.col.cpu().numpy(), ref.col)
        assert np.all(np.abs(C.val.cpu().numpy() - ref.val) <= 1e-12 * ref.mag)
    batch.destroy()


@pytest.mark.parametrize("m", [1, 2, 9, 33])
def test_few_rows_times_a_large_matrix(m):
    """More blocks than rows of A: the others check B, of which every entry is looked at."""
    import paper_2004_13907_gb300 as sp
    n = 5_000
    A = _lens_matrix([7] * m, n, m)
    B = _lens_matrix([30] * n, n, m + 1)
    rp, col, val, *_ = run_gpu(A, B)
    assert_parity(A, B, rp, col, val)
    for at in (1, 2_049, 75_001, B.nnz - 1):
        bad = B.col.copy()
        bad[at] = n
        dA = sp.DeviceCSR.from_host(A, "cuda")
        dB = sp.DeviceCSR.from_host(synth.CSR(n, n, B.row_ptr, bad, B.val), "cuda")
        with pytest.raises(sp.SpgemmError) as ei:
            plan = sp.spgemm_plan(dA, dB)
            sp.spgemm_symbolic(plan)
        assert ei.value.name == "INVALID_CSR"
