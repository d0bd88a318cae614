"""The canonical-CSR check of the general path at its edges: violations at the first and last entries
of a block's share (4,096 entries), rows that start there, long runs of empty rows, rows longer than a
share; int32 and int64 row pointers; an invalid B beside a valid A, and one matrix given as both."""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _matrix(lens, n):
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    col = np.concatenate([np.arange(m) for m in lens]).astype(np.int32) if len(lens) else np.zeros(0, np.int32)
    return synth.CSR(len(lens), n, rp, col, np.ones(col.size))


LENS = {"long": [5_000, 0, 0, 3_192, 10, 4_096, 1, 4_095],
        "short": [3, 0, 5, 1] * 3_000,
        "empty_run": [7, 4_089] + [0] * 9_000 + [4_096] + [0] * 300 + [2]}


def _refused(A, B, idx64):
    import paper_2004_13907_gb300 as sp
    dA = sp.DeviceCSR.from_host(A, "cuda", idx64=idx64)
    dB = dA if B is A else sp.DeviceCSR.from_host(B, "cuda", idx64=idx64)
    try:
        plan = sp.spgemm_plan(dA, dB, opts=sp.spgemm_opts_default(general_path=1))
    except sp.SpgemmError as e:
        return e.name == "INVALID_CSR"
    sp.spgemm_plan_destroy(plan)
    return False


@pytest.mark.parametrize("idx64", [False, True])
@pytest.mark.parametrize("name", sorted(LENS))
def test_violations_are_found(name, idx64):
    n = max(len(LENS[name]), 6_000)
    M = _matrix(LENS[name], n)
    I = synth.identity(n)
    assert not _refused(M, I, idx64)
    starts = set(M.row_ptr[:-1].tolist())
    at = [j for j in (1, 4_095, 4_096, 4_097, 8_191, 8_192, M.nnz - 1) if 0 < j < M.nnz]
    for j in at:
        for value in (-1, n):                      # out of range
            col = M.col.copy()
            col[j] = value
            assert _refused(synth.CSR(M.rows, n, M.row_ptr, col, M.val), I, idx64), (j, value)
        if j not in starts:                        # not above its predecessor
            col = M.col.copy()
            col[j] = col[j - 1]
            assert _refused(synth.CSR(M.rows, n, M.row_ptr, col, M.val), I, idx64), j
    for r in (0, 1, M.rows // 2, M.rows):          # row pointers
        rp = M.row_ptr.copy()
        rp[r] += 1 if r < M.rows else -1
        if r in (0, M.rows) or rp[r] > rp[r + 1] or M.row_ptr[r] in starts:
            expect = r in (0, M.rows) or rp[r] > rp[r + 1]
            if expect:
                assert _refused(synth.CSR(M.rows, n, rp, M.col, M.val), I, idx64), r
    # an invalid B
    col = I.col.copy()
    col[4_096] = n
    assert _refused(M, synth.CSR(n, n, I.row_ptr, col, I.val), idx64)


@pytest.mark.parametrize("idx64", [False, True])
def test_one_matrix_as_both(idx64):
    M = _matrix([3, 0, 5, 1] * 1_600, 6_400)
    rp, col, val, *_ = run_gpu(M, M, None, idx64_in=idx64)
    assert_parity(M, M, rp, col, val)
    import paper_2004_13907_gb300 as sp
    d = sp.DeviceCSR.from_host(M, "cuda", idx64=idx64)
    C = sp.multiply(d, d, opts=sp.spgemm_opts_default(general_path=1)).to_host()
    assert_parity(M, M, C.row_ptr.numpy(), C.col.numpy(), C.val.numpy())
    bad = M.col.copy()
    bad[4_097] = bad[4_096] = 0
    assert _refused(*[synth.CSR(M.rows, M.cols, M.row_ptr, bad, M.val)] * 2, idx64)
