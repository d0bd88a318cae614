"""Stacking of a batch at the edges of a block's share (4,096 rows or entries), and the fall back of
the small path, which stops at the first row of C over 1,024 entries, on valid and invalid inputs."""

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _diagonal(n, entries, seed):
    """n x n, `entries` rows of one entry each at the front, the rest empty."""
    rp = np.minimum(np.arange(n + 1), entries).astype(np.int64)
    val = np.random.default_rng(seed).uniform(-1.0, 1.0, entries)
    return synth.CSR(n, n, rp, np.arange(entries, dtype=np.int32), val)


@pytest.mark.parametrize("prec", ["f64", "f32c"])
@pytest.mark.parametrize("sizes", [[(4_095, 4_095), (4_096, 4_096), (4_097, 4_097)], [(0, 0), (1, 1), (8_193, 4_097)],
                                   [(0, 0)], [(5, 0), (0, 0)]])
def test_jobs_at_the_edges_of_a_share(sizes, prec):
    import paper_2004_13907_gb300 as sp
    if prec == "f32c":
        dt, tol = torch.float32, 2.0 ** -23      # inputs and the one product rounded to FP32
    else:
        dt, tol = torch.float64, 2.0 ** -52
    jobs = [(_diagonal(n, e, 2 * j), _diagonal(n, e, 2 * j + 1)) for j, (n, e) in enumerate(sizes)]
    dA = [sp.DeviceCSR.from_host(A, "cuda", dtype=dt, idx64=j % 2 == 0) for j, (A, _) in enumerate(jobs)]
    dB = [sp.DeviceCSR.from_host(B, "cuda", dtype=dt, idx64=j % 2 == 1) for j, (_, B) in enumerate(jobs)]
    batch = sp.spgemm_batch(dA, dB, prec)
    batch.check()
    for _ in range(2 if prec == "f64" else 1):      # replay takes FP64 batches
        torch.cuda.synchronize()
        for j, (A, B) in enumerate(jobs):
            C = batch.result(j)
            want = dA[j].val.cpu().numpy().astype(np.float64) * dB[j].val.cpu().numpy().astype(np.float64)
            assert np.array_equal(C.row_ptr.cpu().numpy(), A.row_ptr)
            assert np.array_equal(C.col.cpu().numpy(), A.col)
            assert np.all(np.abs(C.val.cpu().numpy().astype(np.float64) - want) <= tol * np.abs(want))
        for d in dA:
            d.val.mul_(0.5)
        if prec == "f64":
            batch.replay()
    batch.destroy()


def test_a_long_row_among_many_short_ones():
    """One warp finds the only row over 1,024 entries; the others stop early or have already finished."""
    n = 30_000
    A = synth.uniform_random(n, n, 1e-4, seed=1)
    rp = A.row_ptr.copy()
    at, extra = 17_000, np.arange(0, n, 60, dtype=np.int32)     # a row of 500 entries, 1,500 or so in C
    lo, hi = int(rp[at]), int(rp[at + 1])
    rng = np.random.default_rng(2)
    col = np.concatenate([A.col[:lo], extra, A.col[hi:]]).astype(np.int32)
    val = np.concatenate([A.val[:lo], rng.uniform(-1, 1, extra.size), A.val[hi:]])
    rp[at + 1:] += extra.size - (hi - lo)
    A = synth.CSR(n, n, rp, col, val)
    B = synth.uniform_random(n, n, 1e-4, seed=3)
    ref = oracle.spgemm(A, B)
    assert np.diff(ref.row_ptr).max() > 1_024
    got_rp, got_col, got_val, *_ = run_gpu(A, B)
    assert_parity(A, B, got_rp, got_col, got_val)


def test_an_invalid_input_behind_a_long_row_is_refused():
    import paper_2004_13907_gb300 as sp
    A = synth.uniform_random(400, 400, 0.5, seed=4)
    B = synth.uniform_random(400, 20_000, 0.01, seed=5)
    acol, bcol = A.col.copy(), B.col.copy()
    acol[-1] = 400
    bcol[1], bcol[0] = bcol[0], bcol[1]
    for Ai, Bi in ((synth.CSR(400, 400, A.row_ptr, acol, A.val), B),
                   (A, synth.CSR(400, 20_000, B.row_ptr, bcol, B.val))):
        dA, dB = sp.DeviceCSR.from_host(Ai, "cuda"), sp.DeviceCSR.from_host(Bi, "cuda")
        with pytest.raises(sp.SpgemmError) as ei:
            plan = sp.spgemm_plan(dA, dB)
            sp.spgemm_symbolic(plan)
        assert ei.value.name == "INVALID_CSR"
