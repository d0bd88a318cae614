"""Rows merged by one thread (at most 8 A entries and 64 partial products) against the oracle, with
enough of them that the merge kernels run: neighbouring rows that leave as one run and rows that do not
(other classes between them, rows longer than the warp's room), 0 to 8 A entries, B rows of 0 to 64
entries; the class counts a plan reports; a batch."""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _rows(lens, n, seed):
    """A matrix whose row i has lens[i] distinct columns out of n, near i * n / rows."""
    rng = np.random.default_rng(seed)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    row = np.repeat(np.arange(len(lens)), lens)
    t = np.arange(rp[-1]) - rp[row]
    span = 3
    col = np.minimum(row * n // len(lens), n - span * 64 - 1) + t * span + rng.integers(0, span, rp[-1])
    return synth.CSR(len(lens), n, rp, col.astype(np.int32), rng.random(int(rp[-1])) * 2 - 1)


def _check(A, B, **kw):
    import paper_2004_13907_gb300 as sp
    rp, col, val, _, info, _ = run_gpu(A, B, sp.spgemm_opts_default(general_path=1, **kw))
    assert_parity(A, B, rp, col, val)
    assert sum(info["num_class_rows"]) == A.rows and sum(info["sym_class_rows"]) == A.rows
    assert sum(info["num_class_products"]) == info["products"]
    return dict(zip(sp._native.NUM_CLASSES, info["num_class_rows"]))


@pytest.mark.parametrize("na,nb", [((1, 9), (1, 2)), ((5, 6), (5, 6)), ((7, 8), (7, 8)), ((8, 9), (8, 9)),
                                   ((0, 9), (0, 8)), ((2, 3), (20, 33)), ((1, 2), (33, 65)), ((3, 9), (1, 20))])
@pytest.mark.parametrize("kw", [dict(), dict(tiny_max=0), dict(validate=0)])
def test_merge_rows(na, nb, kw):
    rng = np.random.default_rng(na[1] + 10 * nb[1])
    m = 70_000
    A = _rows(rng.integers(*na, m), m, 1)
    B = _rows(rng.integers(*nb, m), 90_000, 2)
    _check(A, B, **kw)


@pytest.mark.parametrize("g", [33, 40])
def test_stencil3d(g):
    A = synth.laplacian3d(g)
    cls = _check(A, A)
    assert cls["warp64"] > 30_000   # the merge rows report as the warp table they come from


def test_merge_rows_between_other_classes():
    rng = np.random.default_rng(5)
    m = 120_000
    lens = np.where(rng.random(m) < 0.02, 40, 7)        # a long row now and then
    A = _rows(lens, m, 3)
    B = _rows(np.where(rng.random(m) < 0.3, 0, 7), 100_000, 4)
    _check(A, B)


def test_merge_rows_in_a_batch():
    import paper_2004_13907_gb300 as sp
    jobs = [(synth.laplacian3d(g), synth.laplacian3d(g)) for g in (34, 21, 36)]
    dev = [tuple(sp.DeviceCSR.from_host(M, "cuda") for M in job) for job in jobs]
    batch = sp.spgemm_batch([a for a, _ in dev], [b for _, b in dev], "f64", sp.spgemm_opts_default(general_path=1))
    batch.check()
    for j, (A, B) in enumerate(jobs):
        C = batch.result(j).to_host()
        assert_parity(A, B, C.row_ptr.numpy(), C.col.numpy(), C.val.numpy())
