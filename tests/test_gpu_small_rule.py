"""Small products on both sides of the rule for sorted short rows: 8,192 and 8,193 columns, 16,384 and 16,385, one row fewer
and more than one per warp of the chip, averages at and over the limits; groups of four rows with 32 and 33
products, and a batch whose widest job decides."""

import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_parity, gpu_or_skip, run_gpu
from test_gpu_small_rows import _lens_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


@pytest.mark.parametrize("n", [8_192, 8_193, 16_384, 16_385, 30_001])
@pytest.mark.parametrize("m", [152 * 64 - 1, 152 * 64])
@pytest.mark.parametrize("alen,blen", [(8, 2), (8, 3), (9, 1), (1, 16), (2, 8)])
def test_both_sides(n, m, alen, blen):
    lens = np.full(m, alen)
    lens[:8] = [0, 1, 2, 32 // blen, 33, 1, 0, 0]
    A = _lens_matrix(lens, 40, n + m)
    B = _lens_matrix(np.full(40, blen), n, n + blen)
    rp, col, val, *_ = run_gpu(A, B)
    assert_parity(A, B, rp, col, val)


@pytest.mark.parametrize("widest", [400, 8_193, 16_385])
def test_batch(widest):
    import paper_2004_13907_gb300 as sp
    jobs = [(_lens_matrix(np.random.default_rng(j).integers(0, 6, m), 60, j), _lens_matrix(np.full(60, 3), n, 50 + j))
            for j, (m, n) in enumerate([(5_000, 90), (3_000, widest), (2_500, 400)])]
    batch = sp.spgemm_batch([sp.DeviceCSR.from_host(A, "cuda") for A, _ in jobs],
                            [sp.DeviceCSR.from_host(B, "cuda") for _, B in jobs])
    batch.check()
    torch.cuda.synchronize()
    for j, (A, B) in enumerate(jobs):
        ref, C = oracle.spgemm(A, B), batch.result(j)
        assert np.array_equal(C.row_ptr.cpu().numpy(), ref.row_ptr) and np.array_equal(C.col.cpu().numpy(), ref.col)
        assert np.all(np.abs(C.val.cpu().numpy() - ref.val) <= 1e-12 * ref.mag)
