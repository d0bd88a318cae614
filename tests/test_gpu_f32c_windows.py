"""FP32-compensated rows over the list of windows: slots of a sum and a compensation where every product
is non-negative and few (windows of 4,096 entries), wide slots (2,048 entries) where the signs mix or a
row of A has more entries than the count bound allows (about 4,000); and values whose signs change
between numeric passes of one plan."""

import numpy as np
import pytest

import oracle
import synth
from gpu_util import gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _matrix(rows, k, lens, seed, signed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.permutation(k)[:min(m, k)]) for m in lens]
    rp = np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int64)
    val = rng.uniform(-1.0 if signed else 0.0, 1.0, int(rp[-1]))
    return synth.CSR(rows, k, rp, np.concatenate(cols).astype(np.int32), val.astype(np.float32))


def _within(A, B, rp, col, val):
    """The path's contract: 2u|c| of the exact sum (and the oracle's own FP64 rounding)."""
    ref = oracle.spgemm(A, B)
    assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
    assert np.all(np.abs(val.astype(np.float64) - ref.val) <= 2.001 * U32 * np.abs(ref.val) + 2e-12 * ref.mag)


@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("n", [1_023, 1_025, 32_769, 90_000])
@pytest.mark.parametrize("fill", [1, 2_048, 4_096])
def test_slots(n, signed, fill):
    import paper_2004_13907_gb300 as sp
    k = 6_000
    A = _matrix(8, k, [1, 255, 256, 257, 300, 3_900, 4_200, 6_000], n, signed)
    B = _matrix(k, n, np.random.default_rng(n + 1).integers(0, 60, k), n + 2, signed)
    rp, col, val, _, info, _ = run_gpu(A, B, sp.spgemm_opts_default(force_window=1, window_hash_fill=fill), prec="f32c")
    assert sum(info["num_class_rows"][:4]) == A.rows
    _within(A, B, rp, col, val)


def test_signs_change_between_passes_of_a_plan():
    import paper_2004_13907_gb300 as sp
    import torch
    k, n = 2_000, 40_000
    A = _matrix(20, k, [1_500] * 20, 1, False)
    B = _matrix(k, n, [40] * k, 2, False)
    dA = sp.DeviceCSR.from_host(A, "cuda", dtype=torch.float32)
    dB = sp.DeviceCSR.from_host(B, "cuda", dtype=torch.float32)
    plan = sp.spgemm_plan(dA, dB, "f32c")
    sp.spgemm_symbolic(plan)
    C = sp.alloc_output(plan)
    for flip in (False, True, True):               # non-negative, mixed, non-negative again
        if flip:
            dA.val[1::2] *= -1
        sp.spgemm_numeric(plan, C)
        sp.spgemm_plan_check(plan)
        torch.cuda.synchronize()
        H = C.to_host()
        A.val[:] = dA.val.cpu().numpy()
        _within(A, B, H.row_ptr.numpy().astype(np.int64), H.col.numpy(), H.val.numpy())
    sp.spgemm_plan_destroy(plan)
