"""Block rows (513 to block_max entries of C) against the oracle: column spaces on both sides of the
one-level and two-level bitmaps and of the hash table, rows whose products stay in registers and
rows that enumerate them again, rows of more than one chunk of A entries, a batch whose jobs differ
in width; FP64 and FP32 compensated."""

import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _opts(**kw):
    import paper_2004_13907_gb300 as sp
    return sp.spgemm_opts_default(general_path=1, **kw)


def _block_rows(info):
    import paper_2004_13907_gb300 as sp
    cls = dict(zip(sp._native.NUM_CLASSES, info["num_class_rows"]))
    return cls["block8192"] + cls["block2048"]


def _check_f32(A, B, rp, col, val):
    ref = oracle.spgemm(A, B)
    assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
    assert np.all(np.abs(val - ref.val) <= 2 * 2.0 ** -24 * np.abs(ref.val) + 2e-12 * ref.mag)


# (columns, entries per row of A, entries per row of B): about 900, 1,500 and 3,500 entries of C
SHAPES = [(n, a, b) for n in (4_000, 32_768, 65_536, 65_537, 131_072, 1 << 20, 1 << 22, (1 << 22) + 1)
          for a, b in ((20, 45), (30, 52))] + [(9_000, 60, 80), (1 << 20, 60, 62), (6_000, 400, 12), (1 << 18, 300, 6)]


@pytest.mark.parametrize("prec", ["f64", "f32c"])
@pytest.mark.parametrize("n,a,b", SHAPES)
def test_block_rows(n, a, b, prec):
    k, dt = 700, np.float64 if prec == "f64" else np.float32
    lo = -1.0 if prec == "f64" else 0.0   # FP32 block rows need non-negative values
    A = synth.uniform_random(90, k, a / k, seed=n + a, dtype=dt, lo=lo)
    B = synth.uniform_random(k, n, b / n, seed=n + b + 1, dtype=dt, lo=lo)
    rp, col, val, _, info, _ = run_gpu(A, B, _opts(block_max=4096), prec=prec)
    assert _block_rows(info) >= 60
    if prec == "f64":
        assert_parity(A, B, rp, col, val)
    else:
        _check_f32(A, B, rp, col, val)


def test_block_rows_batch_of_widths():
    import paper_2004_13907_gb300 as sp
    jobs = [(synth.uniform_random(40, 500, 30 / 500, seed=2 * j), synth.uniform_random(500, n, 50 / n, seed=2 * j + 1))
            for j, n in enumerate((3_000, 65_536, 200_001, 40_000))]
    dev = [tuple(sp.DeviceCSR.from_host(M, "cuda") for M in job) for job in jobs]
    batch = sp.spgemm_batch([a for a, _ in dev], [b for _, b in dev], "f64", _opts())
    batch.check()
    for j, (A, B) in enumerate(jobs):
        C = batch.result(j).to_host()
        assert_parity(A, B, C.row_ptr.numpy(), C.col.numpy(), C.val.numpy())
