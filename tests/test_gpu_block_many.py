"""Block rows with many products per entry of C against the oracle: narrow column spaces (a byte per column
in the symbolic pass, sums by column in the numeric one), bands of a wide column space from any first
column and around the widths that are summed by column (2,048 and 4,096), bands that need one level of
words from their first column, scattered columns in two levels, rows of one and of several chunks of A
entries, empty rows of B, a batch; FP64 and FP32 compensated (whose two-level rows of very many products
hash)."""

import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_parity, gpu_or_skip, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _opts():
    import paper_2004_13907_gb300 as sp
    return sp.spgemm_opts_default(general_path=1, block_max=4096)


def _rows(lists, cols, rng, lo):
    rp = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    return synth.CSR(len(lists), cols, rp, np.concatenate(lists).astype(np.int32), rng.random(int(rp[-1])) * (1 - lo) + lo)


def _product(n, first, span, distinct, na, nb, seed, lo=-1.0, m=40, k=500):
    """B: rows of about nb of `distinct` columns in [first, first + span), both ends among them, every seventh
    row empty; A: m rows of na entries."""
    rng = np.random.default_rng(seed)
    pool = np.unique(np.concatenate([[first, first + span - 1], first + rng.choice(span, min(distinct, span), replace=False)]))
    B = _rows([np.zeros(0, int) if r % 7 == 3 else np.sort(rng.choice(pool, min(nb, pool.size), replace=False)) for r in range(k)],
              n, rng, lo)
    A = _rows([np.sort(rng.choice(k, na, replace=False)) for _ in range(m)], k, rng, lo)
    return A, B


def _check(A, B, prec):
    dt = np.float64 if prec == "f64" else np.float32
    A, B = A.astype(dt), B.astype(dt)
    rp, col, val, _, info, _ = run_gpu(A, B, _opts(), prec=prec)
    import paper_2004_13907_gb300 as sp
    cls = dict(zip(sp._native.NUM_CLASSES, info["num_class_rows"]))
    assert cls["block8192"] + cls["block2048"] == A.rows and info["products"] >= 8 * info["nnz_c"]
    if prec == "f64":
        assert_parity(A, B, rp, col, val)
    else:
        ref = oracle.spgemm(A, B)
        assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
        assert np.all(np.abs(val - ref.val) <= 2 * 2.0 ** -24 * np.abs(ref.val) + 2e-12 * ref.mag)


@pytest.mark.parametrize("prec", ["f64", "f32c"])
@pytest.mark.parametrize("n", [520, 1_024, 1_025, 1_500, 2_047, 2_048, 2_049, 4_095, 4_096])
def test_narrow(n, prec):
    for na, nb in ((60, n // 3), (280, n // 5)):
        _check(*_product(n, 0, n, n, na, nb, n + na, lo=-1.0 if prec == "f64" else 0.0), prec)


@pytest.mark.parametrize("prec", ["f64", "f32c"])
@pytest.mark.parametrize("n", [32_768, 65_536, 65_537, 131_072, 131_073, 300_001, 1 << 22, (1 << 22) + 1])
@pytest.mark.parametrize("span,distinct", [(600, 600), (1_024, 900), (2_017, 900), (2_048, 900), (2_049, 900), (4_096, 900),
                                           (4_097, 900), (20_000, 900), (32_768, 900), (2_048, 1_900), (4_096, 1_900),
                                           (4_097, 1_900), (32_000, 3_900)])
def test_bands(n, span, distinct, prec):
    for first in {0, 31, 32, min(12_345, n - span), n - span}:
        if 0 <= first <= n - span:
            _check(*_product(n, first, span, distinct, 60, distinct // 4, n + span + first, lo=-1.0 if prec == "f64" else 0.0,
                             m=12), prec)


@pytest.mark.parametrize("prec", ["f64", "f32c"])
def test_scattered(prec):
    for n, distinct, na in ((200_000, 900, 40), (200_000, 900, 280), (1 << 22, 1_900, 250), (1 << 22, 3_900, 250)):
        _check(*_product(n, 5, n - 9, distinct, na, distinct // 4, n + na, lo=-1.0 if prec == "f64" else 0.0), prec)


def test_batch():
    import paper_2004_13907_gb300 as sp
    jobs = [_product(n, first, span, d, 100, d // 4, n) for n, first, span, d in
            ((3_000, 0, 3_000, 1_500), (66_000, 40_001, 1_500, 1_200), (200_001, 199_000, 1_001, 900), (900, 0, 900, 900))]
    dev = [tuple(sp.DeviceCSR.from_host(M, "cuda") for M in job) for job in jobs]
    batch = sp.spgemm_batch([a for a, _ in dev], [b for _, b in dev], "f64", _opts())
    batch.check()
    for j, (A, B) in enumerate(jobs):
        C = batch.result(j).to_host()
        assert_parity(A, B, C.row_ptr.numpy(), C.col.numpy(), C.val.numpy())
