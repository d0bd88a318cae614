"""Host threads with a stream each, in the library at the same time: products that take the same kernels
with different amounts of shared memory (windowed rows of narrow and wide column spaces, merged rows of
short and long means, block rows of narrow and wide tables). Every call succeeds, and the results are
the product's on one thread (FP64 sums in another order), which the oracle checks."""

import threading

import numpy as np
import pytest
import torch

import synth
from gpu_util import assert_parity, gpu_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _banded(n, k, seed):
    """n x n with k consecutive columns a row, from its own on: rows of 2 k - 1 entries in its square."""
    rng = np.random.default_rng(seed)
    col = np.minimum(np.arange(n)[:, None], n - k) + np.arange(k)[None, :]
    rp = np.arange(n + 1, dtype=np.int64) * k
    return synth.CSR(n, n, rp, col.reshape(-1).astype(np.int32), rng.random(n * k) + 0.5)


def _pairs(kind):
    if kind == "windowed":   # a bitmap of 512 bytes, 19, 87 and 128 KB
        return [(synth.uniform_random(40, 300, 0.1, seed=n), synth.uniform_random(300, n, min(0.3, 300 / n), seed=n + 1),
                 dict(force_window=1)) for n in (1_000, 150_000, 700_000, 1 << 20)]
    if kind == "merged":     # rows of 15, 11 and 9 entries of C, staged in shared memory
        return [(M, M, {}) for M in (_banded(33_000, 8, 1), _banded(33_000, 6, 2), _banded(33_000, 5, 3))]
    # block rows of 1,200 entries: two levels and one, tables of 2,048 and of 4,096 entries
    return [(synth.uniform_random(40, 200, 0.15, seed=n), synth.uniform_random(200, n, 45 / n, seed=n + 1), dict(block_max=bm))
            for n, bm in ((130_000, 2_048), (900_000, 4_096), (65_000, 2_049), (1 << 22, 4_096))]


def _on_threads(work, items):
    """work(item) on two threads per item, all at once, each on a stream of its own."""
    start = threading.Barrier(2 * len(items))
    errors = []

    def run(item):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                start.wait()
                work(item)
                stream.synchronize()
        except Exception as e:   # noqa: BLE001 - reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=run, args=(i,)) for i in items for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, (len(errors), errors[0])


@pytest.mark.parametrize("kind", ["windowed", "merged", "block"])
def test_kernels_of_different_sizes(kind):
    import paper_2004_13907_gb300 as sp
    items = []
    for A, B, kw in _pairs(kind):
        dA = sp.DeviceCSR.from_host(A, "cuda")
        dB = dA if B is A else sp.DeviceCSR.from_host(B, "cuda")
        opts = sp.spgemm_opts_default(general_path=1, **kw)
        C = sp.multiply(dA, dB, opts=opts, check=True)
        H = C.to_host()
        assert_parity(A, B, H.row_ptr.numpy().astype(np.int64), H.col.numpy(), H.val.numpy())
        items.append((dA, dB, opts, C))
    torch.cuda.synchronize()

    def passes(item):
        dA, dB, opts, ref = item
        for _ in range(10):
            for _ in range(20):   # the symbolic pass
                plan = sp.spgemm_plan(dA, dB, opts=opts)
                nnz, _ = sp.spgemm_symbolic(plan)
                assert nnz == ref.nnz
                sp.spgemm_plan_destroy(plan)
            plan = sp.spgemm_plan(dA, dB, opts=opts)
            sp.spgemm_symbolic(plan)
            C = sp.alloc_output(plan)
            for _ in range(200):   # the numeric pass
                sp.spgemm_numeric(plan, C)
            sp.spgemm_plan_check(plan)
            sp.spgemm_plan_destroy(plan)
            assert torch.equal(C.row_ptr, ref.row_ptr) and torch.equal(C.col, ref.col)
            assert torch.allclose(C.val, ref.val, rtol=1e-9, atol=1e-12)

    _on_threads(passes, items)
