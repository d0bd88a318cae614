"""Windowed rows where the device has no room for the list of all windows: the numeric pass lists the rows
in groups instead, with the same result, and again on the next numeric call; without room for one
row's windows it reports OOM."""

import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_parity, gpu_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


class _Limited:
    """Device allocator that refuses blocks of more than `limit` bytes after `passes` more calls."""

    def __init__(self):
        from paper_2004_13907_gb300 import _native
        self.limit, self.passes, self.refused, self.blocks = 1 << 40, 0, 0, {}

        def alloc(size, stream, ctx):
            self.passes -= 1
            if self.passes < 0 and size > self.limit:
                self.refused += 1
                return None
            t = torch.empty(size, dtype=torch.uint8, device="cuda")
            self.blocks[t.data_ptr()] = t
            return t.data_ptr()

        def free(ptr, stream, ctx):
            self.blocks.pop(ptr)

        self._fns = _native.ALLOC_FN(alloc), _native.FREE_FN(free)
        self.native = _native.Allocator(*self._fns, None)


def _plan(A, B, prec, mem):
    import paper_2004_13907_gb300 as sp
    from paper_2004_13907_gb300 import _native
    opts = sp.spgemm_opts_default(general_path=1, force_window=1, window_hash_fill=64)
    dA, dB = sp.DeviceCSR.from_host(A, "cuda"), sp.DeviceCSR.from_host(B, "cuda")
    a, b, h = dA.as_in(), dB.as_in(), ctypes.c_void_p()
    _native.check(sp.lib().spgemm_plan(ctypes.byref(a), ctypes.byref(b), sp._prec(prec), ctypes.byref(opts),
                                       ctypes.byref(mem.native), torch.cuda.current_stream().cuda_stream, ctypes.byref(h)))
    plan = sp.Plan(h.value, dA, dB, sp._prec(prec))
    sp.spgemm_symbolic(plan)
    return plan


def _inputs(prec, seed):
    dt = np.float64 if prec == "f64" else np.float32
    return (synth.uniform_random(150, 400, 0.08, seed=seed, dtype=dt),
            synth.uniform_random(400, 70_001, 2e-3, seed=seed + 1, dtype=dt))


# room for 29, 3 and 1 rows of up to 69 windows of 64 bytes
@pytest.mark.parametrize("prec", ["f64", "f32c"])
@pytest.mark.parametrize("limit", [130_000, 17_000, 4_700])
def test_list_in_groups_of_rows(limit, prec):
    import paper_2004_13907_gb300 as sp
    A, B = _inputs(prec, limit)
    mem = _Limited()
    plan = _plan(A, B, prec, mem)
    mem.limit, mem.passes = limit, 3 if prec == "f32c" else 0   # (FP32: the workspaces of the FP64 reruns come first)
    for _ in range(2):
        C = sp.alloc_output(plan)
        sp.spgemm_numeric(plan, C)
        sp.spgemm_plan_check(plan)
        H = C.to_host()
        rp, col, val = H.row_ptr.numpy().astype(np.int64), H.col.numpy(), H.val.numpy().astype(np.float64)
        if prec == "f64":
            assert_parity(A, B, rp, col, val)
        else:
            ref = oracle.spgemm(A, B)
            assert np.array_equal(rp, ref.row_ptr) and np.array_equal(col, ref.col)
            assert np.all(np.abs(val - ref.val) <= 2.001 * 2.0 ** -24 * np.abs(ref.val) + 2e-12 * ref.mag)
    assert mem.refused >= 2
    sp.spgemm_plan_destroy(plan)
    torch.cuda.synchronize()
    assert not mem.blocks


def test_no_room_for_one_row():
    import paper_2004_13907_gb300 as sp
    A, B = _inputs("f64", 7)
    mem = _Limited()
    plan = _plan(A, B, "f64", mem)
    mem.limit = 1_000
    C = sp.alloc_output(plan)
    with pytest.raises(sp.SpgemmError) as ei:
        sp.spgemm_numeric(plan, C)
    assert ei.value.name == "OOM"
    mem.limit = 1 << 40                      # and once there is room
    sp.spgemm_numeric(plan, C)
    sp.spgemm_plan_check(plan)
    H = C.to_host()
    assert_parity(A, B, H.row_ptr.numpy().astype(np.int64), H.col.numpy(), H.val.numpy())
    sp.spgemm_plan_destroy(plan)
