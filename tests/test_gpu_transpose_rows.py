"""Transposition: row pointers that do not cover the entries are refused (each entry's row is its column
in the transpose); index widths past 2^20, where the sort takes three and four passes, and COO rows past
2^20, against the same order made by torch."""

import numpy as np
import pytest
import torch

from gpu_util import gpu_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


def _matrix(rp, cols, col, idx64):
    import paper_2004_13907_gb300 as sp
    col = torch.as_tensor(col, dtype=torch.int32, device="cuda")
    return sp.DeviceCSR(len(rp) - 1, cols, torch.as_tensor(rp, dtype=torch.int64 if idx64 else torch.int32, device="cuda"),
                        col, torch.arange(col.numel(), dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("idx64", [False, True])
@pytest.mark.parametrize("rp", [[1, 3, 3, 6], [0, 3, 3, 5], [2, 3, 4, 5], [0, 4, 3, 6], [0, 3, 7, 6], [-1, 3, 3, 6], [0]])
def test_entries_of_no_row_are_refused(rp, idx64):
    import paper_2004_13907_gb300 as sp
    with pytest.raises(sp.SpgemmError) as ei:
        sp.csr_transpose(_matrix(rp, 9, [1, 4, 5, 0, 2, 8], idx64))
    assert ei.value.name == "INVALID_CSR"


@pytest.mark.parametrize("idx64", [False, True])
def test_valid_row_pointers(idx64):
    import paper_2004_13907_gb300 as sp
    T = sp.csr_transpose(_matrix([0, 3, 3, 6], 9, [1, 4, 5, 0, 4, 8], idx64))
    assert T.row_ptr.cpu().tolist() == [0, 1, 2, 2, 2, 4, 5, 5, 5, 6]
    assert T.col.cpu().tolist() == [2, 0, 0, 2, 0, 2] and T.val.cpu().tolist() == [3, 0, 1, 4, 2, 5]
    T = sp.csr_transpose(_matrix([0], 4, [], idx64))
    assert T.row_ptr.cpu().tolist() == [0] * 5 and T.nnz == 0


@pytest.mark.parametrize("nnz", [4_097, 300_001])
@pytest.mark.parametrize("rows,cols", [(1 << 24, 3), (3, 1 << 24), (5_000, (1 << 18) + 1), (7, (1 << 27) + 1), ((1 << 27) + 1, 7),
                                       ((1 << 25) + 3, 1 << 22)])
def test_wide_indices(rows, cols, nnz):
    import paper_2004_13907_gb300 as sp
    g = torch.Generator(device="cuda")
    g.manual_seed(rows + cols + nnz)
    key = torch.unique(torch.randint(0, rows * cols, (nnz,), device="cuda", generator=g))
    r, c = key // cols, key % cols
    val = torch.rand(key.numel(), dtype=torch.float64, device="cuda", generator=g)

    def row_ptr(x, n):
        return torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(torch.bincount(x, minlength=n), 0)])

    p = torch.randperm(key.numel(), device="cuda", generator=g)
    C = sp.coo_to_csr(rows, cols, r[p].int(), c[p].int(), val[p])
    assert torch.equal(C.row_ptr.long(), row_ptr(r, rows)) and torch.equal(C.col.long(), c) and torch.equal(C.val, val)
    T = sp.csr_transpose(C)
    o = torch.argsort(c * rows + r)
    assert torch.equal(T.row_ptr.long(), row_ptr(c, cols)) and torch.equal(T.col.long(), r[o]) and torch.equal(T.val, val[o])
