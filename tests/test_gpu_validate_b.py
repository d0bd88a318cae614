"""The canonical-CSR check of B (a pass of its own on the general path; A is checked as it is counted):
violations at the edges of a block's pieces (2,048 entries), in the second and later pieces of its
share, beside and inside runs of empty rows of any length, and in the row pointers; int32 and int64 row
pointers. Rows of one entry among many empty ones, whose starts are found by search. A B with millions of
empty rows is checked as fast as one without."""

import numpy as np
import pytest
import torch

from gpu_util import gpu_or_skip

pytestmark = pytest.mark.gpu

PIECE = 2_048


@pytest.fixture(autouse=True)
def _gpu():
    gpu_or_skip()


class _Check:
    """B with rows of the given lengths, columns 0, 1, ... in each; A is one row that names B's first row."""

    def __init__(self, lens, idx64, **opts):
        import paper_2004_13907_gb300 as sp
        self.opts = opts
        lens = np.asarray(lens, np.int64)
        self.rows, self.cols = lens.size, int(max(lens.max(initial=0), 4))
        rp = np.concatenate([[0], np.cumsum(lens)])
        self.starts = np.unique(rp[:-1][lens > 0])
        col = np.arange(rp[-1]) - np.repeat(rp[:-1], lens)
        dt = torch.int64 if idx64 else torch.int32
        self.nnz = int(rp[-1])
        self.rp = torch.from_numpy(rp).to("cuda", dt)
        self.col = torch.from_numpy(col.astype(np.int32)).cuda()
        self.val = torch.ones(self.nnz, dtype=torch.float64, device="cuda")
        one = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.A = sp.DeviceCSR(1, self.rows, torch.tensor([0, 1], dtype=torch.int32, device="cuda"), one,
                              torch.ones(1, dtype=torch.float64, device="cuda"))

    def plan(self, rp=None, col=None, **opts):
        import paper_2004_13907_gb300 as sp
        B = sp.DeviceCSR(self.rows, self.cols, self.rp if rp is None else rp, self.col if col is None else col, self.val)
        return sp.spgemm_plan(self.A, B, opts=sp.spgemm_opts_default(general_path=1, **opts))

    def refused(self, rp=None, col=None):
        import paper_2004_13907_gb300 as sp
        try:
            sp.spgemm_plan_destroy(self.plan(rp, col, **self.opts))
        except sp.SpgemmError as e:
            return e.name == "INVALID_CSR"
        return False

    def with_col(self, j, value):
        col = self.col.clone()
        col[j] = value
        return self.refused(col=col)

    def with_rp(self, r, change):
        rp = self.rp.clone()
        rp[r] += change
        return self.refused(rp=rp)

    def violations(self, at):
        at = [j for j in at if 0 < j < self.nnz]
        for j in at:
            assert self.with_col(j, -1) and self.with_col(j, self.cols), j
            if j not in self.starts:   # not above its predecessor
                assert self.with_col(j, int(self.col[j - 1])), j
        assert self.with_rp(0, 1) and self.with_rp(self.rows, -1)


def _canonical(rp, col):
    if rp[0] != 0 or rp[-1] != col.size or np.any(np.diff(rp) < 0):
        return False
    inside = np.ones(col.size, bool)
    inside[rp[:-1][rp[:-1] < rp[1:]]] = False
    return bool(np.all(np.diff(col)[inside[1:]] > 0))


EDGES = [1, PIECE - 1, PIECE, PIECE + 1, 2 * PIECE - 1, 2 * PIECE, 2 * PIECE + 1]
LENS = {"long": [5_000, 0, 0, 3_192, 10, 4_096, 1, 4_095],
        "short": [3, 0, 5, 1] * 3_000,
        "ones": [1] * 10_000,
        "empty_first": [0] * 20_000 + [2_500, 3] + [7] * 900,
        "empty_between": [1_000, 1_047] + [0] * 4_096 + [1, 2_047] + [0] * 50_000 + [1, 3_000] + [0] * 4_095 + [9],
        "empty_last": [2_047, 1, 2_050] + [0] * 30_000,
        "ones_among_empty": ([1] + [0] * 9) * 6_000,
        "twos_among_empty": ([0] * 40 + [2]) * 3_000}


@pytest.mark.parametrize("idx64", [False, True])
@pytest.mark.parametrize("name", sorted(LENS))
def test_violations_of_b_are_found(name, idx64):
    M = _Check(LENS[name], idx64)
    assert not M.refused()
    M.violations(EDGES + [M.nnz - 1])
    # a row that starts one entry later
    rp, col = M.rp.cpu().numpy().astype(np.int64), M.col.cpu().numpy()
    for r in sorted({1, 2, M.rows // 2, M.rows // 2 + 1, M.rows - 1}):
        moved = rp.copy()
        moved[r] += 1
        assert M.with_rp(r, 1) == (not _canonical(moved, col)), r


@pytest.mark.parametrize("idx64", [False, True])
def test_shares_of_several_pieces(idx64):
    # 4e6 entries: a block takes several pieces
    rng = np.random.default_rng(5)
    lens = np.concatenate([rng.integers(0, 13, 200_000), np.zeros(50_000, int), np.full(300, 5_000),
                           rng.integers(0, 13, 200_000), np.zeros(50_000, int), [1] * 3_000])
    M = _Check(lens, idx64)
    assert M.nnz > 912 * 2 * PIECE
    assert not M.refused()
    rp = M.rp.cpu().numpy().astype(np.int64)
    long_rows = rp[250_000]                      # the first of the rows of 5,000
    pieces = (int(long_rows) // PIECE + 1) * PIECE
    share = 3 * PIECE
    M.violations([share - 1, share, share + PIECE, share + PIECE + 1, share + 2 * PIECE, M.nnz - 1]
                 + [pieces + k * PIECE + d for k in range(4) for d in (-1, 0, 1)])
    for r in (225_000, 240_000, M.rows - 3_500):  # inside runs of empty rows
        assert M.with_rp(r, 1) and M.with_rp(r, -1), r


@pytest.mark.parametrize("name", ["long", "ones", "ones_among_empty"])
def test_on_one_sm(name):
    # six blocks, each with a share of the same number of pieces
    M = _Check(LENS[name] * 6, False, max_sms=1)
    assert not M.refused()
    pieces = -(-M.nnz // PIECE)
    share = -(-pieces // 6) * PIECE
    assert share > PIECE
    M.violations([share - 1, share, share + PIECE - 1, share + PIECE, share + PIECE + 1, 3 * share + PIECE, M.nnz - 1])


@pytest.mark.parametrize("where", ["first", "between", "last"])
def test_time_with_millions_of_empty_rows(where):
    # 4e5 entries in rows of four beside 10^7 empty rows: 80 MB of row pointers, tens of microseconds; a block
    # that walks them takes over 10 ms
    full, empty = [4] * 50_000, [0] * 10_000_000
    lens = {"first": empty + full + full, "between": full + empty + full, "last": full + full + empty}[where]
    M = _Check(lens, False)
    import paper_2004_13907_gb300 as sp
    ms = []
    for _ in range(4):
        plan = M.plan(record_timings=1)
        ms.append(sp.spgemm_plan_get_timings(plan)["validate"][0])
        sp.spgemm_plan_destroy(plan)
    assert min(ms) < 2.0, ms
    assert M.with_col(200_001, 0) and M.with_col(399_999, 9) and M.with_rp(5_000_000, 1)
