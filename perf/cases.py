"""Performance cases of the SpGEMM framework: what its users have it compute, through the public
Python entry points, over the sizes its configurations, tests and benchmark use.

Every matrix is made on the GPU from a seed. The matrices are those of the benchmark in torch:
uniform random patterns (the single product of 10,000 rows and the jobs of the batched and served
workloads), 2D and 3D five- and seven-point stencils, the multigrid Galerkin operator, and R-MAT
graphs; stencil and prolongator values are drawn too (a heterogeneous diffusion operator). A
case fixes each random pattern up to the index its rows and columns start from, which the seed
gives: two seeds are different matrices whose results have the same sizes.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2004_13907_gb300 as sp

DEVICE = "cuda"
# the drawn cases stay within the largest listed one (R-MAT 2^19: about 8e9 partial products)
MAX_PRODUCTS = 6e9
MAX_ENTRIES = 3e9


# ---------------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest served and batched jobs: launches, the host's work and latency
        {"name": "uniform_tiny", "kind": "uniform", "m": 300, "k": 300, "n": 300, "density": 1e-2,
         "prec": "f64", "idx64": False},
        # the benchmark's single small product
        {"name": "uniform_10k", "kind": "uniform", "m": 10_000, "k": 10_000, "n": 10_000, "density": 1e-3,
         "prec": "f64", "idx64": False},
        # a middle job of the batched and served workloads, rectangular: rows of C of about 1,500 entries
        {"name": "uniform_20k", "kind": "uniform", "m": 20_011, "k": 19_997, "n": 20_003, "density": 2e-3,
         "prec": "f64", "idx64": True},
        # a heavy job of the batched and served workloads: rows of C of about 16,000 entries
        {"name": "uniform_30k_dense", "kind": "uniform", "m": 30_000, "k": 30_000, "n": 30_000, "density": 5e-3,
         "prec": "f64", "idx64": False},
        # squares of stencil matrices: the benchmark's 1024^2 grid, and a served 3D grid of odd size
        {"name": "stencil2d_1024", "kind": "stencil", "dims": 2, "grid": 1024},
        {"name": "stencil3d_97", "kind": "stencil", "dims": 3, "grid": 97},
        # multigrid setup: R = P^T, then the coarse operator R*(A*P), the second product reading
        # the first one's result
        {"name": "galerkin_1024", "kind": "galerkin", "grid": 1024},
        # R-MAT squares: new values on a kept plan (numeric pass only), the FP32 compensated
        # product, and the largest whole FP64 product whose result can be held twice
        {"name": "rmat_17_recompute", "kind": "rmat", "scale": 17, "degree": 16, "prec": "f64", "recompute": True},
        {"name": "rmat_17_f32c", "kind": "rmat", "scale": 17, "degree": 16, "prec": "f32c", "recompute": False},
        {"name": "rmat_19", "kind": "rmat", "scale": 19, "degree": 16, "prec": "f64", "recompute": False},
        # small jobs of the batched workload as one batch
        {"name": "batch_20", "kind": "batch", "jobs": 20, "sizes": 1},
        # assembly: graph edges in arrival order to canonical CSR
        {"name": "coo_18", "kind": "coo", "scale": 18, "degree": 16},
    ]


def draw(rng):
    def logu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    while True:
        kind = rng.choice(["uniform", "uniform", "uniform", "stencil", "galerkin", "rmat", "rmat", "batch", "coo"])
        if kind == "uniform":
            n = logu(100, 50_000)
            m, k, n = (max(1, int(n * rng.uniform(0.8, 1.2))) for _ in range(3))
            case = {"kind": kind, "m": m, "k": k, "n": n, "density": float("%.3g" % logu(1e-4, 1e-2)),
                    "prec": rng.choice(["f64", "f64", "f32c"]), "idx64": rng.random() < 0.3}
        elif kind == "stencil":
            dims = rng.choice([2, 3])
            case = {"kind": kind, "dims": dims, "grid": int(logu(48, 1500) if dims == 2 else logu(24, 128))}
        elif kind == "galerkin":
            case = {"kind": kind, "grid": 2 * int(logu(32, 700))}
        elif kind == "rmat":
            case = {"kind": kind, "scale": rng.randint(10, 18), "degree": rng.randint(4, 16),
                    "prec": rng.choice(["f64", "f64", "f32c"]), "recompute": rng.random() < 0.3}
        elif kind == "batch":
            case = {"kind": kind, "jobs": rng.randint(2, 20), "sizes": rng.randint(2, 1 << 20)}
        else:
            case = {"kind": kind, "scale": rng.randint(10, 19), "degree": rng.randint(4, 16)}
        products, entries = _expected(case)
        if products <= MAX_PRODUCTS and entries <= MAX_ENTRIES:
            return case


# ---------------------------------------------------------------------------------- inputs

def _generator(*numbers):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(random.Random(repr(numbers)).getrandbits(62))
    return g


def _rotated(keys, rows, cols, down, right):
    """Ascending keys row * cols + column of the pattern moved cyclically by (down, right)."""
    r = torch.div(keys, cols, rounding_mode="floor")
    c = (keys - r * cols + right) % cols
    return torch.sort((r + down) % rows * cols + c).values


def _from_keys(rows, cols, keys, val, idx64):
    """CSR from ascending keys row * cols + column."""
    r = torch.div(keys, cols, rounding_mode="floor")
    rp = torch.zeros(rows + 1, dtype=torch.int64, device=DEVICE)
    rp[1:] = torch.cumsum(torch.bincount(r, minlength=rows), 0)
    return sp.DeviceCSR(rows, cols, rp if idx64 else rp.to(torch.int32), (keys - r * cols).to(torch.int32), val)


def _uniform(m, n, density, pattern, down, right, gen, dtype, idx64):
    count = max(1, int(round(m * n * density)))
    keys = torch.unique(torch.randint(0, m * n, (count,), generator=pattern, device=DEVICE))
    val = torch.rand(keys.numel(), generator=gen, device=DEVICE, dtype=dtype) * 2 - 1
    return _from_keys(m, n, _rotated(keys, m, n, down, right), val, idx64)


def _uniform_pair(m, k, n, density, seed, job, dtype, idx64):
    pattern, gen = _generator(m, k, n, density, job), _generator(seed, job)
    rng = random.Random(repr((seed, job)))
    down, inner, right = rng.randrange(m), rng.randrange(k), rng.randrange(n)
    return (_uniform(m, k, density, pattern, down, inner, gen, dtype, idx64),
            _uniform(k, n, density, pattern, inner, right, gen, dtype, idx64))


def _rmat_keys(scale, degree, seed):
    """Distinct edges, row * 2^scale + column ascending, quadrants (.57, .19, .19, .05), the
    vertices numbered from one that the seed gives."""
    count, n = degree << scale, 1 << scale
    pattern = _generator(scale, degree)
    r = torch.zeros(count, dtype=torch.int64, device=DEVICE)
    c = torch.zeros(count, dtype=torch.int64, device=DEVICE)
    for _ in range(scale):
        u = torch.rand(count, generator=pattern, device=DEVICE)
        r = r * 2 + (u >= 0.76)
        c = c * 2 + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    first = random.Random(seed).randrange(n)
    return _rotated(torch.unique((r << scale) | c), n, n, first, first)


def _rmat(scale, degree, seed, dtype):
    keys = _rmat_keys(scale, degree, seed)
    val = torch.rand(keys.numel(), generator=_generator(seed), device=DEVICE, dtype=dtype)
    return _from_keys(1 << scale, 1 << scale, keys, val, False)


def _stencil(dims, grid, gen):
    """Nearest-neighbour stencil of a grid^dims box, drawn off-diagonals, a dominant diagonal."""
    rows = grid ** dims
    idx = torch.arange(rows, device=DEVICE)
    strides = [grid ** (dims - 1 - d) for d in range(dims)]
    parts = [idx * rows + idx]
    for s in strides:
        x = torch.div(idx, s, rounding_mode="floor") % grid
        parts += [(idx * rows + idx - s)[x > 0], (idx * rows + idx + s)[x < grid - 1]]
    keys = torch.sort(torch.cat(parts)).values
    val = -0.5 - torch.rand(keys.numel(), generator=gen, device=DEVICE, dtype=torch.float64)
    val = torch.where(torch.div(keys, rows, rounding_mode="floor") == keys % rows, 2.0 * dims - val, val)
    return _from_keys(rows, rows, keys, val, False)


def _prolongator(grid, gen):
    """One entry per fine node: its 2x2 aggregate, with a drawn weight."""
    half = grid // 2
    f = torch.arange(grid * grid, device=DEVICE)
    col = torch.div(f, 2 * grid, rounding_mode="floor") * half + torch.div(f % grid, 2, rounding_mode="floor")
    val = 0.5 + torch.rand(f.numel(), generator=gen, device=DEVICE, dtype=torch.float64)
    return sp.DeviceCSR(grid * grid, half * half, torch.arange(grid * grid + 1, dtype=torch.int32, device=DEVICE),
                        col.to(torch.int32), val)


def _job_sizes(case):
    """(n, density) of a batch's jobs: the batched workload's distribution below 1e6 partial products."""
    rng, out = random.Random(case["sizes"]), []
    while len(out) < case["jobs"]:
        n = int(round(math.exp(rng.uniform(math.log(100), math.log(50_000)))))
        d = math.exp(rng.uniform(math.log(1e-4), math.log(1e-2)))
        if n ** 3 * d * d < 1e6:
            out.append((n, d))
    return out


def _dtype(prec):
    return torch.float64 if prec == "f64" else torch.float32


def _inputs(case, seed):
    kind, gen = case["kind"], _generator(seed)
    if kind == "uniform":
        return list(_uniform_pair(case["m"], case["k"], case["n"], case["density"], seed, 0, _dtype(case["prec"]),
                                  case["idx64"]))
    if kind == "stencil":
        return [_stencil(case["dims"], case["grid"], gen)] * 2
    if kind == "galerkin":
        return [_stencil(2, case["grid"], gen), _prolongator(case["grid"], gen)]
    if kind == "rmat":
        return [_rmat(case["scale"], case["degree"], seed, _dtype(case["prec"]))] * 2
    if kind == "batch":
        pairs = [_uniform_pair(n, n, n, d, seed, j, torch.float64, False) for j, (n, d) in enumerate(_job_sizes(case))]
        return [[A for A, _ in pairs], [B for _, B in pairs]]
    keys = _rmat_keys(case["scale"], case["degree"], seed)
    keys = keys[torch.randperm(keys.numel(), generator=gen, device=DEVICE)]
    val = torch.rand(keys.numel(), generator=gen, device=DEVICE, dtype=torch.float64)
    return [(keys >> case["scale"]).to(torch.int32), (keys & ((1 << case["scale"]) - 1)).to(torch.int32), val]


def prepare(case, seed):
    state = {"case": case, "in": _inputs(case, seed)}
    if case.get("recompute"):
        A, B = state["in"]
        plan = sp.spgemm_plan(A, B, case["prec"])
        sp.spgemm_symbolic(plan)
        state["plan"], state["C"] = plan, sp.alloc_output(plan)
    return state


# ---------------------------------------------------------------------------------- one pass

def _arrays(M):
    return [M.row_ptr, M.col, M.val]


class _Owned(list):
    """Results that are views of memory another object owns, held with that owner."""

    owner = None


def run(state):
    case, ins = state["case"], state["in"]
    kind = case["kind"]
    if kind == "galerkin":
        A, P = ins
        R = sp.csr_transpose(P)
        AP = sp.multiply(A, P)
        return [_arrays(R), _arrays(AP), _arrays(sp.multiply(R, AP))]
    if kind == "batch":
        batch = sp.spgemm_batch(*ins)
        out = _Owned(_arrays(batch.result(j)) for j in range(len(batch)))
        out.owner = batch
        return out
    if kind == "coo":
        n = 1 << case["scale"]
        return _arrays(sp.coo_to_csr(n, n, *ins))
    if "plan" in state:
        return _arrays(sp.spgemm_numeric(state["plan"], state["C"]))
    return _arrays(sp.multiply(*ins, case.get("prec", "f64")))


# ---------------------------------------------------------------------------------- work

def _rmat_expected(scale, degree):
    """Expected (entries of A, partial products of A*A, entries of A*A) of an R-MAT graph whose
    repeated edges are merged. A pair (i, j) is described by how many of its bits are (0,0), (0,1),
    (1,0), (1,1); an edge is there with probability 1 - exp(-samples * its quadrant product)."""
    lq = np.log(np.array([[0.57, 0.19], [0.19, 0.05]]))
    samples = float(degree << scale)

    def edge(log_q):
        return -np.expm1(-samples * np.exp(log_q))

    fact = [math.lgamma(t + 1) for t in range(scale + 1)]
    nnz = products = entries = 0.0
    for n00 in range(scale + 1):
        for n01 in range(scale + 1 - n00):
            for n10 in range(scale + 1 - n00 - n01):
                n11 = scale - n00 - n01 - n10
                pairs = math.exp(fact[scale] - fact[n00] - fact[n01] - fact[n10] - fact[n11])
                nnz += pairs * float(edge(n00 * lq[0, 0] + n01 * lq[0, 1] + n10 * lq[1, 0] + n11 * lq[1, 1]))
                log_ik, log_kj, log_ways = 0.0, 0.0, 0.0
                for axis, (cnt, bi, bj) in enumerate(((n00, 0, 0), (n01, 0, 1), (n10, 1, 0), (n11, 1, 1))):
                    ones = np.arange(cnt + 1)   # middle indices by how many of these bits are 1
                    shape = [1] * 4
                    shape[axis] = cnt + 1
                    ways = fact[cnt] - np.array([fact[t] + fact[cnt - t] for t in ones])
                    log_ways = log_ways + ways.reshape(shape)
                    log_ik = log_ik + (ones * lq[bi, 1] + (cnt - ones) * lq[bi, 0]).reshape(shape)
                    log_kj = log_kj + (ones * lq[1, bj] + (cnt - ones) * lq[0, bj]).reshape(shape)
                mean = float(np.sum(np.exp(log_ways) * edge(log_ik) * edge(log_kj)))
                products += pairs * mean
                entries += pairs * -math.expm1(-mean)
    return nnz, products, entries


def _stencil_counts(dims, grid):
    """Entries of a stencil matrix, partial products and entries of its square."""
    axis = [0.0] * 4   # neighbours per axis: sum of 1, c, c^2, and two-step neighbours over a line
    for x in range(grid):
        c = (x > 0) + (x < grid - 1)
        axis[0] += 1
        axis[1] += c
        axis[2] += sum(1 + (0 < y < grid - 1) for y in (x - 1, x + 1) if 0 <= y < grid)
        axis[3] += (x > 1) + (x < grid - 2)
    line, c1, c2, far = axis
    rows = line ** dims
    one = dims * c1 * line ** (dims - 1)                                  # neighbour pairs
    cross = dims * (dims - 1) * c1 * c1 * line ** (dims - 2)              # steps on two axes, in order
    two = dims * c2 * line ** (dims - 1)                                  # two steps on one axis
    nnz = rows + one
    products = rows + 2 * one + cross + two
    entries = rows + one + cross / 2 + dims * far * line ** (dims - 1)
    return nnz, products, entries


def _expected(case):
    """Expected partial products and entries of the results."""
    kind = case["kind"]
    if kind == "uniform":
        per = case["k"] * case["density"] ** 2
        return case["m"] * case["n"] * per, case["m"] * case["n"] * -math.expm1(-per)
    if kind == "stencil":
        return _stencil_counts(case["dims"], case["grid"])[1:]
    if kind == "galerkin":
        nnz, half = _stencil_counts(2, case["grid"])[0], (case["grid"] // 2) ** 2
        ap = 3.0 * 4 * half     # a fine node reaches three aggregates
        return nnz + ap, ap + 5.0 * half
    if kind == "rmat":
        return _rmat_expected(case["scale"], case["degree"])[1:]
    if kind == "batch":
        per = [(n, n * d * d) for n, d in _job_sizes(case)]
        return sum(n * n * p for n, p in per), sum(n * n * -math.expm1(-p) for n, p in per)
    return 0.0, _rmat_expected(case["scale"], case["degree"])[0]


def work(case):
    """Each input read once and each output written once; a multiplication and an addition per
    partial product."""
    kind = case["kind"]
    products, entries = _expected(case)
    v = 4 if case.get("prec") == "f32c" else 8
    if kind == "uniform":
        p = 8 if case["idx64"] else 4
        inputs = (4 + v) * case["density"] * case["k"] * (case["m"] + case["n"]) + p * (case["m"] + case["k"])
        rows = 4 * case["m"]
    elif kind == "stencil":
        n = case["grid"] ** case["dims"]
        inputs, rows = 12 * _stencil_counts(case["dims"], case["grid"])[0] + 4 * n, 4 * n
    elif kind == "galerkin":
        n, half = case["grid"] ** 2, (case["grid"] // 2) ** 2
        inputs = 12 * (_stencil_counts(2, case["grid"])[0] + n) + 8 * n
        rows = 12 * n + 4 * (n + 2 * half)              # R's entries and the three row pointers
    elif kind == "rmat":
        inputs, rows = (4 + v) * _rmat_expected(case["scale"], case["degree"])[0] + (4 << case["scale"]), 4 << case["scale"]
    elif kind == "batch":
        inputs = sum(2 * (12 * n * n * d + 4 * n) for n, d in _job_sizes(case))
        rows = sum(8 * n for n, _ in _job_sizes(case))
    else:
        inputs, rows = 16 * entries, 4 << case["scale"]
    return {"bytes": inputs + rows + (4 + v) * entries, "flops": 2 * products}


# ---------------------------------------------------------------------------------- 64 bits

def _multiply64(A, B, cols, chunk=1 << 27):
    """(row_ptr, col, val) of A*B from (row_ptr, col, val) triples: the partial products of a run
    of rows are listed, sorted by (row, column) and summed per group."""
    arp, acol, aval = A[0].to(torch.int64), A[1].to(torch.int64), A[2].to(torch.float64)
    brp, bcol, bval = B[0].to(torch.int64), B[1], B[2].to(torch.float64)
    rows = arp.numel() - 1
    per_entry = (brp[1:] - brp[:-1])[acol]
    upto = torch.zeros(acol.numel() + 1, dtype=torch.int64, device=arp.device)
    torch.cumsum(per_entry, 0, out=upto[1:])
    row_upto = upto[arp].cpu().numpy()
    row_of = torch.repeat_interleave(torch.arange(rows, device=arp.device), arp[1:] - arp[:-1])
    counts = torch.zeros(rows, dtype=torch.int64, device=arp.device)
    out_col, out_val, r0 = [], [], 0
    while r0 < rows:
        r1 = max(r0 + 1, int(np.searchsorted(row_upto, row_upto[r0] + chunk, side="right")) - 1)
        e0, e1 = int(arp[r0]), int(arp[r1])
        ent = torch.repeat_interleave(torch.arange(e0, e1, device=arp.device), per_entry[e0:e1])
        j = torch.arange(ent.numel(), device=arp.device) + int(row_upto[r0]) - upto[ent] + brp[acol[ent]]
        keys, order = torch.sort(row_of[ent].sub_(r0).mul_(cols).add_(bcol[j]))
        v = (aval[ent] * bval[j])[order]
        del ent, j, order
        keys, terms = torch.unique_consecutive(keys, return_counts=True)
        out_val.append(torch.segment_reduce(v, "sum", lengths=terms, unsafe=True) if v.numel() else v)
        r = torch.div(keys, cols, rounding_mode="floor")
        counts[r0:r1] = torch.bincount(r, minlength=r1 - r0)
        out_col.append((keys - r * cols).to(torch.int32))
        del keys, terms, r, v
        r0 = r1
    rp = torch.zeros(rows + 1, dtype=torch.int64, device=arp.device)
    rp[1:] = torch.cumsum(counts, 0)
    return rp, torch.cat(out_col), torch.cat(out_val)


def exact(case, seed):
    ins, kind = _inputs(case, seed), case["kind"]

    def product(A, B):
        return [None, None, _multiply64(_arrays(A), _arrays(B), B.cols)[2]]

    if kind == "galerkin":
        A, P = ins
        order = torch.sort(P.col.to(torch.int64), stable=True).indices
        rp = torch.zeros(P.cols + 1, dtype=torch.int64, device=DEVICE)
        rp[1:] = torch.cumsum(torch.bincount(P.col, minlength=P.cols), 0)
        R = (rp, order, P.val[order])
        AP = _multiply64(_arrays(A), _arrays(P), P.cols)
        return [[None, None, R[2]], [None, None, AP[2]], [None, None, _multiply64(R, AP, P.cols)[2]]]
    if kind == "batch":
        return [product(A, B) for A, B in zip(*ins)]
    if kind == "coo":
        row, col, val = ins
        return [None, None, val[torch.argsort((row.to(torch.int64) << case["scale"]) | col)]]
    return product(*ins)
