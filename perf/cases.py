"""The work that performance is judged by: CSR products through the public entry points, on synthetic matrices made on the GPU.

Matrix families (the ones this repository's generators draw, made here on the device so that they are quick to make):
  scatter    nnz = 1 % of rows x 2048 positions, uniform over the matrix: the small operators of the paper's Table 6
  grid5      5-point Laplacian on an N x N grid: one smoothing or CG step of a 2-D solver
  stencil27  27-point stencil on an N^3 grid: the same for a 3-D solver
  uniform    a fixed number of uniformly random columns in every row: k-nearest-neighbour graphs, hashed features, fixed fan-out
  rmat       R-MAT graph with 8 edges per vertex: power-law rows (most of them empty or tiny, a few of tens of thousands),
             with its hubs packed at the low indices or (relabel) spread over all of them
  skewed     row lengths drawn from a log-normal: meshes of mixed elements, bags of tokens, sampled neighbourhoods
A pass is one call (the "fresh" operation: plan, product, and the plan's release).  Everything is seeded."""
import math

import torch

import paper_2603_07169_b200 as b200sp

DEV = "cuda"


# ---------------------------------------------------------------------------------------------------------------- the cases
def _case(op, matrix, dtype, alpha=1.0, beta=0.0, k=1, relabel=False, **size):
    return dict(op=op, matrix=matrix, dtype=dtype, alpha=alpha, beta=beta, k=k, relabel=relabel, **size)


def listed():
    return [
        # the smallest operator of the paper's SpMV sizes: nothing but launch latency and the host's share of a call
        dict(_case("spmv", "scatter", "f32", m=1024, n=2048), name="spmv scatter 1k f32"),
        # one step of a 2-D solver whose grid is small: a few microseconds of work, called thousands of times
        dict(_case("spmv", "grid5", "f32", m=256 * 256, n=256 * 256), name="spmv grid5 256^2 f32"),
        # fixed fan-out graph, the headline workload of the benchmark: random gathers of x, y updated in place
        dict(_case("spmv", "uniform", "f32", alpha=1.5, beta=0.5, m=1 << 20, n=1 << 20, per_row=16), name="spmv uniform 2^20 f32"),
        # one PageRank-like step on a power-law graph
        dict(_case("spmv", "rmat", "f32", m=1 << 22, n=1 << 22), name="spmv rmat 2^22 f32"),
        # one step of a large 3-D solver with half-width storage: the largest matrix, bound by memory
        dict(_case("spmv", "stencil27", "bf16", m=160 ** 3, n=160 ** 3), name="spmv stencil27 160^3 bf16"),
        # the same product with the matrix held by columns (A given, A^T x wanted)
        dict(_case("spmv_csc", "uniform", "f32", alpha=1.5, beta=0.5, m=1 << 20, n=1 << 20, per_row=16), name="spmv csc 2^20 f32"),
        # block of right-hand sides / node features, the ordinary width
        dict(_case("spmm", "uniform", "f32", k=64, m=1 << 19, n=1 << 19, per_row=32), name="spmm uniform k64 f32"),
        # wide features with half-width storage: the most arithmetic of all cases
        dict(_case("spmm", "uniform", "bf16", k=256, m=1 << 19, n=1 << 19, per_row=32), name="spmm uniform k256 bf16"),
        # feature aggregation over a power-law graph
        dict(_case("spmm", "rmat", "f32", k=64, m=1 << 22, n=1 << 22), name="spmm rmat k64 f32"),
        # the paper's SpMM shape: few columns, very wide B (a sparse weight matrix times activations)
        dict(_case("spmm", "scatter", "f32", k=4096, m=1 << 16, n=2048), name="spmm scatter k4096 f32"),
        # odd sizes throughout: features whose width is no multiple of a vector, rows of uneven length
        dict(_case("spmm", "skewed", "bf16", k=50, beta=1.0, m=150_001, n=120_007, per_row=11), name="spmm skewed k50 bf16"),
        # a sampled neighbourhood: the pattern is new in every step, so the plan is made and dropped with it
        dict(_case("spmm_fresh", "skewed", "f32", k=128, m=20_011, n=90_001, per_row=10), name="spmm fresh k128 f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    dtype = rng.choice(("f32", "bf16"))
    alpha, beta = rng.choice(((1.0, 0.0), (1.0, 0.0), (1.5, 0.5), (1.0, 1.0)))
    if beta == 1.0:
        alpha = -0.5
    kind = rng.choice(("small", "grid", "uniform", "rmat", "csc", "mm_uniform", "mm_rmat", "mm_scatter", "mm_skewed", "mm_fresh"))
    if kind == "small":
        return _case("spmv", "scatter", dtype, alpha, beta, m=_log(rng, 1024, 32768), n=2048)
    if kind == "grid":
        if rng.random() < 0.5:
            m = _log(rng, 64, 1024) ** 2
            return _case("spmv", "grid5", dtype, alpha, beta, m=m, n=m)
        m = _log(rng, 24, 160) ** 3
        return _case("spmv", "stencil27", dtype, alpha, beta, m=m, n=m)
    if kind in ("uniform", "csc"):
        per_row = rng.choice((4, 7, 8, 11, 16, 16, 20, 32))
        m = _log(rng, 1 << 14, (1 << 24) // per_row)
        return _case("spmv" if kind == "uniform" else "spmv_csc", "uniform", dtype, alpha, beta, m=m, n=m, per_row=per_row)
    if kind == "rmat":
        m = 1 << rng.randint(15, 22)
        return _case("spmv", "rmat", dtype, alpha, beta, m=m, n=m, relabel=rng.random() < 0.5)
    if kind == "mm_uniform":
        per_row = rng.choice((6, 8, 13, 16, 32, 32))
        k = rng.choice((8, 16, 32, 64, 64, 72, 100, 128, 256))
        m = _log(rng, 1 << 14, (1 << 24) // per_row // max(1, k // 128))
        return _case("spmm", "uniform", dtype, alpha, beta, k=k, m=m, n=m, per_row=per_row)
    if kind == "mm_rmat":
        m = 1 << rng.randint(14, 21)
        return _case("spmm", "rmat", dtype, alpha, beta, k=rng.choice((16, 32, 64, 64, 128)), m=m, n=m, relabel=rng.random() < 0.5)
    if kind == "mm_scatter":
        return _case("spmm", "scatter", dtype, alpha, beta, k=8 * _log(rng, 32, 512), m=_log(rng, 1024, 65536), n=2048)
    if kind == "mm_skewed":
        m = _log(rng, 5000, 300_000)
        return _case("spmm", "skewed", dtype, alpha, beta, k=rng.randint(2, 130), m=m, n=max(3000, int(m * rng.uniform(0.5, 2.0))), per_row=rng.randint(4, 24))
    m = _log(rng, 4000, 50_000)
    return _case("spmm_fresh", "skewed", dtype, alpha, beta, k=rng.choice((32, 64, 100, 128, 256)), m=m, n=int(m * rng.uniform(1.0, 8.0)), per_row=rng.randint(4, 24))


# ------------------------------------------------------------------------------------------------------------- the matrices
def _nnz(c):
    if c["matrix"] == "scatter":
        return c["m"] * c["n"] // 100
    if c["matrix"] == "grid5":
        side = math.isqrt(c["m"])
        return 5 * side * side - 4 * side
    if c["matrix"] == "stencil27":
        return (3 * round(c["m"] ** (1 / 3)) - 2) ** 3
    if c["matrix"] == "rmat":
        return 8 * c["m"]
    return c["m"] * c["per_row"]


def _distinct(keys_of, nnz, g):
    """Exactly nnz distinct keys, ascending: keys_of(count) drawn until there are enough, then a random subset of them."""
    keys = torch.unique(keys_of(nnz + nnz // 8 + 64))
    while keys.numel() < nnz:
        keys = torch.unique(torch.cat((keys, keys_of(nnz // 4 + 64))))
    if keys.numel() > nnz:
        keep = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
        keep[torch.randperm(keys.numel(), generator=g, device=DEV)[: keys.numel() - nnz]] = False
        keys = keys[keep]
    return keys


def _rmat_keys(scale, g, rename):
    def keys_of(count):
        r = torch.zeros(count, dtype=torch.int64, device=DEV)
        c = torch.zeros(count, dtype=torch.int64, device=DEV)
        for _ in range(scale):                  # quadrant probabilities 0.57, 0.19, 0.19, 0.05 at every level
            u = torch.rand(count, generator=g, device=DEV)
            r = 2 * r + (u >= 0.76)
            c = 2 * c + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
        if rename is not None:
            r, c = rename[r], rename[c]
        return (r << scale) + c
    return keys_of


def _pattern(c, g):
    """(row of every nonzero or None, row_ptr or None, col_idx), rows ascending and columns ascending in a row."""
    m, n, nnz = c["m"], c["n"], _nnz(c)
    if c["matrix"] == "uniform":
        col = torch.randint(0, n, (m, c["per_row"]), generator=g, device=DEV, dtype=torch.int32).sort(dim=1).values.reshape(-1)
        return None, torch.arange(m + 1, device=DEV, dtype=torch.int64) * c["per_row"], col
    if c["matrix"] == "scatter":
        keys = _distinct(lambda q: torch.randint(0, m * n, (q,), generator=g, device=DEV), nnz, g)
        return keys // n, None, keys % n
    if c["matrix"] == "rmat":
        scale = m.bit_length() - 1
        rename = torch.randperm(m, generator=g, device=DEV) if c["relabel"] else None
        keys = _distinct(_rmat_keys(scale, g, rename), nnz, g)
        return keys >> scale, None, keys & (m - 1)
    if c["matrix"] == "skewed":
        w = torch.randn(m, generator=g, device=DEV, dtype=torch.float64).mul_(0.9).exp_()
        ends = (w.cumsum(0) * (nnz / float(w.sum()))).round().long()
        ends[-1] = nnz
        row_ptr = torch.cat((ends.new_zeros(1), ends))
        row = torch.repeat_interleave(torch.arange(m, device=DEV), row_ptr.diff(), output_size=nnz)
        keys = (row * n + torch.randint(0, n, (nnz,), generator=g, device=DEV)).sort().values
        return None, row_ptr, keys % n
    # grids: every cell's neighbours in row-major order, those outside the grid dropped
    dims = 2 if c["matrix"] == "grid5" else 3
    side = round(m ** (1 / dims))
    cell = torch.arange(m, device=DEV)
    at = [(cell // side ** (dims - 1 - d)) % side for d in range(dims)]
    steps = [(-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)] if dims == 2 else [(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1)]
    col = torch.empty(m, len(steps), device=DEV, dtype=torch.int32)
    for j, s in enumerate(steps):
        inside = torch.ones(m, dtype=torch.bool, device=DEV)
        to = torch.zeros_like(cell)
        for d in range(dims):
            inside &= (at[d] + s[d] >= 0) & (at[d] + s[d] < side)
            to = to * side + at[d] + s[d]
        col[:, j] = torch.where(inside, to, -1).int()
    lens = (col >= 0).sum(1)
    col = col.reshape(-1)
    return None, torch.cat((lens.new_zeros(1), lens.cumsum(0))), col[col >= 0]


def _values(c, row_ptr, col, g):
    nnz = col.numel()
    if c["matrix"] in ("grid5", "stencil27"):   # the operator: the diagonal, and the off-diagonals (perturbed in 3-D)
        diag, spread = (4.0, 0.0) if c["matrix"] == "grid5" else (26.0, 0.01)
        off = torch.randn(nnz, generator=g, device=DEV).mul_(spread).sub_(1.0)
        row = torch.repeat_interleave(torch.arange(c["m"], device=DEV, dtype=torch.int32), row_ptr.diff(), output_size=nnz)
        return torch.where(row == col, torch.full_like(off, diag), off)
    if c["matrix"] == "rmat":                   # edge weights in (0, 1]
        return 1.0 - torch.rand(nnz, generator=g, device=DEV)
    return torch.randn(nnz, generator=g, device=DEV)


def _stored(t, dtype):
    """FP32, or the 16-bit patterns of BF16 that the library takes."""
    return t if dtype == "f32" else t.to(torch.bfloat16).view(torch.int16)


class _Cached:
    """Forgets what the library keeps for an array's address before the array goes away, as its users have to."""

    def __init__(self, key, everything=False):
        self.key, self.everything = key, everything

    def __del__(self):
        if self.everything:                     # a CSC pattern: the plan of its row-major copy is cached under an address of the library's own
            b200sp.b200sp_cache_clear()
        else:
            b200sp.b200sp_cache_drop(self.key)


def prepare(case, seed):
    c = dict(case)
    m, n, k, dtype = c["m"], c["n"], c["k"], c["dtype"]
    g = torch.Generator(DEV).manual_seed(seed)
    row, row_ptr, col = _pattern(c, g)
    if row_ptr is None:
        row_ptr = torch.searchsorted(row, torch.arange(m + 1, device=DEV))
    col = col.int()
    vals = _values(c, row_ptr, col, g)
    s = {"c": c, "nnz": col.numel()}
    if c["op"] == "spmv_csc":                   # the same entries by columns
        if row is None:
            row = torch.repeat_interleave(torch.arange(m, device=DEV), row_ptr.diff(), output_size=col.numel())
        order = (col.long() * m + row).sort().indices
        ends = torch.searchsorted(col[order].contiguous(), torch.arange(n + 1, device=DEV, dtype=torch.int32))
        s["ptr"], s["idx"], s["vals"] = ends.int(), row[order].int(), _stored(vals[order], dtype)
    else:
        s["ptr"], s["idx"], s["vals"] = row_ptr.int(), col, _stored(vals, dtype)
    if k == 1:
        x = torch.rand(n, generator=g, device=DEV).mul_(2).sub_(1) if c["matrix"] != "rmat" else 1.0 - torch.rand(n, generator=g, device=DEV)
    else:
        x = torch.randn(n * k, generator=g, device=DEV)
    s["x"] = _stored(x, dtype)
    s["y"] = _stored(torch.rand(m * k, generator=g, device=DEV).mul_(2).sub_(1), dtype)
    s["out"] = s["y"].view(torch.bfloat16).view(m, k) if dtype == "bf16" else s["y"].view(m, k)
    if c["op"] != "spmm_fresh":
        s["cached"] = _Cached(s["ptr"], everything=c["op"] == "spmv_csc")
    return s


def run(s):
    c = s["c"]
    m, n, k, nnz, alpha, beta, dtype = c["m"], c["n"], c["k"], s["nnz"], c["alpha"], c["beta"], c["dtype"]
    if c["op"] == "spmv":
        b200sp.spmv_csr(m, n, nnz, s["ptr"], s["idx"], s["vals"], s["x"], s["y"], alpha, beta, dtype)
    elif c["op"] == "spmv_csc":
        b200sp.spmv_csc(m, n, nnz, s["ptr"], s["idx"], s["vals"], s["x"], s["y"], alpha, beta, dtype)
    elif c["op"] == "spmm":
        b200sp.spmm_csr(m, n, nnz, k, s["ptr"], s["idx"], s["vals"], s["x"], s["y"], alpha, beta, dtype)
    else:
        plan = b200sp.b200sp_plan_create(m, n, nnz, s["ptr"])
        b200sp.b200sp_spmm(plan, k, s["idx"], s["vals"], s["x"], s["y"], alpha, beta, dtype)
        b200sp.b200sp_plan_destroy(plan)
    return s["out"]


def work(case):
    m, n, k, nnz = case["m"], case["n"], case["k"], _nnz(case)
    e = 4 if case["dtype"] == "f32" else 2
    ptr = (n if case["op"] == "spmv_csc" else m) + 1
    passes_over_y = 2 if case["beta"] else 1
    return {"bytes": nnz * (4 + e) + 4 * ptr + n * k * e + passes_over_y * m * k * e, "flops": 2 * nnz * k}


def tolerance(case):
    # Four times the distance from the product in 64 bits: FP32 sums 1.5e-7 (single entries that cancel 1.3e-5), BF16 storage
    # 1.7e-3 (3.9e-3), the one rounding of the result to eight bits.
    return {"rel": 6e-7, "max": 5.2e-5} if case["dtype"] == "f32" else {"rel": 6.8e-3, "max": 1.6e-2}
