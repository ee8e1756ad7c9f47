"""What a user of the SpGEMM library has it do, as measurable cases: C = A * B for CSR matrices in device memory (one
call, or the execute of a plan that is kept), the same through the host-buffer entry point, and the row analysis that
allocates nothing.  Matrices follow the recipes of the gen package, drawn with torch on the GPU.

Matrix kinds
  er      every row holds exactly `k` distinct uniform columns (no heavy row: the light path alone)
  grid    5-point stencil with varying coefficients on a `side` x `side` grid
  rmat    R-MAT graph of 2**scale vertices and ef * 2**scale edge draws, (0.57, 0.19, 0.19, 0.05), merged
  zipf    A (n x 4n) times B (4n x 16n), row lengths clipped Zipf: very short rows, a very wide C
  block   block rows coupling to 6 block columns with dense blocks (most rows heavy, a narrow column space)
All but zipf are squared (A * A).

Calls
  product       plan + execute + release, as one call: a product of matrices not met before
  execute       a plan is kept and executed: same structure, values that change (re-assembly, iteration)
  host          A, B and C in pinned host memory, copies included
  row_products  intermediate products per row of A * A, without any allocation
"""
import math
from types import SimpleNamespace

import torch

import paper_2607_22866_b200 as gm

QUADRANTS = (0.57, 0.19, 0.19, 0.05)
ZIPF_A, ZIPF_B = (1.8, 4096), (2.0, 2048)  # exponent and longest row
BLOCK_FILL, BLOCK_DENSE, BLOCKS_PER_ROW = 0.7, 0.7, 6


def listed():
    return [
        # the smallest call: a matrix of a few thousand entries, nothing but latency
        {"name": "er 1000 f32", "kind": "er", "n": 1000, "k": 5, "dtype": "f32", "call": "product"},
        # the benchmark's smallest workload
        {"name": "er 4096 f32", "kind": "er", "n": 4096, "k": 8, "dtype": "f32", "call": "product"},
        # a sparse operator squared again and again with new values
        {"name": "er 30011 f64 kept plan", "kind": "er", "n": 30011, "k": 12, "dtype": "f64", "call": "execute"},
        # a discretised operator squared (the benchmark's workload): a million short rows
        {"name": "grid 1024 f64", "kind": "grid", "side": 1024, "dtype": "f64", "call": "product"},
        # a small power-law graph: light and heavy rows, a single chunk per row
        {"name": "rmat 12 f32", "kind": "rmat", "scale": 12, "ef": 16, "dtype": "f32", "call": "product"},
        # an ordinary one, its structure planned once
        {"name": "rmat 15 f32 kept plan", "kind": "rmat", "scale": 15, "ef": 16, "dtype": "f32", "call": "execute"},
        # double precision, several chunks per row
        {"name": "rmat 17 f64", "kind": "rmat", "scale": 17, "ef": 8, "dtype": "f64", "call": "product"},
        # the largest: the benchmark's graph at half its vertices (its C at full size, 78 GB, does not fit twice)
        {"name": "rmat 19 f32", "kind": "rmat", "scale": 19, "ef": 16, "dtype": "f32", "call": "product"},
        # a rectangular pair of web-like matrices (the benchmark's workload): two multisplit levels
        {"name": "zipf 1048576 f32", "kind": "zipf", "n": 1048576, "dtype": "f32", "call": "product"},
        # structural and power-network matrices (the benchmark's workload): forty products per entry of C
        {"name": "block 1024x64 f32", "kind": "block", "blocks": 1024, "block": 64, "dtype": "f32", "call": "product"},
        # matrices that live on the host
        {"name": "rmat 13 f32 host", "kind": "rmat", "scale": 13, "ef": 8, "dtype": "f32", "call": "host"},
        # sizing a product before it is made, where the library must not allocate
        {"name": "rmat 15 row products", "kind": "rmat", "scale": 15, "ef": 16, "dtype": "f32", "call": "row_products"},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["product", "product", "product", "execute", "execute", "host", "row_products"])
    # (the row analysis of an er or a grid matrix has the same answer whatever the numbering: not drawn)
    kind = rng.choice(["rmat", "rmat", "zipf", "block"] if call == "row_products" else ["er", "grid", "rmat", "rmat", "zipf", "block"])
    case = {"kind": kind, "dtype": rng.choice(["f32", "f64"]), "call": call}
    # kept plans are moderate (several are kept at a time), C on the host is tens of megabytes, and the row analysis
    # without allocation takes at most 2**20 entries of A
    if kind == "er":
        case["n"] = log_int(200, 20000 if call == "host" else 200000)
        case["k"] = rng.randint(2, 16)
    elif kind == "grid":
        case["side"] = log_int(24, 400 if call == "host" else 1024)
    elif kind == "rmat":
        case["scale"] = rng.randint(10, {"product": 18, "execute": 16, "host": 13, "row_products": 16}[call])
        case["ef"] = rng.randint(4, 15)
    elif kind == "zipf":
        case["n"] = log_int(1 << 12, {"product": 1 << 20, "execute": 1 << 19, "host": 1 << 16, "row_products": 1 << 17}[call])
    else:
        case["block"] = rng.randint(17, 64)
        case["blocks"] = log_int(24, {"product": 1000, "execute": 400, "host": 60, "row_products": 80}[call])
    return case


# ---------------------------------------------------------------------------------------------------------------------
# inputs
#
# The structure belongs to the case, up to the numbering of its rows and columns; numbering and values come from the
# seed.  The renumberings keep the recipe's distribution: any permutation (er, zipf), a permutation of the bits of the
# vertex numbers (rmat), a rotation of the block rows (block), none (grid).
# ---------------------------------------------------------------------------------------------------------------------
def _csr(rows, cols, n_rows, n_cols, dtype, g):
    """rows, cols: distinct pairs in any order."""
    key = torch.sort(rows * n_cols + cols).values
    row_ptr = torch.searchsorted(key, torch.arange(n_rows + 1, device="cuda") * n_cols)
    val = torch.rand(key.numel(), generator=g, device="cuda", dtype=dtype) * 2 - 1
    return gm.DeviceCSR(n_rows, n_cols, row_ptr, (key % n_cols).to(torch.int32), val)


def _distinct_columns(lengths, n_cols, s):
    """Rows of the given lengths with distinct uniform columns."""
    rows = torch.repeat_interleave(torch.arange(lengths.numel(), device="cuda"), lengths)
    cols = torch.randint(n_cols, (rows.numel(),), generator=s, device="cuda")
    while True:
        cols = torch.sort(rows * n_cols + cols).values - rows * n_cols
        again = torch.nonzero((cols[1:] == cols[:-1]) & (rows[1:] == rows[:-1])).flatten() + 1
        if not again.numel():
            return rows, cols
        cols[again] = torch.randint(n_cols, (again.numel(),), generator=s, device="cuda")


def _zipf_cdf(exponent, cap):
    zeta = sum(k ** -exponent for k in range(1, 10000)) + 10000.0 ** (1 - exponent) / (exponent - 1) + 0.5 * 10000.0 ** -exponent
    cdf = torch.cumsum(torch.arange(1, cap + 1, dtype=torch.float64) ** -exponent, 0) / zeta
    cdf[-1] = 1.0  # the longest row stands for the whole tail
    return cdf


def _zipf_rows(n_rows, n_cols, exponent, cap, s):
    u = torch.rand(n_rows, generator=s, device="cuda", dtype=torch.float64)
    lengths = torch.searchsorted(_zipf_cdf(exponent, cap).cuda(), u, right=True) + 1
    return _distinct_columns(torch.clamp(lengths, max=min(cap, n_cols)), n_cols, s)


def _grid(side):
    p = torch.arange(side * side, device="cuda")
    x, y = p % side, p // side
    keep = torch.stack([y > 0, x > 0, x >= 0, x < side - 1, y < side - 1], 1)
    cols = p[:, None] + torch.tensor([-side, -1, 0, 1, side], device="cuda")
    return p[:, None].expand(side * side, 5)[keep], cols[keep]


def _rmat(scale, ef, s, g):
    a, b, c, _ = QUADRANTS
    n = 1 << scale
    rows = torch.zeros(ef * n, dtype=torch.int64, device="cuda")
    cols = torch.zeros_like(rows)
    for _ in range(scale):
        u = torch.rand(rows.numel(), generator=s, device="cuda")
        rows = rows * 2 + (u >= a + b)
        cols = cols * 2 + (((u >= a) & (u < a + b)) | (u >= a + b + c))
    key = torch.unique(rows * n + cols)
    bits = torch.arange(scale, device="cuda")
    number = ((torch.arange(n, device="cuda")[:, None] >> bits & 1) << torch.randperm(scale, generator=g, device="cuda")).sum(1)
    return number[key // n], number[key % n]


def _block(blocks, block, s, g):
    n = blocks * block
    own = torch.arange(blocks, device="cuda")
    dense = torch.rand(blocks, generator=s, device="cuda") < BLOCK_DENSE
    far = torch.randint(blocks, (blocks, BLOCKS_PER_ROW - 3), generator=s, device="cuda")
    choice = torch.cat([torch.stack([own, (own + 1) % blocks, (own - 1) % blocks], 1), far], 1)
    inner = torch.arange(block, device="cuda")
    keys = []
    for j in range(BLOCKS_PER_ROW):  # coupled blocks of the dense block rows
        rows, cols = own[dense] * block, choice[dense, j] * block
        key = (rows[:, None] + inner)[:, :, None] * n + (cols[:, None] + inner)[:, None, :]
        keys.append(key[torch.rand(key.shape, generator=s, device="cuda") < BLOCK_FILL])
    first = own[~dense] * block  # the other block rows: the diagonal and about two entries of the diagonal block
    key = (first[:, None] + inner)[:, :, None] * n + (first[:, None] + inner)[:, None, :]
    keep = torch.rand(key.shape, generator=s, device="cuda") < 2.0 / block
    keys.append(key[keep | torch.eye(block, dtype=torch.bool, device="cuda")])
    key = torch.unique(torch.cat(keys))
    turn = torch.randint(blocks, (1,), generator=g, device="cuda") * block
    return (key // n + turn) % n, (key % n + turn) % n


def _matrices(case, seed):
    s = torch.Generator(device="cuda").manual_seed(20)
    g = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.float32 if case["dtype"] == "f32" else torch.float64
    kind = case["kind"]
    if kind == "zipf":
        n = case["n"]
        outer, middle, inner = (torch.randperm(k * n, generator=g, device="cuda") for k in (1, 4, 16))
        rows, cols = _zipf_rows(n, 4 * n, *ZIPF_A, s)
        A = _csr(outer[rows], middle[cols], n, 4 * n, dtype, g)
        rows, cols = _zipf_rows(4 * n, 16 * n, *ZIPF_B, s)
        return A, _csr(middle[rows], inner[cols], 4 * n, 16 * n, dtype, g)
    if kind == "er":
        n = case["n"]
        number = torch.randperm(n, generator=g, device="cuda")
        rows, cols = _distinct_columns(torch.full((n,), case["k"], device="cuda"), n, s)
        rows, cols = number[rows], number[cols]
    elif kind == "grid":
        n = case["side"] ** 2
        rows, cols = _grid(case["side"])
    elif kind == "rmat":
        n = 1 << case["scale"]
        rows, cols = _rmat(case["scale"], case["ef"], s, g)
    else:
        n = case["blocks"] * case["block"]
        rows, cols = _block(case["blocks"], case["block"], s, g)
    A = _csr(rows, cols, n, n, dtype, g)
    return A, A


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()


def _on_host(M):
    return SimpleNamespace(n_rows=M.n_rows, n_cols=M.n_cols, row_ptr=_pinned(M.row_ptr), col=_pinned(M.col), val=_pinned(M.val))


def prepare(case, seed):
    A, B = _matrices(case, seed)
    state = {"call": case["call"], "A": A, "B": B}
    if case["call"] == "execute":
        state["plan"] = gm.spgemm_plan(A, B)
    elif case["call"] == "row_products":
        state["out"] = torch.empty(A.n_rows, dtype=torch.int64, device="cuda")
    elif case["call"] == "host":
        # room for C: no row has more entries than products, or than columns
        lengths = B.row_ptr[1:] - B.row_ptr[:-1]
        before = torch.zeros(A.nnz + 1, dtype=torch.int64, device="cuda")
        before[1:] = torch.cumsum(lengths[A.col.long()], 0)
        products = before[A.row_ptr[1:]] - before[A.row_ptr[:-1]]
        room = int(torch.clamp(products, max=B.n_cols).sum())
        hA = _on_host(A)
        hB = hA if B is A else _on_host(B)
        state = {"call": "host", "A": hA, "B": hB, "row_ptr": torch.empty(A.n_rows + 1, dtype=torch.int64, pin_memory=True).numpy(),
                 "col": torch.empty(room, dtype=torch.int32, pin_memory=True).numpy(),
                 "val": torch.empty(room, dtype=A.val.dtype, pin_memory=True).numpy()}
    return state


def run(state):
    call = state["call"]
    if call == "row_products":
        return gm.row_products_noalloc(state["A"], state["B"], state["out"])
    if call == "host":
        nnz = gm.spgemm_host(state["A"], state["B"], state["row_ptr"], state["col"], state["val"])
        return {"row_ptr": state["row_ptr"], "col": state["col"][:nnz], "val": state["val"][:nnz]}
    if call == "execute":
        C = gm.spgemm_execute(state["plan"])
    else:
        C, _, _ = gm.spgemm(state["A"], state["B"])
    return {"row_ptr": C.row_ptr, "col": C.col, "val": C.val}


# ---------------------------------------------------------------------------------------------------------------------
# work: expected sizes of the random matrices
# ---------------------------------------------------------------------------------------------------------------------
def _hit(x):
    return -math.expm1(-x)  # chance of at least one of x expected events


def _rmat_sizes(scale, ef):
    """Entries of A, products of A * A and entries of C.  Vertices with the same number w of one bits share
    their degree; cells of A (of A * A) with the same mix of quadrant picks (of pairs of picks) share their probability."""
    a, b, c, d = QUADRANTS
    draws = ef * 2.0 ** scale

    def cells(w, qa, qb, qc, qd, events):  # expected occupied cells of a row with w one bits
        z = scale - w
        return sum(math.comb(z, i) * math.comb(w, j) * _hit(events * qa ** i * qb ** (z - i) * qc ** j * qd ** (w - j))
                   for i in range(z + 1) for j in range(w + 1))

    # a pair of picks: row bit of the first, column bit of the second, any bit in between
    pair = (a * a + b * c, a * b + b * d, c * a + d * c, c * b + d * d)
    degree = [cells(w, a, b, c, d, draws) for w in range(scale + 1)]
    nnz = sum(math.comb(scale, w) * degree[w] for w in range(scale + 1))
    products = sum(math.comb(scale, w) * degree[w] ** 2 for w in range(scale + 1))  # (b = c: columns have the degrees of rows)
    # merging the draws takes products away, most of them from entries of C that have others: the cube root of what is
    # left comes within 5 % of the entries counted on generated graphs (scales 12 to 21)
    events = draws * draws * (products / (draws * draws * sum(pair) ** scale)) ** (1 / 3)
    return nnz, products, sum(math.comb(scale, w) * cells(w, *pair, events) for w in range(scale + 1))


def _sizes(case):
    """(rows of A, rows of B, entries of A, of B, products, entries of C); B counts nothing where it is A."""
    kind = case["kind"]
    if kind == "er":
        n, k = case["n"], min(case["k"], case["n"])
        return n, 0, n * k, 0, n * k * k, n * n * _hit(k * k / n)
    if kind == "grid":
        s = case["side"]
        n = s * s
        return n, 0, 5 * n - 4 * s, 0, 25 * n - 44 * s + 8, 13 * n - 20 * s + 4
    if kind == "rmat":
        nnz, products, nnz_c = _rmat_sizes(case["scale"], case["ef"])
        return 1 << case["scale"], 0, nnz, 0, products, nnz_c
    if kind == "zipf":
        n = case["n"]
        mean_a, mean_b = (float((1 - _zipf_cdf(s, cap)[:-1]).sum()) + 1 for s, cap in (ZIPF_A, ZIPF_B))
        return n, 4 * n, n * mean_a, 4 * n * mean_b, n * mean_a * mean_b, n * mean_a * mean_b
    n, block = case["blocks"] * case["block"], case["block"]
    apart = case["blocks"] * _hit(BLOCKS_PER_ROW / case["blocks"])  # block columns that do not fall together
    heavy = BLOCK_FILL * block * apart
    mean = BLOCK_DENSE * heavy + (1 - BLOCK_DENSE) * 3
    # a dense block row reaches its own 6 block columns, and through each dense one of them 4 or 6 more
    reach = case["blocks"] * _hit((6 + 2 * BLOCK_DENSE * 4 + 3 * BLOCK_DENSE * 6) / case["blocks"])
    return n, 0, n * mean, 0, n * (BLOCK_DENSE * heavy * mean + (1 - BLOCK_DENSE) * 9), n * (BLOCK_DENSE * reach * block + (1 - BLOCK_DENSE) * 6)


def work(case):
    n_a, n_b, nnz_a, nnz_b, products, nnz_c = _sizes(case)
    entry = 8 if case["dtype"] == "f32" else 12
    if case["call"] == "row_products":
        rows = n_a + n_b + 1
        return {"bytes": 4 * nnz_a + 8 * rows + 8 * n_a, "flops": 0}
    return {"bytes": entry * (nnz_a + nnz_b + nnz_c) + 8 * (2 * n_a + n_b + 3), "flops": 2 * products}


def tolerance(case):
    if case["call"] == "row_products":
        return "exact"
    # Products of one entry of C are summed in any order.  A hub's entry sums tens of thousands of products of either
    # sign, so a single entry can be off by more than the whole.
    return {"rel": 2e-6, "max": 1e-4} if case["dtype"] == "f32" else {"rel": 1e-14, "max": 5e-13}
