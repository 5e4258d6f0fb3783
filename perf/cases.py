"""Performance cases: the iterated arrow-SpMM as a program calls it, over the range it is used on.

A case is one call of a public entry point (``ArrowMatrix.spmm``, ``ArrowBatch.spmm``, or a burst of
``ArrowServer`` requests) on matrices whose decomposition the program keeps.  The matrices are the
four families of ``workloads/`` (2D and 3D grid stencils, random-geometric graphs, GCN-normalised
R-MAT graphs), generated here on the GPU so that preparing a case is quick; values are rounded to
the type the device stores, so that a 64-bit product has the same matrix.
"""
import math

import numpy as np
import torch

import paper_2402_19364_gb300 as arrow

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_SIZE = {"f32": 4, "bf16": 2, "f16": 2}
# seeds of the matrices and the features of one state
_A_SEED, _X_SEED = 1_000_003, 7_000_009


# ---- matrices ------------------------------------------------------------------------------------
class Csr:
    """Host CSR as ``ArrowMatrix`` takes it, and the same matrix on the GPU (for the 64-bit product)."""

    def __init__(self, n, rowptr, col, val, store, keep_device):
        val = val.to(_TORCH[store]).double()
        self.n = n
        self.device = (rowptr, col, val) if keep_device else None
        self.rowptr = rowptr.cpu().numpy()
        self.colidx = col.to(torch.int32).cpu().numpy()
        self.values = val.cpu().numpy()


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _rows(rowptr):
    n = rowptr.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device="cuda"), rowptr[1:] - rowptr[:-1])


def _pointers(r, n):
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(r, minlength=n), 0, out=rowptr[1:])
    return rowptr


def _row_normalised(rowptr, g):
    """U(0.5, 1.5) values, every row divided by its sum."""
    val = 0.5 + torch.rand(int(rowptr[-1]), generator=g, device="cuda", dtype=torch.float64)
    r = _rows(rowptr)
    sums = torch.zeros(rowptr.numel() - 1, dtype=torch.float64, device="cuda").index_add_(0, r, val)
    return val / sums[r]


def _grid(dims, g):
    """5- or 7-point stencil with its diagonal; row-major vertex ids."""
    n = math.prod(dims)
    v = torch.arange(n, device="cuda")
    cand, ok, stride = [], [], n
    for d in dims:                     # ascending columns: -s0, -s1, ..., 0, ..., +s1, +s0
        stride //= d
        c = (v // stride) % d
        cand.append((v - stride, c > 0))
        ok.append((v + stride, c < d - 1))
    both = cand + [(v, torch.ones_like(v, dtype=torch.bool))] + ok[::-1]
    mask = torch.stack([m for _, m in both], 1)
    col = torch.stack([c for c, _ in both], 1)[mask]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(mask.sum(1), 0, out=rowptr[1:])
    return n, rowptr, col, _row_normalised(rowptr, g)


def _from_pairs(n, r, c):
    ar = torch.arange(n, device="cuda")
    key = torch.unique(torch.cat([r * n + c, c * n + r, ar * n + ar]))
    r, c = key // n, key % n
    return _pointers(r, n), c


def _rgg(n, g):
    """n points in the unit square, edge below the distance of a mean degree of 8, self-loops."""
    radius = math.sqrt(8.0 / (math.pi * n))
    side = max(1, int(1.0 / radius))
    pts = torch.rand(n, 2, generator=g, device="cuda", dtype=torch.float64)
    cell = (pts * side).long().clamp_(max=side - 1)
    order = torch.argsort(cell[:, 0] * side + cell[:, 1], stable=True)
    first = _pointers((cell[:, 0] * side + cell[:, 1]), side * side)
    rs, cs = [], []
    v = torch.arange(n, device="cuda")
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            x, y = cell[:, 0] + dx, cell[:, 1] + dy
            inside = (x >= 0) & (x < side) & (y >= 0) & (y < side)
            q = torch.where(inside, x * side + y, 0)
            cnt = torch.where(inside, first[q + 1] - first[q], 0)
            a = torch.repeat_interleave(v, cnt)
            off = torch.arange(a.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
            b = order[first[q[a]] + off]
            near = ((pts[a] - pts[b]).square().sum(1) < radius * radius) & (a < b)
            rs.append(a[near])
            cs.append(b[near])
    rowptr, col = _from_pairs(n, torch.cat(rs), torch.cat(cs))
    return n, rowptr, col, _row_normalised(rowptr, g)


def _rmat(scale, g):
    """R-MAT (0.57, 0.19, 0.19, 0.05), edge factor 16, symmetrised, D^-1/2 (A + I) D^-1/2."""
    n = 1 << scale
    u = torch.zeros(16 * n, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(scale):
        t = torch.rand(16 * n, generator=g, device="cuda")
        u = 2 * u + (t >= 0.76)
        v = 2 * v + (((t >= 0.57) & (t < 0.76)) | (t >= 0.95))
    keep = u != v
    rowptr, col = _from_pairs(n, u[keep], v[keep])
    rs = (rowptr[1:] - rowptr[:-1]).double().rsqrt()
    return n, rowptr, col, rs[_rows(rowptr)] * rs[col]


def _matrix(graph, size, store, seed, keep_device=False):
    g = _gen(seed)
    if graph == "grid":
        n, rowptr, col, val = _grid([int(d) for d in str(size).split("x")], g)
    elif graph == "rgg":
        n, rowptr, col, val = _rgg(int(size), g)
    else:
        n, rowptr, col, val = _rmat(int(size), g)
    return Csr(n, rowptr, col, val, store, keep_device)


def _features(n, k, dtype, seed):
    return torch.randn(n, k, generator=_gen(seed), device="cuda", dtype=torch.float32).to(_TORCH[dtype])


def _rows_and_entries(graph, size):
    """n and the (expected) number of entries of a matrix, for the work of a case."""
    if graph == "grid":
        dims = [int(d) for d in str(size).split("x")]
        n = math.prod(dims)
        return n, n + sum(2 * (n - n // d) for d in dims)
    if graph == "rgg":
        return int(size), 9 * int(size)
    n = 1 << int(size)
    return n, int(n * (31.4 - 3.0 * 0.83 ** (int(size) - 16)))


# ---- cases ---------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the 64 x 64 grid of the latency configuration, as the quick start calls it
        dict(name="grid2d_64", kind="spmm", graph="grid", size="64x64", b=64, k=16, v="f32", x="f32", iters=10),
        # a small power iteration by a program that autotunes first (a ragged grid, narrow features)
        dict(name="small_tuned_rescale", kind="spmm", graph="grid", size="83x61", b=64, k=8, v="f32", x="f32", iters=20,
             rescale=True, autotune=True),
        # one graph-network layer: a single product with the rectifier, 16-bit features on 32-bit values
        dict(name="layer_rgg_bf16", kind="spmm", graph="rgg", size=300007, b=548, k=64, v="f32", x="bf16", iters=1, relu=True),
        # the quick start: 100^3 grid, 20 iterations of the FP64-normalised power iteration
        dict(name="grid3d_100_rescale", kind="spmm", graph="grid", size="100x100x100", b=4096, k=16, v="f32", x="f32",
             iters=20, rescale=True),
        # the headline workload one size down (inputs far larger than L2), autotuned as the benchmark does
        dict(name="grid3d_200_rescale", kind="spmm", graph="grid", size="200x200x200", b=4096, k=16, v="f32", x="f32",
             iters=20, rescale=True, autotune=True),
        # power-law graph, wide BF16 features: hub rows split into segments (GCN propagation)
        dict(name="rmat_20_bf16", kind="spmm", graph="rmat", size=20, b=8192, k=128, v="bf16", x="bf16", iters=8),
        # the same in FP32 at a size that L2 holds, with both fused parts of sigma
        dict(name="rmat_16_f32_sigma", kind="spmm", graph="rmat", size=16, b=1024, k=64, v="f32", x="f32", iters=3, relu=True,
             rownorm=True),
        # mesh-like graph in FP16 under the band predicate, an odd number of rows
        dict(name="rgg_f16_band", kind="spmm", graph="rgg", size=1000003, b=1001, k=32, v="f16", x="f16", iters=10, band=True),
        # features wider than one chunk of columns, on a ragged 2D grid
        dict(name="grid2d_wide", kind="spmm", graph="grid", size="317x211", b=256, k=256, v="f32", x="f32", iters=5),
        # many random-geometric graphs of mixed sizes and widths in FP16, replayed as one CUDA graph
        dict(name="batch_rgg_f16", kind="batch", count=24, lo=1000, hi=1000000, kmax=64, v="f16", x="f16", iters=10, graph=True),
        # a batch of small FP32 problems without a graph (new outputs on every call)
        dict(name="batch_small_f32", kind="batch", count=40, lo=300, hi=6000, kmax=32, v="f32", x="f32", iters=10, graph=False),
        # a burst of requests on a continuous-batching server, grids, meshes and power-law graphs mixed
        dict(name="serve_bf16", kind="serve", count=16, lo=10000, hi=250000, kmax=128, v="bf16", x="bf16", iters=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmm", "spmm", "spmm", "batch", "serve"])
    v, x = rng.choice([("f32", "f32"), ("f32", "f32"), ("bf16", "bf16"), ("f16", "f16"), ("f32", "bf16")])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 40), lo=300, hi=_log_int(rng, 3000, 400000), kmax=64, v=v, x=x,
                    iters=rng.randint(1, 10), graph=rng.random() < 0.5)
    if kind == "serve":
        return dict(kind="serve", count=rng.randint(3, 16), lo=2000, hi=_log_int(rng, 5000, 250000), kmax=128, v=v, x=x,
                    iters=rng.randint(2, 12))
    graph = rng.choice(["grid2", "grid3", "rgg", "rmat"])
    if graph == "grid2":
        size = "x".join(str(_log_int(rng, 20, 1500)) for _ in range(2))
    elif graph == "grid3":
        size = "x".join(str(_log_int(rng, 8, 150)) for _ in range(3))
    elif graph == "rgg":
        size = _log_int(rng, 1000, 1000000)
    else:
        size = rng.randint(11, 19)
    vec = 4 if x == "f32" else 8
    n, _ = _rows_and_entries("grid" if graph.startswith("grid") else graph, size)
    k = vec * rng.choice([1, 2, 4, 4, 8, 16, 32, 64] if n < 500000 else [1, 2, 4, 4, 8, 16])
    case = dict(kind="spmm", graph="grid" if graph.startswith("grid") else graph, size=size, b=max(16, math.isqrt(n)), k=k, v=v,
                x=x, iters=rng.choice([1, 2, 3, 5, 10, 20]))
    if rng.random() < 0.3:
        case["rescale"] = True
    if rng.random() < 0.3:
        case["relu"] = True
    if rng.random() < 0.2 and k // vec <= 32:
        case["rownorm"] = True
    if rng.random() < 0.2:
        case["band"] = True
    return case


# ---- members of a batch, requests of a burst -----------------------------------------------------
def _members(case):
    """(graph, size, b, k, iters) of every problem of a case; fixed by the case, not by the seed."""
    if case["kind"] == "spmm":
        return [(case["graph"], case["size"], case["b"], case["k"], case["iters"])]
    rng = np.random.default_rng(case["count"] * 1009 + case["hi"])
    vec = 16 // _SIZE[case["x"]]
    ks = [k for k in (8, 16, 32, 64, 128) if vec <= k <= case["kmax"]]
    out = []
    for i in range(case["count"]):
        n = int(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))
        k = int(rng.choice(ks))
        if case["kind"] == "batch":
            out.append(("rgg", n, math.isqrt(n) + 1, k, case["iters"]))
            continue
        graph, size = [("rgg", n), ("grid", f"{math.isqrt(n)}x{math.isqrt(n) + 1}"),
                       ("rmat", max(8, int(math.log2(n)) - 2))][i % 3]
        out.append((graph, size, math.isqrt(n) + 1, k, int(rng.integers(2, case["iters"] + 1))))
    return out


def prepare(case, seed):
    members = _members(case)
    mats, xs = [], []
    for i, (graph, size, b, k, _) in enumerate(members):
        a = _matrix(graph, size, case["v"], seed * _A_SEED + i)
        mats.append(arrow.ArrowMatrix(a, b, value_dtype=case["v"], predicate="band" if case.get("band") else "block"))
        xs.append(_features(a.n, k, case["x"], seed * _X_SEED + i))
    state = dict(case=case, mats=mats, xs=xs, iters=[m[4] for m in members])
    if case["kind"] == "spmm":
        if case.get("autotune"):
            mats[0].autotune(xs[0], case["iters"], rescale=bool(case.get("rescale")))
    elif case["kind"] == "batch":
        state["batch"] = arrow.ArrowBatch(mats)
        state["outs"] = [torch.empty_like(x) for x in xs] if case["graph"] else None
    else:
        state["outs"] = [torch.empty_like(x) for x in xs]
        state["server"] = arrow.ArrowServer(2 << 30, 64, x_dtype=case["x"])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "spmm":
        return state["mats"][0].spmm(state["xs"][0], case["iters"], rescale=bool(case.get("rescale")),
                                     relu=bool(case.get("relu")), rownorm=bool(case.get("rownorm")))
    if case["kind"] == "batch":
        return state["batch"].spmm(state["xs"], case["iters"], outs=state["outs"], graph=case["graph"])
    server = state["server"]
    for m, x, y, it in zip(state["mats"], state["xs"], state["outs"], state["iters"]):
        server.submit(m, x, y, it)
    server.drain()
    server.poll()
    return state["outs"]


def work(case):
    """Every iteration reads the matrix (value, column, row pointer) and its input and writes its
    output; the order of the features in between is the program's affair, so no permutation counts."""
    total, flops = 0, 0
    sv, sx = _SIZE[case["v"]], _SIZE[case["x"]]
    for graph, size, _, k, iters in _members(case):
        n, nnz = _rows_and_entries(graph, size)
        total += iters * (nnz * (sv + 4) + 4 * (n + 1) + 2 * n * k * sx)
        flops += iters * 2 * nnz * k
    return {"bytes": total, "flops": flops}


def exact(case, seed):
    """The same iteration with torch's sparse product in 64 bits, nothing rounded in between."""
    outs = []
    for i, (graph, size, _, k, iters) in enumerate(_members(case)):
        a = _matrix(graph, size, case["v"], seed * _A_SEED + i, keep_device=True)
        rowptr, col, val = a.device
        y = _features(a.n, k, case["x"], seed * _X_SEED + i).double()
        m = torch.sparse_csr_tensor(rowptr, col, val, (a.n, a.n), check_invariants=False)
        for _ in range(iters):
            y = m @ y
            if case.get("relu"):
                y = y.clamp_(min=0)
            if case.get("rownorm"):
                norm = y.norm(dim=1, keepdim=True)
                y = torch.where(norm > 0, y / norm, torch.zeros_like(y))
            if case.get("rescale"):
                norm = y.norm(dim=0, keepdim=True)
                y = torch.where(norm > 0, y / norm, y)
        outs.append(y)
        del m
    return outs[0] if case["kind"] == "spmm" else outs
