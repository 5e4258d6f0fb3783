"""GPU test of the length-ordered rows of a tile (row descriptors) at the sizes where their fields end.

Rows of 0 to 140 entries, unsplit (long_row 256): below, at and above the length the descriptor
holds itself (63), one tile of 2048 rows, tiles of 32 rows, and a last tile of one row.  Tolerances:
FP32 1e-5 per column against the FP64 oracle (a sum of at most 140 products with relative error
2^-24 each stays below 140 * 2^-24 = 8.4e-6 of the sum of magnitudes, and the values are positive).
"""
import numpy as np
import pytest

import workloads as w
from oracle import spmm as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def arrow():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_19364_gb300 import build
    build.build()
    import paper_2402_19364_gb300 as pkg
    return pkg


def _matrix(n):
    rng = np.random.default_rng(11)
    special = np.array([0, 1, 7, 8, 9, 15, 16, 17, 61, 62, 63, 64, 65, 127, 128, 140])
    counts = np.where(rng.random(n) < 0.5, special[rng.integers(0, special.size, n)], rng.integers(0, 20, n))
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(counts, out=rowptr[1:])
    cols = [np.sort(rng.choice(n, c, replace=False)) for c in counts]
    colidx = np.concatenate(cols).astype(np.int32)
    vals = rng.uniform(0.5, 1.5, colidx.size).astype(np.float32).astype(np.float64)
    return w.Csr(n, rowptr, colidx, vals)


@pytest.mark.parametrize("tile", [(2048, 8192), (32, 1024), (256, 2048)])
@pytest.mark.parametrize("k", [4, 16, 128])
def test_rows_by_length(arrow, tile, k):
    A = _matrix(2049)
    M = arrow.ArrowMatrix(A, 64, long_row=256)
    M.set_tuning(tile[0], tile[1], 2, 70)
    X = np.abs(w.features(A.n, k, seed=3))
    Xd = torch.from_numpy(X).cuda()
    R = S.iterate(A, X.astype(np.float64), 1)
    for got in (M.spmm(Xd, 1), arrow.ArrowBatch([M]).spmm([Xd], 1)[0]):
        Y = got.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(Y - R) <= 1e-5 * np.max(R, axis=0))


@pytest.mark.parametrize("k,rescale", [(16, True), (128, True), (16, False)])
def test_smaller_workspace_still_taken(arrow, k, rescale):
    """A workspace with FP64 sums for one CTA per tile only (less than workspace_size asks for where
    several CTAs share a tile) is accepted and gives the result of the full one."""
    A = w.grid_stencil((40, 37), seed=3)
    M = arrow.ArrowMatrix(A, 40)
    X = torch.from_numpy(w.features(A.n, k, seed=4)).cuda()
    full = M.workspace_size(k, "f32", rescale)
    rows = -(-A.n * k * 4 // 256) * 256
    one = 2 * rows + -(-k * 4 // 256) * 256                      # features, (no) segment partials
    if rescale:
        one += -(-M.stats()["tiles"] * k * 8 // 256) * 256 + -(-2 * k * 8 // 256) * 256
    assert one <= full and (one < full or not rescale)
    Y = M.spmm(X, 3, rescale=rescale)
    Yw = M.spmm_ws(X, 3, torch.empty(one, dtype=torch.uint8, device="cuda"), rescale=rescale)
    assert torch.allclose(Y, Yw, rtol=0, atol=1e-5 * 3 * float(Y.abs().max()))
    with pytest.raises(arrow.ArrowError):
        M.spmm_ws(X, 3, torch.empty(one - 256, dtype=torch.uint8, device="cuda"), rescale=rescale)


def _matrix_of(counts, seed):
    rng = np.random.default_rng(seed)
    n = counts.size
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(counts, out=rowptr[1:])
    colidx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in counts]).astype(np.int32)
    vals = rng.uniform(0.5, 1.5, colidx.size).astype(np.float32).astype(np.float64)
    return w.Csr(n, rowptr, colidx, vals)


@pytest.mark.parametrize("case", ["rows", "entries"])
@pytest.mark.parametrize("k", [4, 16, 128])
def test_descriptor_fields_at_their_ends(arrow, case, k):
    """A tile of 2048 rows (the largest row number, 2047) before one of a single row, and tiles of
    more than 8192 entries (starts that need all their bits; 12288 entries of 512 rows at most is as
    large as shared memory takes).  At most 100 entries a row: 100 * 2^-24 = 6e-6 of the sum."""
    rng = np.random.default_rng(12)
    if case == "rows":
        A, tile = _matrix_of(rng.integers(1, 4, 2049), 13), (2048, 8192)
    else:
        A, tile = _matrix_of(rng.integers(0, 101, 700), 14), (512, 12288)
    M = arrow.ArrowMatrix(A, 64, long_row=256)
    M.set_tuning(tile[0], tile[1], 1, 100)
    pg = M.program()
    rows, entries = np.diff(pg["tile_row"]), np.diff(pg["tile_ent"])
    if case == "rows":
        assert list(rows) == [2048, 1] and np.diff(pg["rowptr"])[2047] > 0
    else:
        assert entries.max() > 8192 + 200
    X = np.abs(w.features(A.n, k, seed=3))
    Xd = torch.from_numpy(X).cuda()
    R = S.iterate(A, X.astype(np.float64), 1)
    for got in (M.spmm(Xd, 1), arrow.ArrowBatch([M]).spmm([Xd], 1)[0]):
        Y = got.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(Y - R) <= 1e-5 * np.max(R, axis=0))


@pytest.mark.parametrize("fold_in", [0, 1])
@pytest.mark.parametrize("shift", [1, 250, -1, -250])
def test_x_and_y_overlap_in_part(arrow, fold_in, shift):
    """Y begins some rows into X, or X some rows into Y: every call has read its X (or keeps the
    permute-out pass) before it stores into Y, so the result is that of buffers apart."""
    A = w.rmat_gcn(9, 16, seed=6)
    M = arrow.ArrowMatrix(A, 32, long_row=16, segment=64)
    t = M.tuning
    M.set_tuning(t["tile_rows"], t["tile_nnz"], t["ctas_per_sm"], t["carveout"], fold_in)
    X0 = torch.from_numpy(w.features(A.n, 16, seed=7)).cuda()
    for iters in (1, 3):
        ref = M.spmm(X0, iters)
        buf = torch.zeros(A.n + abs(shift), 16, device="cuda")
        at = max(0, -shift)
        X, Y = buf[at:at + A.n], buf[at + shift:at + shift + A.n]
        X.copy_(X0)
        M.spmm(X, iters, out=Y)
        torch.cuda.synchronize()
        assert torch.equal(Y, ref)


@pytest.mark.parametrize("dims", [(40, 37), (150, 150), (250, 200), (300, 290)])
@pytest.mark.parametrize("dt,k", [("f32", 8), ("f32", 64), ("f32", 256), ("bf16", 128)])
def test_rescale_with_shared_tiles(arrow, dims, dt, k):
    """The column rescale where tiles are shared by several CTAs, by two and by none (6 to 340 tiles),
    narrow and wide rows, against the FP64 oracle (FP32 1e-5 per iteration, BF16 2e-2 in the 2-norm)."""
    A = w.grid_stencil(dims, seed=8)
    M = arrow.ArrowMatrix(A, 64, value_dtype=dt)
    X = torch.from_numpy(w.features(A.n, k, seed=9)).to("cuda", {"f32": torch.float32, "bf16": torch.bfloat16}[dt])
    Y = M.spmm(X, 3, rescale=True)
    assert torch.equal(Y, M.spmm(X, 3, rescale=True)) and M.status() == 0
    Y = Y.float().cpu().numpy().astype(np.float64)
    R = S.iterate(A, X.float().cpu().numpy().astype(np.float64), 3, rescale=True)
    if dt == "f32":
        assert np.max(np.max(np.abs(Y - R), axis=0) / np.max(np.abs(R), axis=0)) <= 1e-5 * 3
    else:
        assert np.max(np.linalg.norm(Y - R, axis=0) / np.linalg.norm(R, axis=0)) <= 2e-2


@pytest.mark.parametrize("case", ["even", "uneven", "long"])
@pytest.mark.parametrize("dt,k", [("f32", 128), ("f32", 384), ("bf16", 256)])
def test_wide_rows_in_row_order(arrow, case, dt, k):
    """Rows of 32 vectors come in row order where the lengths are even (one length, or 100 to 140: longer than
    a descriptor holds) and by length where they are not: the bits of narrower calls on slices of
    the columns, which always come by length."""
    n = 2049
    rng = np.random.default_rng(15)
    A = {"even": lambda: w.rgg(n, seed=16), "uneven": lambda: _matrix(n),
         "long": lambda: _matrix_of(rng.integers(100, 141, n), 17)}[case]()
    ln = np.diff(A.rowptr).astype(np.float64)
    assert ((ln ** 2).mean() <= 1.2 * ln.mean() ** 2) == (case != "uneven")
    M = arrow.ArrowMatrix(A, 64, value_dtype=dt, long_row=256)
    X = torch.from_numpy(w.features(n, k, seed=18)).to("cuda", {"f32": torch.float32, "bf16": torch.bfloat16}[dt])
    for tile in ((256, 2048), (2048, 8192), (32, 1024)):
        M.set_tuning(tile[0], tile[1], 2, 70)
        Y = M.spmm(X, 2)
        for c in range(0, k, 64):
            assert torch.equal(Y[:, c:c + 64], M.spmm(X[:, c:c + 64].contiguous(), 2))
    assert M.status() == 0
