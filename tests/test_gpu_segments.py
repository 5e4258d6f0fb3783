"""GPU test of the split-row segment kernels around their round sizes.

Split rows of 33 to 1,100 entries (one to three segments of 512, remainders of every kind for the 8- and
16-gather rounds of 1 to 32 teams).  A single call on few segments takes the look-ahead form; the
same matrix often enough in one batch takes the other: both must give the same bits, and match
the FP64 oracle: with positive values a sum of 1,100 products in any order has a relative error
below 1,100 * 2^-24 = 6.6e-5, so 1e-4 per iteration bounds every element.
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


def _matrix(n=1500):
    rng = np.random.default_rng(21)
    counts = rng.integers(0, 4, n)
    special = [33, 34, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 520, 1023, 1024, 1025, 1100]
    counts[rng.choice(n, len(special) * 3, replace=False)] = special * 3
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(counts, out=rowptr[1:])
    colidx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in counts]).astype(np.int32)
    vals = rng.uniform(0.5, 1.5, colidx.size).astype(np.float32).astype(np.float64)
    return w.Csr(n, rowptr, colidx, vals)


@pytest.mark.parametrize("k", [4, 8, 16, 32, 64, 128])
def test_few_and_many_segments(arrow, k):
    A = _matrix()
    M = arrow.ArrowMatrix(A, 64, long_row=32)
    seg = M.stats()["segments"]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert 0 < seg <= 8 * sms
    X = np.abs(w.features(A.n, k, seed=3))
    Xd = torch.from_numpy(X).cuda()
    Y = M.spmm(Xd, 2)
    copies = 8 * sms // seg + 2                       # more segments than the look-ahead form takes
    Ys = arrow.ArrowBatch([M] * copies).spmm([Xd] * copies, 2)
    assert all(torch.equal(Y, y) for y in Ys)
    t = M.tuning
    M.set_tuning(t["tile_rows"], t["tile_nnz"], t["ctas_per_sm"], t["carveout"], 0, 1)
    assert torch.equal(Y, M.spmm(Xd, 2))
    R = S.iterate(A, X.astype(np.float64), 2)
    assert np.all(np.abs(Y.cpu().numpy().astype(np.float64) - R) <= 2 * 1e-4 * np.max(R, axis=0))
