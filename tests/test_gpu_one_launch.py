"""GPU test of the one-launch path's column sums at every number of columns (4 to 256).

With the column rescale each stored column has unit norm up to rounding, so the result is compared with
the FP64 oracle at the FP32 bar (1e-5 per iteration, as the multi-launch path) or, for 16-bit storage,
2e-2 in the 2-norm; grids of one CTA, of fewer CTAs than SMs and of one per SM.
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


@pytest.mark.parametrize("dt,k", [("f32", 4), ("f32", 8), ("f32", 32), ("f32", 128), ("bf16", 8), ("bf16", 256)])
@pytest.mark.parametrize("dims", [(5, 3), (61, 37), (113, 97)])
def test_rescale_at_every_width(arrow, dt, k, dims):
    A = w.grid_stencil(dims, seed=4)
    X = w.features(A.n, k, seed=5)
    Xd = torch.from_numpy(X).to("cuda", {"f32": torch.float32, "bf16": torch.bfloat16}[dt])
    M = arrow.ArrowMatrix(A, 32, value_dtype=dt)
    t = M.tuning
    M.set_tuning(t["tile_rows"], t["tile_nnz"], t["ctas_per_sm"], t["carveout"], 0, 1)
    it = 4
    Y = M.spmm(Xd, it, rescale=True)
    assert torch.equal(Y, M.spmm(Xd, it, rescale=True))
    assert M.status() == 0
    Y = Y.float().cpu().numpy().astype(np.float64)
    R = S.iterate(A, Xd.float().cpu().numpy().astype(np.float64), it, rescale=True)
    if dt == "f32":
        assert np.max(np.max(np.abs(Y - R), axis=0) / np.max(np.abs(R), axis=0)) <= 1e-5 * it
    else:
        assert np.max(np.linalg.norm(Y - R, axis=0) / np.linalg.norm(R, axis=0)) <= 2e-2


@pytest.mark.parametrize("rescale", [False, True])
def test_overlapping_calls_on_one_handle(arrow, rescale):
    """Calls with workspaces of their own on two streams may overlap on one handle: each counts its
    grid barrier's arrivals in its own workspace, so every one gives the bits of a call alone."""
    A = w.rmat_gcn(9, 16, seed=4)
    M = arrow.ArrowMatrix(A, 32)
    t = M.tuning
    M.set_tuning(t["tile_rows"], t["tile_nnz"], t["ctas_per_sm"], t["carveout"], 0, 1)
    assert M.stats()["segments"] > 0
    X = torch.from_numpy(w.features(A.n, 32, seed=6)).cuda()
    ref = M.spmm(X, 6, rescale=rescale)
    streams = [torch.cuda.Stream() for _ in range(2)]
    ws = [torch.empty(M.workspace_size(32, "f32", rescale), dtype=torch.uint8, device="cuda") for _ in streams]
    outs = [[torch.empty_like(X) for _ in range(20)] for _ in streams]
    torch.cuda.synchronize()
    for i in range(20):
        for s, b, ys in zip(streams, ws, outs):
            M.spmm_ws(X, 6, b, rescale=rescale, out=ys[i], stream=s)
    torch.cuda.synchronize()
    assert M.status() == 0
    assert all(torch.equal(y, ref) for ys in outs for y in ys)
