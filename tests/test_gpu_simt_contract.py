"""SIMT contraction over its tile shapes: replicated tiles (few rows), one tile a thread, row groups, singles from the maps
themselves and from separate ones, cell counts that are not a multiple of a chunk.  FP32 products and sums of at most 512
cells: within 1e-6 of sum_x |g_j g_k h_i|; FP64: 1e-13."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-13)])
@pytest.mark.parametrize("grid", [(2, 2, 2), (6, 6, 10), (20, 24, 30)])
@pytest.mark.parametrize("ng,nh", [(1, 0), (3, 0), (8, 0), (13, 0), (13, 1), (23, 64), (33, 0), (64, 17)])
def test_tile_shapes(prec, tol, grid, ng, nh):
    import paper_2404_07249_gb300 as pkg
    dt = np.float32 if prec == "fp32" else np.float64
    rng = np.random.Generator(np.random.PCG64(100 * ng + nh))
    g = rng.standard_normal((ng,) + grid).astype(dt)
    h = g if nh == 0 else rng.standard_normal((nh,) + grid).astype(dt)
    pb = pkg.PolyBin(grid, 800.0, 2.0 * np.pi / 800.0 * np.array([0.5, 1.5]), prec=prec)
    M = pb.contract(torch.from_numpy(g).cuda(), None if nh == 0 else torch.from_numpy(h).cuda())
    G, H = g.astype(np.float64).reshape(ng, -1), h.astype(np.float64).reshape(h.shape[0], -1)
    for p, (j, k) in enumerate(pkg.pair_list(ng)):
        ref = H @ (G[j] * G[k])
        mag = np.abs(H) @ np.abs(G[j] * G[k])
        assert np.all(np.abs(M[p] - ref) <= tol * mag), (j, k)
    pb.close()
