"""Split-FP16 tensor-core contraction at the edges of its cell stages (64 cells), windows (16 and 32 singles) and scale
factors: maps whose magnitudes differ by many powers of two, a map of zeros and a map with one dominant cell, against the
FP64 sums.  Each product and each single is kept to 22 bits and the sums of 64 cells run in FP32 on the tensor core, so a sum
is within 1e-6 of sum_x |g_j g_k h_i| at every scale (the scales are powers of two and drop out)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(2, 2, 2), (4, 4, 6), (10, 6, 6), (30, 30, 50)])
@pytest.mark.parametrize("ng,nh", [(2, 0), (16, 0), (17, 0), (31, 0), (5, 32), (22, 9)])
def test_scales_and_ragged_cells(grid, ng, nh):
    import paper_2404_07249_gb300 as pkg
    rng = np.random.Generator(np.random.PCG64(1000 * ng + nh))
    n = int(np.prod(grid))
    g = rng.standard_normal((ng, n)).astype(np.float32)
    g *= 2.0 ** rng.integers(-30, 30, ng)[:, None].astype(np.float32)
    g[0] = 0.0
    g[-1, n // 2] = 1.0e4 * np.abs(g[-1]).max()
    h = g if nh == 0 else (rng.standard_normal((nh, n)) * 2.0 ** rng.integers(-20, 20, nh)[:, None]).astype(np.float32)
    pb = pkg.PolyBin(grid, 800.0, 2.0 * np.pi / 800.0 * np.array([0.5, 1.5]), prec="split")
    tg = torch.from_numpy(g.reshape((ng,) + grid)).cuda()
    M = pb.contract(tg) if nh == 0 else pb.contract(tg, torch.from_numpy(h.reshape((nh,) + grid)).cuda())
    assert pb.last_path() == pkg.PATH_TENSOR_SPLIT_TF32X3
    G, H = g.astype(np.float64), h.astype(np.float64)
    for p, (j, k) in enumerate(pkg.pair_list(ng)):
        ref = H @ (G[j] * G[k])
        mag = np.abs(H) @ np.abs(G[j] * G[k])
        assert np.all(np.abs(M[p] - ref) <= 1e-6 * mag), (j, k)
    pb.close()


def test_non_finite_maps_stay_in_their_sums():
    import paper_2404_07249_gb300 as pkg
    rng = np.random.Generator(np.random.PCG64(5))
    grid, ng = (8, 8, 8), 4
    g = rng.standard_normal((ng,) + grid).astype(np.float32)
    g[3, 1, 2, 3] = np.inf
    pb = pkg.PolyBin(grid, 800.0, 2.0 * np.pi / 800.0 * np.array([0.5, 1.5]), prec="split")
    M = pb.contract(torch.from_numpy(g).cuda())
    G = g.astype(np.float64).reshape(ng, -1)
    for p, (j, k) in enumerate(pkg.pair_list(ng)):
        for i in range(ng):
            if 3 in (j, k, i):
                assert not np.isfinite(M[p, i])
            else:
                assert abs(M[p, i] - np.sum(G[j] * G[k] * G[i])) <= 1e-6 * np.sum(np.abs(G[j] * G[k] * G[i]))
    pb.close()
