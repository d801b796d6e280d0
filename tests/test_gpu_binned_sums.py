"""Branches of the binned sums, the SIMT contraction and the batched call that depend on values and sizes: conversions of FP32
spectra to FP64 (scaling a field by a power of two scales P exactly, zeros stay zero, infinities and NaN do not turn into
numbers), more pair rows than the contraction's table of row places has room for, and more contexts in a batch than it has
branches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BOX = 800.0
KF = 2.0 * np.pi / BOX


def test_scaled_fields():
    import paper_2404_07249_gb300 as pkg
    g = torch.Generator().manual_seed(5)
    f = torch.randn((36, 40, 48), generator=g)
    pb = pkg.PolyBin((36, 40, 48), BOX, KF * np.arange(1.0, 14.0, 2.0), lmax=4, prec="fp32")
    P = pb.pk(f.cuda())
    for e in (-40, 40):
        assert np.array_equal(pb.pk((f * 2.0 ** e).cuda()), P * 4.0 ** e)
    assert not pb.pk((f * 0.0).cuda()).any()
    bad = f.clone()
    bad[1, 2, 3] = float("nan")
    assert np.isnan(pb.pk(bad.cuda())).all()
    pb.close()


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-13)])
def test_contraction_without_table(prec, tol):
    import paper_2404_07249_gb300 as pkg
    dt = np.float32 if prec == "fp32" else np.float64
    rng = np.random.Generator(np.random.PCG64(9))
    ng, nh, grid = 40, 5, (6, 10, 12)                  # 820 pair rows, one tile column
    g, h = rng.standard_normal((ng,) + grid).astype(dt), rng.standard_normal((nh,) + grid).astype(dt)
    pb = pkg.PolyBin(grid, BOX, KF * np.array([0.5, 1.5]), prec=prec)
    M = pb.contract(torch.from_numpy(g).cuda(), torch.from_numpy(h).cuda())
    G, H = g.astype(np.float64).reshape(ng, -1), h.astype(np.float64).reshape(nh, -1)
    for p, (j, k) in enumerate(pkg.pair_list(ng)):
        assert np.all(np.abs(M[p] - H @ (G[j] * G[k])) <= tol * (np.abs(H) @ np.abs(G[j] * G[k]))), (j, k)
    pb.close()


def test_more_contexts_than_branches():
    import paper_2404_07249_gb300 as pkg
    edges = KF * np.array([1.0, 3.0, 5.0, 7.0])
    stream = torch.cuda.current_stream().cuda_stream
    specs = [((24 + 6 * (i % 3),) * 3, ("split", "fp32", "fp64")[i % 3]) for i in range(7)]
    pbs = [pkg.PolyBin(g, BOX, edges, prec=p, stream=stream) for g, p in specs]
    order = [i % 7 for i in range(17)]
    fields = [torch.randn(specs[i][0], generator=torch.Generator().manual_seed(60 + n)).cuda() for n, i in enumerate(order)]
    single = [pbs[i].bk_ideal(f)[0] for i, f in zip(order, fields)]
    for _ in range(2):
        multi = pkg.bk_ideal_multi([pbs[i] for i in order], fields)
        assert all(np.array_equal(a, b) for a, b in zip(multi, single))
    for pb in pbs:
        pb.close()
