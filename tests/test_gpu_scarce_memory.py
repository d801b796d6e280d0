"""Calls whose batches and tables do not fit the device's memory run without them: a Fisher term and a local line-of-sight numerator
of a new context with little memory left, against the same calls with all of it (the same sums in other batches: FP32
rounding, 2e-5 of the largest element), and again with room."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

GRID, BOX = (128, 128, 128), 1000.0


def _inputs():
    import paper_2404_07249_gb300 as pkg
    rng = np.random.Generator(np.random.PCG64(4))
    n = (3.0e-4 * (0.5 + rng.random(GRID))).astype(np.float32)
    n[rng.random(GRID) < 0.3] = 0.0
    n = torch.from_numpy(n).cuda()
    d = n * torch.from_numpy(rng.standard_normal(GRID).astype(np.float32)).cuda()
    edges = 2.0 * np.pi / BOX * (1.0 + 6.0 * np.arange(6))
    pb = pkg.PolyBin(GRID, BOX, edges, lmax=4, prec="fp32")
    return pkg, pb, n, pb.fkp_weights(n, 1.0e4), d


def _leave(mib):
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - (mib << 20), dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("mib", [32, 64, 96])
def test_fisher_term(mib):
    pkg, pb, n, w, d = _inputs()
    ref = pb.fisher_draws(n, w, 5, pkg.FISHER_PK, 0, 1)
    pb.close()
    pkg, pb, n, w, d = _inputs()
    pb.shell_maps(pb.forward(d))                               # what the term on the data grid needs of the context
    pb.pk_unwindowed(d, w, with_estimate=False)
    torch.cuda.synchronize()
    hog = _leave(mib)
    try:
        F = pb.fisher_draws(n, w, 5, pkg.FISHER_PK, 0, 1)
    finally:
        del hog
        torch.cuda.empty_cache()
    G = pb.fisher_draws(n, w, 5, pkg.FISHER_PK, 0, 1)
    pb.close()
    assert np.max(np.abs(F - ref)) <= 2e-5 * np.max(np.abs(ref))
    assert np.array_equal(G, ref)


@pytest.mark.parametrize("mib", [16, 24, 32, 64])
def test_local_numerator(mib):
    pkg, pb, n, w, d = _inputs()
    pb.set_observer((0.0, 0.0, 0.0))
    ref = pb.pk_unwindowed_local(d, w, with_estimate=False)[1]
    pb.close()
    pkg, pb, n, w, d = _inputs()
    pb.set_observer((0.0, 0.0, 0.0))
    pb.pk_unwindowed(d, w, with_estimate=False)
    torch.cuda.synchronize()
    hog = _leave(mib)
    try:
        num = pb.pk_unwindowed_local(d, w, with_estimate=False)[1]
    finally:
        del hog
        torch.cuda.empty_cache()
    pb.close()
    assert np.max(np.abs(num - ref)) <= 2e-5 * np.max(np.abs(ref))
