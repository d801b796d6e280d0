"""Fisher terms on the product grid of the masked operator (the smallest grid of more than 4m points an axis): grids where it
is smaller than the data grid on all, some and no axes, uneven grids and two-stage and other lengths, against the oracle on
the data grid.  FP64: the alias argument is exact, 1e-11 of the largest element; FP32 and split: 2e-5 (FP32 transforms of the
draws, the mask and the products, each about 1e-7 relative, seen through sums that cancel)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import binning, ideal, unwindowed

pytestmark = pytest.mark.gpu

BOX = 900.0
CASES = [((64, 64, 64), 1.0 + 2.0 * np.arange(5)),      # m = 8: product grid 36 -> 48
         ((48, 54, 60), 1.0 + 2.0 * np.arange(6)),      # m = 10: 48 x 48 x 48
         ((40, 20, 50), 0.5 + 1.5 * np.arange(5)),      # m = 6: short y axis keeps its length
         ((24, 24, 24), 1.0 + 2.0 * np.arange(5)),      # N <= 4m on every axis: the data grid
         ((30, 64, 24), 1.0 + 1.5 * np.arange(5))]


def _mask(grid, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    n = 3.0e-4 * (0.5 + rng.random(grid))
    n[rng.random(grid) < 0.3] = 0.0
    return n.astype(np.float32)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 2e-5), ("split", 2e-5)])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_fisher_terms(prec, tol, case):
    import paper_2404_07249_gb300 as pkg
    grid, ek = CASES[case]
    edges = binning.kf_of(BOX) * ek
    nb = len(edges) - 1
    n = _mask(grid, case)
    pb = pkg.PolyBin(grid, BOX, edges, lmax=2, prec=prec)
    nd = torch.from_numpy(n).cuda()
    wd = pb.fkp_weights(nd, 1.0e4)
    w = wd.cpu().numpy().astype(np.float64)
    dt = np.float64 if prec == "fp64" else np.float32
    bins, mu2 = binning.bin_grid(grid, BOX, edges), binning.mu2_grid(grid)
    F = pb.fisher_draws(nd, wd, 11, pkg.FISHER_PK, 0, 1)[0]
    ref = unwindowed.pk_fisher_draw(unwindowed.draw(grid, 11, 0, 2, dt), n, w, bins, mu2, nb, [0, 2])
    assert np.max(np.abs(F - ref)) <= tol * np.max(np.abs(ref))
    trip = [tuple(t) for t in pb.triplets()[0].tolist()]
    F = pb.fisher_draws(nd, wd, 11, pkg.FISHER_BK, 0, 1)[0]
    ref = unwindowed.bk_fisher_draw(unwindowed.draw(grid, 11, 0, 0, dt), unwindowed.draw(grid, 11, 0, 1, dt), n, w, bins, nb,
                                    trip)
    assert np.max(np.abs(F - ref)) <= tol * np.max(np.abs(ref))
    pb.close()
