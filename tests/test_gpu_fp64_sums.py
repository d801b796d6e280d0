"""FP64 contraction over many cells of maps that are constants, where every rounding of a long running sum goes the same way.  Sums
are at most 512 terms long, a CTA adds its (4.1e6 cells / 304 CTAs / 512 = 27), and 16 slices of the CTAs are added
(19 each, then 16): with the product's rounding no more than 576 x 2^-53 of the sum, 6.4e-14."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_constant_maps():
    import paper_2404_07249_gb300 as pkg
    grid, nb = (160, 160, 160), 30
    n = 160 ** 3
    c = 0.5 + np.random.Generator(np.random.PCG64(8)).random(nb)
    pb = pkg.PolyBin(grid, 1000.0, 2.0 * np.pi / 1000.0 * np.array([0.5, 1.5]), prec="fp64")
    g = torch.from_numpy(c).cuda()[:, None, None, None].expand((nb,) + grid).contiguous()
    M = pb.contract(g)
    pb.close()
    worst = 0.0
    for p, (j, k) in enumerate(pkg.pair_list(nb)):
        ref = (np.longdouble(c[j]) * np.longdouble(c[k]) * c.astype(np.longdouble)) * n
        worst = max(worst, float(np.max(np.abs(M[p] - ref) / ref)))
    assert worst <= 576 * 2.0 ** -53, worst
