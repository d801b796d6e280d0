"""Batched passes of the masked operator where the last batch is a part of one, with lengths of its own on an axis that keeps the
data grid's (48) and lengths that are no multiple of four (54, 90), against the double-precision context, which goes item by
item through other passes: 2e-5 of the largest element, as for the smaller cases against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BOX = 900.0
CASES = [((108, 48, 120), 1.0 + 1.5 * np.arange(9)),       # m = 12: product grid 54 x 48 x 54, batches of 64
         ((108, 100, 96), 0.5 + 2.35 * np.arange(10))]     # m = 21: 90 x 90 x 90, batches of about 30


@pytest.mark.parametrize("prec", ["fp32", "split"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_fisher_terms(prec, case):
    import paper_2404_07249_gb300 as pkg
    grid, ek = CASES[case]
    rng = np.random.Generator(np.random.PCG64(case))
    n = 3.0e-4 * (0.5 + rng.random(grid))
    n[rng.random(grid) < 0.3] = 0.0
    nd = torch.from_numpy(n.astype(np.float32)).cuda()
    out = []
    for p in ("fp64", prec):
        pb = pkg.PolyBin(grid, BOX, 2.0 * np.pi / BOX * ek, lmax=4, prec=p)
        wd = pb.fkp_weights(nd, 1.0e4)
        out.append([pb.fisher_draws(nd, wd, 11, which, 0, 1)[0] for which in (pkg.FISHER_PK, pkg.FISHER_BK)])
        assert pb.num_triplets() > 64
        pb.close()
    for ref, F in zip(*out):
        assert np.max(np.abs(F - ref)) <= 2e-5 * np.max(np.abs(ref))
