"""Harmonic transforms of the local line of sight where directions degenerate: an observer at a cell's centre (the direction
of that cell is undefined, its line has no azimuth), on a line of cells, in the plane of a layer, far outside; on even and
uneven grids of two-stage lengths.  Power spectrum numerator with ell = 0, 2, 4 against the oracle in FP64: 1e-6 of the
largest value in FP32 (the bound of the local numerator's other tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import binning, local

pytestmark = pytest.mark.gpu

BOX = 640.0
GRIDS = [(64, 64, 64), (48, 60, 80), (54, 64, 90)]


def _observer(kind, grid):
    h = [BOX / n for n in grid]
    centre = [(g // 3 + 0.5) * s - BOX / 2 for g, s in zip(grid, h)]
    return {"cell": tuple(centre), "line": (centre[0], centre[1], centre[2] + 0.3 * h[2]),
            "layer": (0.11 * BOX, -0.07 * BOX, centre[2]), "far": (30.0 * BOX, 2.0 * BOX, -11.0 * BOX)}[kind]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("kind", ["cell", "line", "layer", "far"])
def test_degenerate_directions(grid, kind):
    import paper_2404_07249_gb300 as pkg
    rng = np.random.Generator(np.random.PCG64(sum(grid)))
    d = rng.standard_normal(grid).astype(np.float32)
    w = (0.5 + rng.random(grid)).astype(np.float32)
    edges = binning.kf_of(BOX) * np.array([0.0, 3.0, 6.0, 9.0, 12.0])
    obs = _observer(kind, grid)
    pb = pkg.PolyBin(grid, BOX, edges, lmax=4, prec="fp32")
    pb.set_observer(obs)
    _, p = pb.pk_unwindowed_local(torch.from_numpy(d).cuda(), torch.from_numpy(w).cuda(), with_estimate=False)
    bins = binning.bin_grid(grid, BOX, edges)
    ref = local.pk_numerator_local(d, w, bins, 4, [0, 2, 4], local.position_units(grid, BOX, obs), local.mode_units(grid))
    assert np.max(np.abs(p - ref.ravel())) < 1e-6 * np.max(np.abs(ref))
    pb.close()
