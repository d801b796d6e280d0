"""Tensor-core contraction of maps whose largest values lie in different cells, so that no product comes near the product of
the maps' maxima, and of maps that span many orders of magnitude everywhere, against the FP64 sums.

The bound holds for any data, relative to S = sum_x |g_j g_k h_i|.  Operands: the FP32 product and the parts left out, 2^-23.
Tensor core: an accumulator takes 64 cells in MMAs of 16; each aligns its 16 products and the accumulator to the largest of
the 17 and may drop what lies below 2^-23 of it, so the four MMAs of the leading parts lose up to 4 x 17 x 2^-23 of the 64
cells' sum and the twenty others together 20 x 17 x 2^-23 x 2^-7.  FP32 sums of 32 accumulators: 32 x 2^-24.  Together
1.1e-5, however far below the maxima the terms lie."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

GRID = (64, 64, 64)
BOUND = 2.0 ** -23 + (4 * 17 + 20 * 17 * 2.0 ** -7) * 2.0 ** -23 + 32 * 2.0 ** -24


def _check(g, h):
    import paper_2404_07249_gb300 as pkg
    pb = pkg.PolyBin(GRID, 800.0, 2.0 * np.pi / 800.0 * np.array([0.5, 1.5]), prec="split")
    t = [torch.from_numpy(x.reshape((len(x),) + GRID)).cuda() for x in ((g,) if h is None else (g, h))]
    M = pb.contract(*t)
    assert pb.last_path() == pkg.PATH_TENSOR_SPLIT_TF32X3
    pb.close()
    G = g.astype(np.float64)
    H = G if h is None else h.astype(np.float64)
    for p, (j, k) in enumerate(pkg.pair_list(len(g))):
        ref, mag = H @ (G[j] * G[k]), np.abs(H) @ np.abs(G[j] * G[k])
        assert np.all(np.abs(M[p] - ref) <= BOUND * mag), (j, k, np.max(np.abs(M[p] - ref) / mag))


@pytest.mark.parametrize("separate", [False, True])
@pytest.mark.parametrize("background", ["constant", "positive", "signed"])
@pytest.mark.parametrize("peak", [6, 9, 12, 16, 20])
def test_peaks_in_different_cells(peak, background, separate):
    rng = np.random.Generator(np.random.PCG64(peak))
    n = int(np.prod(GRID))
    make = {"constant": lambda m: np.repeat(np.array([1.3, 1.1, 0.7, 0.9])[:m, None], n, axis=1),
            "positive": lambda m: 0.5 + rng.random((m, n)), "signed": lambda m: rng.standard_normal((m, n))}[background]
    g, h = make(3).astype(np.float32), make(4).astype(np.float32) if separate else None
    for i in range(3):                                    # a cell of its own for every map
        g[i, 1000 + 50001 * i] = np.float32(2.0 ** peak)
    if separate:
        for i in range(4):
            h[i, 2000 + 50001 * i] = np.float32(-2.0 ** peak)
    _check(g, h)


@pytest.mark.parametrize("width", [3.0, 8.0])
def test_wide_ranges_everywhere(width):
    rng = np.random.Generator(np.random.PCG64(int(width)))
    n = int(np.prod(GRID))
    g = np.exp(width * rng.uniform(-1.0, 1.0, (6, n))) * rng.choice([-1.0, 1.0], (6, n))
    g[1] = 1.0 / g[0]                                     # large where the other is small
    _check(g.astype(np.float32), None)
