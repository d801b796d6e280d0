"""Gaussian draws are the FP64 numbers rounded to FP32, number by number.  The reference reduces the angle exactly (u is a multiple
of 2^-33) and has a relative error of a few 2^-53; the few numbers that 4e-15 could round the other way are left out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.philox import philox4x32_10

pytestmark = pytest.mark.gpu


def _reference(n, seed, r, stream):
    j = np.arange(n // 4, dtype=np.uint64)
    x = philox4x32_10(j & np.uint64(0xFFFFFFFF), j >> np.uint64(32), np.uint64(r), np.uint64(stream),
                      np.uint64(seed % 2 ** 32), np.uint64(seed // 2 ** 32))
    z = np.empty((n // 4, 4))
    for h in range(2):
        radius = np.sqrt(-2.0 * np.log((x[2 * h].astype(np.float64) + 0.5) * 2.0 ** -32))
        e = (x[2 * h + 1].astype(np.float64) + 0.5) * 2.0 ** -29        # the angle in eighths of a turn
        o = np.floor(e).astype(int)
        a = np.where(o & 1, o + 1 - e, e - o) * (np.pi / 4.0)           # from the octant's even end
        c, s = np.cos(a), np.sin(a)
        swap = ((o + 1) & 2) != 0
        c, s = np.where(swap, s, c), np.where(swap, c, s)
        z[:, 2 * h] = radius * np.where((o >= 2) & (o < 6), -c, c)
        z[:, 2 * h + 1] = radius * np.where(o >= 4, -s, s)
    return z.ravel()


@pytest.mark.parametrize("seed,r,stream", [(1, 0, 0), (987654321, 17, 3), (2 ** 40 + 5, 1000, 2)])
def test_draws_are_rounded_fp64_numbers(seed, r, stream):
    import paper_2404_07249_gb300 as pkg
    grid = (256, 256, 128)
    pb = pkg.PolyBin(grid, 1000.0, 2.0 * np.pi / 1000.0 * np.array([0.5, 1.5, 2.5]), prec="fp32")
    buf = torch.zeros(grid, dtype=torch.float32, device="cuda")
    assert pb.lib.polybin_mc_draw(pb.ctx, seed, r, stream, buf.data_ptr()) == 0
    pb.close()
    z = _reference(int(np.prod(grid)), seed, r, stream)
    sure = (z * (1.0 - 4e-15)).astype(np.float32) == (z * (1.0 + 4e-15)).astype(np.float32)
    assert np.count_nonzero(~sure) < 100
    assert np.array_equal(buf.cpu().numpy().ravel()[sure], z.astype(np.float32)[sure])
