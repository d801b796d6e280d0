"""FP32 Gaussian draws (double-float Box-Muller) against the oracle's FP64 draws rounded to FP32: the FP32 numbers are those
of a value within 2^-40 of its size, so that about 2^-16 of them may round the other way, by one unit in the last place."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import binning, unwindowed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("grid", [(10, 6, 6), (30, 30, 50), (64, 64, 64)])
def test_draw(grid, shift):
    import paper_2404_07249_gb300 as pkg
    box = 1000.0
    pb = pkg.PolyBin(grid, box, binning.kf_of(box) * np.array([0.5, 1.5, 2.5]), prec="fp32")
    n = int(np.prod(grid))
    buf = torch.zeros(n + 8, dtype=torch.float32, device="cuda")
    assert pb.lib.polybin_mc_draw(pb.ctx, 1234567, 5, 3, buf.data_ptr() + 4 * shift) == 0
    torch.cuda.synchronize()
    out = buf.cpu().numpy()
    ref = unwindowed.draw(grid, 1234567, 5, 3, np.float32).ravel().astype(np.float32)
    got = out[shift:shift + n]
    assert np.all(np.abs(got - ref) <= np.spacing(np.abs(ref)))
    assert np.count_nonzero(got != ref) <= 3 + n * 2.0 ** -14
    assert np.all(out[:shift] == 0) and np.all(out[shift + n:] == 0)
    pb.close()
