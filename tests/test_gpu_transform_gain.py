"""The FP32 transforms have a gain of one: the factor between their results and the FP64 ones, fitted over all modes or cells.  The
rounded constants of a length leave at most 6e-9 (64 points, on the other two axes, 1e-9); the random errors of 6e4 values
and more add 2e-7 / sqrt(6e4) at most: 1e-8.  (The maps' 1 / N is an FP32 number, and so it is in their reference.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LENGTHS = [48, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 144, 150, 160, 180, 192, 200, 216, 240, 256, 270, 288, 300, 320,
           324, 360, 384, 400, 432, 480, 512]


def _factor(x, ref):
    x, ref = x.to(ref.dtype), ref
    return float((x * ref.conj()).real.sum() / (ref * ref.conj()).real.sum())


@pytest.mark.parametrize("n", LENGTHS)
def test_gain(n):
    import paper_2404_07249_gb300 as pkg
    grid, box = (n, 64, 64), 1000.0
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)
    d = torch.randn(grid, generator=gen, device="cuda", dtype=torch.float32)
    top = max(n, 64)                                           # beyond every wave number: the box is the whole spectrum
    pb = pkg.PolyBin(grid, box, 2.0 * np.pi / box * np.array([0.5, top]), prec="fp32")
    S = pb.forward(d)
    assert tuple(S.shape) == (n, 64, 33)
    full = torch.empty((n, 64, 33), dtype=torch.complex64, device="cuda")
    ix = torch.arange(-(n // 2), n // 2, device="cuda") % n
    iy = torch.arange(-32, 32, device="cuda") % 64
    full[ix[:, None], iy[None, :]] = S
    assert abs(_factor(full, torch.fft.rfftn(d.double())) - 1.0) <= 1e-8
    g = pb.shell_maps(S)[0]
    pb.close()
    # the maps hold every mode but k = 0, and no imaginary part where a mode is its own conjugate
    back = full.to(torch.complex128)
    back[0, 0, 0] = 0.0
    norm = float(np.float32(1.0 / (n * 4096))) * (n * 4096)
    assert abs(_factor(g, torch.fft.irfftn(back, s=grid) * norm) - 1.0) <= 1e-8
