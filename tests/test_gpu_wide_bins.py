"""P_0 in one bin of more modes than a grid's y dimension has segments of 1024 modes for (65535 x 1024 = 6.7e7), against the sum
over torch's transform: FP32 transforms and FP64 sums of 1e8 modes of one sign, 1e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_one_bin_of_1e8_modes():
    import paper_2404_07249_gb300 as pkg
    grid, box = (1024, 1024, 256), 1000.0
    kf = 2.0 * np.pi / box
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    d = torch.randn(grid, generator=gen, device="cuda", dtype=torch.float32)
    pb = pkg.PolyBin(grid, box, kf * np.array([0.5, 511.5]), prec="fp32")
    P = np.ravel(pb.pk(d))[0]
    pb.close()
    n = [torch.fft.fftfreq(m, d=1.0 / m, device="cuda").round().int() for m in grid[:2]]
    nz = torch.arange(grid[2] // 2 + 1, device="cuda", dtype=torch.int32)
    s = (n[0] ** 2)[:, None, None] + (n[1] ** 2)[None, :, None] + (nz ** 2)[None, None, :]
    w = torch.where((nz == 0) | (nz == grid[2] // 2), 1.0, 2.0).double()[None, None, :] * ((s > 0) & (s < 511.5 ** 2))
    assert torch.count_nonzero(w) > 65535 * 1024
    del s
    D = torch.fft.rfftn(d)
    ref = float((D.abs().double() ** 2 * w).sum() / w.sum()) * box ** 3 / float(np.prod(grid)) ** 2
    assert abs(P - ref) <= 1e-6 * ref
