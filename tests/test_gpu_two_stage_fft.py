"""Every two-stage FFT length on every axis: the pruned forward transform and the shell maps of a lognormal field against the
FP64 transforms.  FP32 transforms of up to 512 points are within 2e-6 of the L2 norm (the parity tests' bound)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import binning, ideal
from paper_2404_07249_gb300 import synth

pytestmark = pytest.mark.gpu

LENGTHS = [48, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 144, 150, 160, 180, 192, 200, 216, 240, 256, 270, 288, 300,
           320, 324, 360, 384, 400, 432, 480, 512]


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", LENGTHS)
def test_forward_and_shells(n, axis):
    import paper_2404_07249_gb300 as pkg
    grid = [6, 10, 8]
    grid[axis] = n
    grid = tuple(grid)
    box = 1000.0
    # bins up to the Nyquist wave number of the long axis, and just below it
    edges = binning.kf_of(box) * np.array([0.5, 2.5, 0.2 * n, 0.49 * n, 0.51 * n])
    f = synth.lognormal_field(grid, (box,) * 3, n + axis).astype(np.float32)
    pb = pkg.PolyBin(grid, box, edges, prec="fp32")
    spec = pb.forward(torch.from_numpy(f).cuda())
    dims, lo = pb.spectrum_shape()
    D = ideal.forward(f)
    ref = D[np.ix_(*[(np.arange(dims[a]) + lo[a]) % grid[a] for a in range(3)])]
    err = np.linalg.norm(spec.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err < 2e-6, err
    g = pb.shell_maps(spec).cpu().numpy().astype(np.float64)
    gref = ideal.shell_maps(D, binning.bin_grid(grid, box, edges), len(edges) - 1)
    for b in range(len(edges) - 1):
        e = np.linalg.norm(g[b] - gref[b]) / np.linalg.norm(gref[b])
        assert e < 2e-6, (b, e)
    pb.close()


@pytest.mark.parametrize("n", [54, 64])
def test_shell_maps_at_any_float(n):
    """Maps written at an address that is only a multiple of 4 bytes: the values of the aligned call to FP32 rounding."""
    import paper_2404_07249_gb300 as pkg
    grid = (6, 10, n)
    box = 1000.0
    edges = binning.kf_of(box) * np.array([0.5, 2.5, 0.2 * n])
    f = synth.lognormal_field(grid, (box,) * 3, n).astype(np.float32)
    pb = pkg.PolyBin(grid, box, edges, prec="fp32")
    spec = pb.forward(torch.from_numpy(f).cuda())
    ref = pb.shell_maps(spec)
    buf = torch.zeros(ref.numel() + 2, dtype=torch.float32, device="cuda")
    rc = pb.lib.polybin_shell_maps(pb.ctx, spec.data_ptr(), buf.data_ptr() + 4)
    assert rc == 0
    out = buf[1:-1].reshape(ref.shape)
    assert float((out - ref).norm() / ref.norm()) < 2e-6
    assert float(buf[0]) == 0 and float(buf[-1]) == 0
    pb.close()
