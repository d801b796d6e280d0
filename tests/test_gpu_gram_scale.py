"""Tensor-core Gram matrix of rows of one sign.  The tensor core cuts every partial sum towards zero at FP32's 24 bits: 0.36 x 2^-23
of it in the mean (half a unit in the last place of numbers spread evenly between two powers of two), and the partial
sums of an accumulator of n MMAs are 1/n, 2/n, .. of its total, so that the sums come out low by 0.36 x 2^-23 (n + 1) / 2.
With 32 products an accumulator, n = 4: 1.07e-7 (with 64, n = 8: 1.93e-7), apart from random errors of 1e-8."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("na,nb,K", [(40, 40, 65536), (130, 33, 20000)])
def test_one_sign(na, nb, K):
    import paper_2404_07249_gb300 as pkg
    gen = torch.Generator(device="cuda")
    gen.manual_seed(K)
    A = torch.rand((na, K), generator=gen, device="cuda") + 0.5
    B = torch.rand((nb, K), generator=gen, device="cuda") + 0.5
    out = torch.zeros((na, nb), dtype=torch.float64, device="cuda")
    pb = pkg.PolyBin((32, 32, 32), 1000.0, 2.0 * np.pi / 1000.0 * np.array([0.5, 1.5]), prec="split")
    f = getattr(pb.lib, "_ZN2pb11run_gram_tcEP11polybin_ctxPKfiS3_ildPd")
    f.restype = ctypes.c_int
    assert f(pb.ctx, ctypes.c_void_p(A.data_ptr()), na, ctypes.c_void_p(B.data_ptr()), nb, ctypes.c_long(K),
             ctypes.c_double(1.0), ctypes.c_void_p(out.data_ptr())) == 0
    pb.close()
    e = (out / (A.double() @ B.double().T) - 1.0).cpu().numpy()
    assert np.max(np.abs(e)) <= 1.5e-7, (np.mean(e), np.std(e))
