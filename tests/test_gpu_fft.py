"""The mixed-radix mode-3 FFT against float64: lengths of one to five primes
up to 13 in even and odd products, every radix up to 16, lengths with one and
with several tubes per block, tubes around its blocks, and the gathered,
transposed and split forms through the t-products.  Tolerances as the
repository holds its transforms and products; a tube's error is bounded by its
own size, not its neighbours'."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import sampling_ref, tensor_ref
from paper_1704_04362_gb300 import synth
from tests.test_gpu_transforms import check_transforms
from tests.util import TOL_FP32, rel_fro, to_np, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n3", [18, 20, 21, 22, 24, 25, 26, 27, 28, 30, 33, 35, 36, 39, 40, 44, 45, 48,
                                49, 50, 52, 55, 63, 65, 72, 77, 80, 91, 96, 117, 120, 121, 143, 144,
                                168, 169, 195, 210, 225, 243, 256, 315, 343, 504, 512, 625, 1000, 1155,
                                2000, 2197, 4096, 6561, 8190, 8400])
def test_lengths(n3):
    check_transforms(33, 9, n3)


@pytest.mark.parametrize("rows,cols,n3", [(1, 1, 18), (257, 1, 45), (64, 1, 80), (65, 31, 2000),
                                          (401, 333, 21), (200, 517, 80), (512, 300, 168)])
def test_numbers_of_tubes(rows, cols, n3):
    check_transforms(rows, cols, n3)


@pytest.mark.parametrize("prec", [tp.TP_FP32, tp.TP_TF32X3, tp.TP_BF16X3])
@pytest.mark.parametrize("n3", [18, 35, 45, 80, 168])
def test_products(n3, prec):
    A = synth.iid_normal((45, 70, n3), seed=3)
    B = synth.iid_normal((70, 37, n3), seed=4)
    ref = tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))
    C = tp.tprod(tp.as_tprod_layout(A), tp.as_tprod_layout(B), precision=prec)
    assert rel_fro(to_np(C), ref) < tol_for(prec)
    Z, _, _ = tp.tprod_sampled(tp.as_tprod_layout(A), tp.as_tprod_layout(B), 20, seed=5,
                               precision=prec)
    Zr, _, _ = sampling_ref.tprod_sampled(A, B, 20, 5)
    assert rel_fro(to_np(Z), Zr) < tol_for(prec)


@pytest.mark.parametrize("n3", [24, 45, 2000])
def test_a_tube_keeps_to_itself(n3):
    X = synth.iid_normal((21, 6, n3), seed=6)
    X[4] *= 1e12
    X[7, 3, 1] = np.inf
    Xr, Xi = tp.rdft3(tp.as_tprod_layout(X))
    got = to_np(Xr) + 1j * to_np(Xi)
    keep = np.ones((21, 6), bool)
    keep[7, 3] = False
    ref = np.fft.rfft(np.where(keep[:, :, None], X, 0).astype(np.float64), axis=2)
    err = np.linalg.norm(got - ref, axis=2)[keep] / np.linalg.norm(ref, axis=2)[keep]
    assert err.max() < TOL_FP32
    assert not np.isfinite(got[7, 3]).all()
