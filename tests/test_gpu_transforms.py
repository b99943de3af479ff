"""The mode-3 transforms of short tubes (registers, lengths 1 .. 16) and of
tubes whose length has a large prime factor (products with the transform
matrix) against float64: every length of the register form, lengths around the
product's blocks of 4 outputs, 8 samples and its shared-memory parts, tubes
around its tiles, odd lines (unaligned stores), and the gathered, transposed
and split forms through the t-products.  Tolerance: as the repository holds
its transforms and products (1e-5; the precision's own bound)."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import sampling_ref, tensor_ref
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np, tol_for

pytestmark = pytest.mark.gpu

LENGTHS = list(range(1, 17)) + [17, 19, 23, 29, 31, 34, 37, 47, 59, 61, 62, 67, 127, 251, 257, 509]


def check_transforms(rows, cols, n3):
    X = synth.iid_normal((rows, cols, n3), seed=n3)
    Xr, Xi = tp.rdft3(tp.as_tprod_layout(X))
    ref = np.fft.rfft(X.astype(np.float64), axis=2)
    assert rel_fro(to_np(Xr) + 1j * to_np(Xi), ref) < TOL_FP32
    assert rel_fro(to_np(tp.irdft3(Xr, Xi, n3)), X) < TOL_FP32
    # the imaginary parts of the real slices are ignored
    H = synth.iid_normal((rows, cols, n3 // 2 + 1), seed=1).astype(np.float64)
    G = synth.iid_normal((rows, cols, n3 // 2 + 1), seed=2).astype(np.float64)
    out = tp.irdft3(tp.as_tprod_layout(H.astype(np.float32)), tp.as_tprod_layout(G.astype(np.float32)),
                    n3)
    G[:, :, 0] = 0
    if n3 % 2 == 0:
        G[:, :, -1] = 0
    assert rel_fro(to_np(out), np.fft.irfft(H + 1j * G, n=n3, axis=2)) < TOL_FP32


@pytest.mark.parametrize("n3", LENGTHS)
@pytest.mark.parametrize("rows,cols", [(1, 1), (64, 2), (33, 9)])
def test_transforms(rows, cols, n3):
    check_transforms(rows, cols, n3)


@pytest.mark.parametrize("n3", [5, 16, 31, 67])
def test_transforms_of_many_tubes(n3):
    check_transforms(401, 333, n3)


@pytest.mark.parametrize("prec", [tp.TP_FP32, tp.TP_TF32X3, tp.TP_BF16X3])
@pytest.mark.parametrize("n3", [3, 7, 12, 15, 17, 31, 67])
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


@pytest.mark.parametrize("n3", [6, 16, 31])
def test_a_tube_keeps_to_itself(n3):
    """Infinities, and values far larger than their neighbours'."""
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
