"""The tree QR of tall slices (more than 256 rows) behind tsvd_randomized and
tp_sketch_spectrum: row counts at the edges of its 256-row blocks and levels,
column counts at the edges of its register shapes, blocks of zero and of very
small rows, and per-frequency column counts.

Data of tubal rank r <= k is recovered exactly by the range finder, so the
reference is the float64 SVD of every Fourier slice.  Tolerances: a float32
Householder QR is orthonormal to a small multiple of u32 sqrt(p) (2e-6 at
2000 rows; 2e-5 allowed), and the singular values and the reconstruction are
held to the bound of their precision (1e-5; 5e-5 for the bf16 split).
"""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from paper_1704_04362_gb300 import synth
from tests.util import to_np, tol_for

pytestmark = pytest.mark.gpu


def dev(x):
    return tp.as_tprod_layout(x)


def half(x):
    return np.fft.rfft(np.asarray(x, dtype=np.float64), axis=2)


def check(X, r, k, p, precision=tp.TP_FP32, sizes=None):
    import torch
    n1, n2, n3 = X.shape
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    sz = None if sizes is None else torch.tensor(sizes, dtype=torch.int32, device="cuda")
    U, S, V = tp.tsvd_randomized(dev(X), k, p, 1, seed=3, status=st, precision=precision,
                                 sketch_sizes=sz)
    assert int(st.item()) == 0
    Uh, Sh, Vh, Xh = half(to_np(U)), half(to_np(S)), half(to_np(V)), half(X)
    tol = tol_for(precision)
    err = tot = 0.0
    for f in range(n3 // 2 + 1):
        kf = k if sizes is None else min(k, sizes[f])
        # U = Q W with W from the core's float32 QL, whose vectors of the null
        # space (past the data's rank r) are not held to this bound
        G = Uh[:, :r, f].conj().T @ Uh[:, :r, f]
        assert np.abs(G - np.eye(r)).max() < 2e-5
        s = np.linalg.svd(Xh[:, :, f], compute_uv=False)
        got = np.diagonal(Sh[:, :, f].real)
        assert np.abs(got[:kf] - s[:kf]).max() <= tol * s[0]
        R = (Uh[:, :, f] * got) @ Vh[:, :, f].conj().T
        err += np.linalg.norm(R - Xh[:, :, f]) ** 2
        tot += np.linalg.norm(Xh[:, :, f]) ** 2
    assert err <= tol ** 2 * tot


@pytest.mark.parametrize("n1,n2,k,p", [
    (257, 40, 6, 2), (511, 33, 20, 12), (513, 70, 25, 8), (1024, 64, 44, 20), (1025, 100, 60, 5),
    (40, 700, 6, 4), (1300, 2000, 70, 26), (258, 96, 90, 6), (256, 97, 80, 16)])
def test_shapes(n1, n2, k, p):
    check(synth.lowrank_np(n1, n2, 3, 5, seed=n1 + k), 5, k, p)


@pytest.mark.parametrize("precision", [tp.TP_TF32X3, tp.TP_BF16X3])
def test_split_forms(precision):
    X = synth.lowrank_np(600, 300, 4, 6, seed=1)
    check(X, 6, 10, 6, precision)


@pytest.mark.parametrize("scale", [0.0, 1e-12])
def test_blocks_of_zero_and_of_small_rows(scale):
    X = np.array(synth.lowrank_np(900, 50, 4, 5, seed=2))
    X[:300] *= scale
    X[700:] *= scale
    check(np.asfortranarray(X.astype(np.float32)), 5, 8, 4)


def test_per_frequency_columns():
    X = synth.lowrank_np(700, 60, 4, 3, seed=4)
    check(X, 3, 8, 4, sizes=[12, 5, 7])
