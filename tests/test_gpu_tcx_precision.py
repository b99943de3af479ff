"""t-CX whose picks are orthonormalised without the SVD is as accurate as with
it.  A duplicate of one picked slice sends the call to the SVD and leaves the
span as it is, so the two errors against the float64 projection are of the same
result: float32 rounding of the tensor, of the basis and of the products in both.
The mean over the cases may not be larger than the SVD's (each error is a root
mean square over thousands of entries; the sums that start with the small
columns make it a tenth smaller)."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from paper_1704_04362_gb300 import synth
from tests.test_gpu_tcx_qr import project
from tests.util import rel_fro, to_np

pytestmark = pytest.mark.gpu


def error(A, idx):
    import torch
    p = np.zeros(A.shape[1])
    p[idx] = 1.0 / len(idx)
    Z, _, cnt = tp.tcx(tp.as_tprod_layout(A), len(idx), seed=1, prob_mode=tp.TP_PROB_GIVEN,
                       p_given=torch.from_numpy(p).to("cuda"))
    assert int(cnt.item()) == len(idx)
    return rel_fro(to_np(Z), project(A, idx))


def test_error_is_the_svd_forms():
    plain, svd = [], []
    for n1, n2, n3, c in [(69, 120, 8, 38), (100, 249, 15, 63), (256, 200, 16, 64), (128, 340, 11, 30),
                          (300, 150, 9, 50), (72, 297, 19, 18)]:
        A = np.array(synth.lowrank_np(n1, n2, n3, 10, seed=n1, noise=0.01))
        A[:, -1] = A[:, 0]
        A = np.asfortranarray(A.astype(np.float32))
        plain.append(error(A, list(range(c))))
        svd.append(error(A, list(range(c)) + [n2 - 1]))
    assert np.mean(plain) <= np.mean(svd), (plain, svd)
