"""The t-SVD of few slices (a cluster of blocks per slice, columns kept in the
cluster's shared memory) against the float64 oracle: widths at the edges of the
rule (32) and around multiples of its 16 column blocks, so that blocks are odd,
even, short and empty, tall and wide slices, one slice, and repeated singular
values and rank-deficient slices, whose null columns shrink towards underflow.
Tolerances: the reconstruction at the repository's FP32 tolerance, the
singular values at the same relative to the largest."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,n3", [(32, 32, 1), (33, 40, 2), (64, 48, 3), (49, 50, 2), (90, 65, 4),
                                      (40, 113, 2), (200, 97, 1), (256, 129, 2)])
def test_tsvd(n1, n2, n3):
    X = synth.iid_normal((n1, n2, n3), seed=n1)
    X[: n1 // 3] = 0
    X[: n1 // 3, : n1 // 3] += np.eye(n1 // 3, n1 // 3)[:, : min(n2, n1 // 3), None]   # equal values
    U, S, V = (to_np(t) for t in tp.tsvd(tp.as_tprod_layout(X)))
    F, Uh, Sh, Vh = (np.fft.fft(t, axis=2) for t in (X.astype(np.float64), U, S, V))
    for k in range(n3):
        s = np.linalg.svd(F[:, :, k], compute_uv=False)
        assert np.abs(np.sort(np.diag(Sh[:, :, k]).real)[::-1] - s).max() < TOL_FP32 * s[0]
        assert rel_fro(Uh[:, :, k] @ Sh[:, :, k] @ Vh[:, :, k].conj().T, F[:, :, k]) < TOL_FP32
