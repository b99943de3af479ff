"""The cluster Jacobi's two forms against each other by device time: the form in
the cluster's shared memory holds an SM per CTA, so that 33 slices would take
three rounds of it where the form through L2 takes all at once, as it takes 25.
The singular values of both sides of the line against float64 (the float32
paths' tolerance)."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, to_np

pytestmark = pytest.mark.gpu


def sweeps_ms(n1, n2, slices):
    import torch
    X = tp.as_tprod_layout(synth.iid_normal((n1, n2, 2 * slices - 2), seed=n1))
    tp.tsvd(X)
    best = np.inf
    for _ in range(3):
        torch.cuda.synchronize()
        tp.profile_start()
        tp.tsvd(X)
        torch.cuda.synchronize()
        best = min(best, tp.profile_stop()["jacobi_f32"][0])
    return best


@pytest.mark.parametrize("n1,n2", [(64, 48), (160, 96)])
def test_more_slices_than_rings(n1, n2):
    assert sweeps_ms(n1, n2, 33) < 1.25 * sweeps_ms(n1, n2, 25)


@pytest.mark.parametrize("slices", [13, 17, 33])
@pytest.mark.parametrize("n1,n2", [(64, 48), (130, 96)])
def test_singular_values(n1, n2, slices):
    X = synth.iid_normal((n1, n2, 2 * slices - 2), seed=3)
    S = np.fft.rfft(to_np(tp.tsvd(tp.as_tprod_layout(X))[1]), axis=2)
    ref = np.linalg.svd(np.fft.rfft(X.astype(np.float64), axis=2).transpose(2, 0, 1),
                        compute_uv=False)
    got = np.diagonal(S, axis1=0, axis2=1).real
    assert np.linalg.norm(got - ref) < TOL_FP32 * np.linalg.norm(ref)
