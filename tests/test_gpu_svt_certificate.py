"""The thresholding's certificate where it is all that stands between a missed
singular value and the result: the data have one right singular vector that is
orthogonal to every starting vector of the kept block (the signs of a hash,
restated here), so that the block converges on the others and never sees it, and
the Cholesky factorisation has to refuse the slice.  Without it the whole
direction would be missing from L (a tenth and more of its norm; tolerance of
the float32 paths).  A twin whose vector is not orthogonal to the start is found
the ordinary way."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from tests.util import TOL_FP32, rel_fro, to_np

pytestmark = pytest.mark.gpu
KEPT = 32


def start_block(q):
    k, c = np.meshgrid(np.arange(q, dtype=np.uint32), np.arange(KEPT, dtype=np.uint32), indexing="ij")
    with np.errstate(over="ignore"):
        x = k * np.uint32(0x9E3779B1) + c * np.uint32(0x85EBCA77) + np.uint32(0x165667B1)
        x ^= x >> np.uint32(15)
        x *= np.uint32(0x2C1B3C6D)
        x ^= x >> np.uint32(13)
    return np.where(x & np.uint32(0x8000), -1.0, 1.0)


@pytest.mark.parametrize("hidden", [True, False])
@pytest.mark.parametrize("p,q", [(64, 48), (80, 80), (130, 100)])
def test_a_direction_the_block_misses(p, q, hidden):
    import torch
    rng = np.random.default_rng(q)
    S = start_block(q)
    # the last right singular vector: in the null space of S^T, or anywhere
    null = np.linalg.svd(S.T)[2][KEPT:]
    v = null.T @ rng.standard_normal(q - KEPT) if hidden else rng.standard_normal(q)
    V = np.linalg.qr(np.column_stack([v, rng.standard_normal((q, 5))]))[0]
    U = np.linalg.qr(rng.standard_normal((p, 6)))[0]
    s = np.array([5.0, 9.0, 8.0, 7.5, 7.0, 6.0])
    tau = 2.0
    X = np.asfortranarray(((U * s) @ V.T)[:, :, None].astype(np.float32))
    mask = torch.ones((1, q, p), dtype=torch.uint8, device="cuda").permute(2, 1, 0)
    L = to_np(tp.tcomplete_svt(tp.as_tprod_layout(X), mask, 1, mu0=1.0 / tau)[0])[:, :, 0]
    assert rel_fro(L, (U * (s - tau)) @ V.T) <= TOL_FP32
