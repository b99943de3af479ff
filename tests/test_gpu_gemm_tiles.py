"""The FP32 facewise product at the edges of its tiles (rows and columns around
32, 64 and 128) and of its K stages, aligned and unaligned leading dimensions,
against the float64 oracle at the repository's FP32 tolerance."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import tensor_ref
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n4", [1, 31, 33, 64, 65, 130])
@pytest.mark.parametrize("n1", [1, 32, 63, 65, 127, 260])
@pytest.mark.parametrize("K", [1, 15, 16, 17, 33, 257])
def test_tiles(n1, n4, K):
    A = synth.iid_normal((n1, K, 4), seed=1)
    B = synth.iid_normal((K, n4, 4), seed=2)
    C = tp.tprod(tp.as_tprod_layout(A), tp.as_tprod_layout(B))
    ref = tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))
    assert rel_fro(to_np(C), ref) < TOL_FP32
