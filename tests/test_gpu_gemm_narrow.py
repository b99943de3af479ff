"""FP32 products with few rows or columns: against the float64 oracle at the
edges of the 32 x 32 tiles, and by device time well under the same product with
64 columns (a third less arithmetic is done at least)."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import tensor_ref
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,n4", [(32, 300, 700), (33, 300, 700), (700, 300, 32), (700, 300, 33),
                                      (1, 257, 900), (900, 257, 1), (31, 1000, 31), (3000, 5, 17)])
def test_product(n1, n2, n4):
    A, B = synth.iid_normal((n1, n2, 18), seed=1), synth.iid_normal((n2, n4, 18), seed=2)
    ref = tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))
    assert rel_fro(to_np(tp.tprod(tp.as_tprod_layout(A), tp.as_tprod_layout(B))), ref) < TOL_FP32


def product_ms(n4):
    import torch
    A, B = (tp.as_tprod_layout(torch.randn(s, device="cuda")) for s in ((2000, 2000, 17), (2000, n4, 17)))
    best = np.inf
    for _ in range(4):
        torch.cuda.synchronize()
        tp.profile_start()
        tp.tprod(A, B)
        torch.cuda.synchronize()
        best = min(best, tp.profile_stop()["cgemm_fp32"][0])
    return best


def test_time_of_few_columns():
    assert product_ms(20) < 0.85 * product_ms(64)
