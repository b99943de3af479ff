"""The one-launch product of small tensors against the float64 oracle: every
tube length it takes (1 .. 16) and one more, sizes around its 8 x 8 tiles and
16-deep chunks, the edges of its rule (4096 deep, 256 tiles), infinities, and an
output that shares memory with an operand (which takes the general path).
Tolerance: the repository's for FP32."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import tensor_ref
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np

pytestmark = pytest.mark.gpu


def check(n1, n2, n4, n3):
    A = synth.iid_normal((n1, n2, n3), seed=1)
    B = synth.iid_normal((n2, n4, n3), seed=2)
    C = tp.tprod(tp.as_tprod_layout(A), tp.as_tprod_layout(B))
    assert rel_fro(to_np(C), tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))) < TOL_FP32


@pytest.mark.parametrize("n3", list(range(1, 18)))
@pytest.mark.parametrize("n1,n2,n4", [(1, 1, 1), (8, 16, 8), (9, 17, 7), (64, 48, 32)])
def test_lengths(n1, n2, n4, n3):
    check(n1, n2, n4, n3)


@pytest.mark.parametrize("n1,n2,n4", [(7, 15, 9), (17, 33, 8), (8, 128, 24), (128, 40, 128),
                                      (129, 40, 128), (2048, 3, 8), (3, 5, 2049), (100, 127, 101),
                                      (9, 4096, 10), (9, 4097, 10)])
def test_edges(n1, n2, n4):
    check(n1, n2, n4, 6)


def test_infinity_stays_in_its_row():
    A = synth.iid_normal((20, 18, 5), seed=3)
    B = synth.iid_normal((18, 19, 5), seed=4)
    A[3, 2, 1] = np.inf
    got = to_np(tp.tprod(tp.as_tprod_layout(A), tp.as_tprod_layout(B)))
    A[3] = 0
    ref = tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))
    rows = np.arange(20) != 3
    assert rel_fro(got[rows], ref[rows]) < TOL_FP32
    assert not np.isfinite(got[3]).any()


def test_output_over_an_operand():
    A = synth.iid_normal((24, 24, 8), seed=5)
    B = synth.iid_normal((24, 24, 8), seed=6)
    ref = tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))
    Ad, Bd = tp.as_tprod_layout(A), tp.as_tprod_layout(B)
    tp.tprod(Ad, Bd, C=Ad)
    assert rel_fro(to_np(Ad), ref) < TOL_FP32
    Ad = tp.as_tprod_layout(A)
    tp.tprod(Ad, Bd, C=Bd)
    assert rel_fro(to_np(Bd), ref) < TOL_FP32
