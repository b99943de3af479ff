"""Tensor-core products with few output tiles (K cut into parts whose sums are
added afterwards) against the float64 oracle: K around the accumulation chunks
(256 bf16 and 128 tf32 elements) and around as many parts as chunks, sizes at
the tile's edges, a sampled product whose picks leave parts empty, and a
workspace without room for the parts.  Tolerances: the precision's own."""
import ctypes

import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import sampling_ref, tensor_ref
from paper_1704_04362_gb300 import binding, synth
from tests.util import rel_fro, to_np, tol_for

pytestmark = pytest.mark.gpu
PRECISIONS = [tp.TP_TF32X3, tp.TP_BF16X3]


def product(A, B, prec, short=0):
    """C = A * B; short: bytes fewer than the workspace query asks for."""
    import torch
    A, B = tp.as_tprod_layout(A), tp.as_tprod_layout(B)
    n1, n2, n3 = A.shape
    n4 = B.shape[1]
    C = binding.empty_tensor(n1, n4, n3)
    o = binding._opts(binding.TP_OP_TPROD, (n1, n2, n4, n3), prec)
    d = (ctypes.c_int64 * 4)(n1, n2, n4, n3)
    o.workspace_bytes = int(binding.lib().tp_workspace_query(
        binding.TP_OP_TPROD, ctypes.cast(d, ctypes.c_void_p), 4, ctypes.byref(o))) - short
    rc = binding.lib().tprod(ctypes.c_void_p(A.data_ptr()), ctypes.c_void_p(B.data_ptr()),
                        ctypes.c_void_p(C.data_ptr()), n1, n2, n4, n3, ctypes.byref(o),
                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return rc, C


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("n1,n4", [(1, 1), (40, 70), (129, 65)])
@pytest.mark.parametrize("K", [100, 128, 129, 256, 257, 511, 513, 2000, 20001])
def test_product(K, n1, n4, prec):
    A = synth.iid_normal((n1, K, 3), seed=1)
    B = synth.iid_normal((K, n4, 3), seed=2)
    ref = tensor_ref.tprod(A.astype(np.float64), B.astype(np.float64))
    rc, C = product(A, B, prec)
    assert rc == 0 and rel_fro(to_np(C), ref) < tol_for(prec)
    if K >= 512:   # too little room for the parts: the product goes without them
        rc, C = product(A, B, prec, short=256)
        assert rc == 0 and rel_fro(to_np(C), ref) < tol_for(prec)
        parts = 2 * 4 * n1 * n4 * 2 * min(64, -(-K // (128 if prec == tp.TP_TF32X3 else 256)))
        rc, C = product(A, B, prec, short=2 * parts + (1 << 13))
        assert rc != 0


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("c", [3, 130, 900])
def test_sampled(c, prec):
    A = synth.iid_normal((50, 2000, 4), seed=3)
    B = synth.iid_normal((2000, 40, 4), seed=4)
    Z, _, _ = tp.tprod_sampled(tp.as_tprod_layout(A), tp.as_tprod_layout(B), c, seed=6,
                               precision=prec)
    Zr, _, _ = sampling_ref.tprod_sampled(A, B, c, 6)
    assert rel_fro(to_np(Z), Zr) < tol_for(prec)
