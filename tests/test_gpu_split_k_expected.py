"""Sampled tensor-core products with few output tiles: K is cut by the picks to
expect, not by its capacity, and parts past the picks' chunks are neither written
nor added.  Results against the float64 oracle (the precision's tolerance) with
fewer, as many and more picks than expected; one chunk of expected picks (128
tf32 or 256 bf16 elements) launches no second pass."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import tensor_ref
from paper_1704_04362_gb300 import synth
from tests.util import rel_fro, to_np, tol_for

pytestmark = pytest.mark.gpu
N2 = 1500


def sampled(kept, c, prec):
    """Slices `kept` picked for certain (probabilities 1 / c, or 0), c expected."""
    import torch
    A, B = synth.iid_normal((60, N2, 3), seed=3), synth.iid_normal((N2, 50, 3), seed=4)
    p = np.zeros(N2)
    p[kept] = 1.0 / c
    tp.profile_start()
    Z, idx, cnt = tp.tprod_sampled(tp.as_tprod_layout(A), tp.as_tprod_layout(B), c, seed=6,
                                   precision=prec, prob_mode=tp.TP_PROB_GIVEN,
                                   p_given=torch.from_numpy(p).cuda())
    torch.cuda.synchronize()
    names = tp.profile_stop()
    assert int(cnt.item()) == len(kept)
    ref = tensor_ref.tprod(A[:, kept].astype(np.float64), B[kept].astype(np.float64))
    assert rel_fro(to_np(Z), ref) < tol_for(prec) if len(kept) else not np.any(to_np(Z))
    return names


@pytest.mark.parametrize("prec", [tp.TP_TF32X3, tp.TP_BF16X3])
@pytest.mark.parametrize("picks,c", [(0, 600), (1, 1400), (300, 1400), (257, 300), (900, 900),
                                     (1200, 600), (1500, 1500)])
def test_picks_against_expected(picks, c, prec):
    sampled(np.arange(N2)[:picks], c, prec)


@pytest.mark.parametrize("prec,chunk", [(tp.TP_TF32X3, 128), (tp.TP_BF16X3, 256)])
def test_one_chunk_is_not_cut(prec, chunk):
    assert "cgemm_parts" not in sampled(np.arange(chunk), chunk, prec)
    assert "cgemm_parts" in sampled(np.arange(4 * chunk), 4 * chunk, prec)
