"""The slice norms' second pass (partial sums of a row added by 64 groups of
threads) against float64: partial counts around the rule that picks it (8) and
around its groups (64) and batches, rows around its four, one row, and values
whose squares cancel nothing.  Tolerance: the norms are float64 sums of float32
squares kept as float pairs, held to 1e-12 as sums of at most 2^24 terms."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from paper_1704_04362_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n3", [1, 8, 9, 63, 64, 65, 128, 129, 513, 1000])
@pytest.mark.parametrize("n1,n2", [(1, 1), (3, 4), (5, 5), (4, 67), (67, 4), (300, 9)])
def test_norms(n1, n2, n3):
    X = synth.iid_normal((n1, n2, n3), seed=n1 + n2 + n3)
    X[0] *= 1e3
    sq = X.astype(np.float64) ** 2
    for which, axes in ((0, (0, 2)), (1, (1, 2))):
        got = tp.slice_norms(tp.as_tprod_layout(X), which).cpu().numpy()
        ref = sq.sum(axis=axes)
        assert np.abs(got - ref).max() <= 1e-12 * ref.max()
        assert (np.abs(got - ref) <= 1e-12 * ref).all()
