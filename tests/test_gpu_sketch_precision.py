"""Singular values of sketch_spectrum on tall slices (more than 256 rows) with a
power iteration, against the float64 range finder: the last orthonormalisation is in float64, so
what is left is the rounding of float32 operands.

Tolerance on the mean over the cases of the relative error of the spectrum (its
norm is the leading values'): 8e-8.  Rounding the stored value: 2^-24 / sqrt(3) =
3.4e-8 root mean square; the length of the core's float32 vector of up to 36
rotated entries, 3e-8; the tubes' transform, 3e-8; float32 products of 300 to 600
terms averaged over as many columns, 2e-8: together 6e-8, and a third more for
a mean over few cases.  An orthonormalisation in float32 adds its own 1e-7.
"""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import decomp_ref, philox_ref
from tests.test_gpu_sketch_q0 import decaying

pytestmark = pytest.mark.gpu


def test_mean_error_of_tall_sketches():
    errors = []
    for n1, n2, n3, l in [(300, 320, 17, 24), (420, 280, 24, 30), (520, 400, 16, 27),
                          (600, 270, 20, 33), (290, 500, 25, 20), (480, 480, 18, 36)]:
        X = np.asfortranarray(decaying(n1, n2, n3).transpose(2, 1, 0))
        omega = philox_ref.sketch_signs(n2, l, n3 // 2 + 1, n3, 3)
        ref = decomp_ref.tsvd_randomized_hat(X.astype(np.float64), l, 0, 1, omega)[1].T
        got = tp.sketch_spectrum(tp.as_tprod_layout(X), l, 1, seed=3).double().cpu().numpy()
        errors.append(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert np.mean(errors) <= 8e-8, errors
