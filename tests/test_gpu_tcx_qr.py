"""t-CX with the picked slices orthonormalised by the Householder QR (full
column rank, at most 96 picks) against the float64 oracle: picks at the edges
of the rule (1, 96 and 97 picks, as many as rows and one more), rows in one
block and in a tree (256, 257, 700), ill-conditioned picks on both sides of the
rank check, and duplicated, zero, tiny and huge slices, which take the SVD.
Tolerance: the repository's for this entry point (1e-5) while the picks'
condition number times float32's rounding stays below it; the ill-conditioned
ones are the data's own neighbours, so their projection is as accurate."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np

pytestmark = pytest.mark.gpu


def project(A, idx):
    """Every Fourier slice of A on the span of its columns idx, in float64."""
    F = np.fft.fft(A.astype(np.float64), axis=2)
    for k in range(A.shape[2]):
        u, s, _ = np.linalg.svd(F[:, idx, k], full_matrices=False)
        keep = s > max(A.shape[0], len(idx)) * np.spacing(s[0]) if s[0] > 0 else s > 0
        u = u[:, keep]
        F[:, :, k] = u @ (u.conj().T @ F[:, :, k])
    return np.fft.ifft(F, axis=2).real


def check(A, idx, scale=1.0, tol=TOL_FP32):
    """A's slices idx picked for certain."""
    import torch
    n2 = A.shape[1]
    p = np.zeros(n2)
    p[idx] = 1.0 / len(idx)
    Z, got, cnt = tp.tcx(tp.as_tprod_layout((A * scale).astype(np.float32)), len(idx), seed=1,
                         prob_mode=tp.TP_PROB_GIVEN,
                         p_given=torch.from_numpy(p).to("cuda"))
    n = int(cnt.item())
    assert n == len(idx) and got[:n].cpu().tolist() == sorted(idx)
    assert rel_fro(to_np(Z) / scale, project(A, sorted(idx))) < tol


@pytest.mark.parametrize("n1,n2,c", [(5, 9, 1), (64, 70, 63), (64, 70, 64), (64, 70, 65), (256, 120, 96),
                                     (256, 120, 97), (257, 60, 40), (700, 120, 96), (33, 40, 17)])
def test_picks(n1, n2, c):
    A = synth.iid_normal((n1, n2, 6), seed=n1)
    check(A, list(range(n2 - c, n2)))


@pytest.mark.parametrize("noise", [1e-1, 1e-3, 1e-4, 1e-5])
@pytest.mark.parametrize("n1", [100, 300])
def test_ill_conditioned(n1, noise):
    rng = np.random.default_rng(1)
    A = np.einsum("irt,rj->ijt", rng.standard_normal((n1, 6, 5)), rng.standard_normal((6, 90)))
    A = (A + noise * rng.standard_normal(A.shape)).astype(np.float32)
    check(A, list(range(40)))


@pytest.mark.parametrize("n1", [48, 300])
def test_rank_deficient_and_scaled(n1):
    A = synth.iid_normal((n1, 40, 4), seed=2)
    check(A, list(range(20)), scale=2.0 ** -44)
    check(A, list(range(20)), scale=2.0 ** 44)
    A[:, 3] = 0          # a zero slice
    check(A, list(range(20)))
    A[:, 5] = A[:, 4]    # and a duplicated one
    check(A, list(range(20)))
