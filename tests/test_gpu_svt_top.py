"""The ADMM's thresholding of slices with few singular values above the
threshold (vectors kept from iteration to iteration, certified by a Cholesky
factorisation) against the float64 oracle: slice widths at the edges of its
range (48 .. 384) and of its blocks of 16 and 32, wide and tall slices, data
whose rank is above the number of vectors it keeps (those slices take the
Jacobi), a rank at the edge, noise at the threshold, a zero tensor, and the
three precisions.  Tolerance: one iteration is held to its precision's bound
(1e-5; 5e-5 for the bf16 form) and thresholding is non-expansive, so k
iterations are held to k times that (60 iterations to 1e-4, as the repository
holds its longer runs)."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import completion_ref
from paper_1704_04362_gb300 import synth
from tests.util import TOL_FP32, rel_fro, to_np, tol_for

pytestmark = pytest.mark.gpu


def run(X, mask, iters, mu0, precision=tp.TP_FP32, batch=False):
    import torch
    Xd = tp.as_tprod_layout(X)
    Md = tp.as_tprod_layout(mask, torch.uint8)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    if batch:
        z = [torch.zeros_like(Xd) for _ in range(3)]
        mu = torch.full((1,), mu0, dtype=torch.float64, device="cuda")
        tp.tcomplete_svt_batched([(Xd, Md, *z, mu)], iters, status=st, precision=precision)
        L, E = z[:2]
    else:
        L, E, _, _ = tp.tcomplete_svt(Xd, Md, iters, mu0=mu0, status=st, precision=precision)
    assert int(st.item()) == 0
    return to_np(L), to_np(E)


def compare(X, mask, iters, mu0, precision=tp.TP_FP32, batch=False):
    L, E = run(X, mask, iters, mu0, precision, batch)
    Lr, Er, _, _ = completion_ref.tcomplete_svt(X.astype(np.float64), mask, iters, mu0=mu0)
    tol = iters * tol_for(precision)
    assert rel_fro(L, Lr) <= tol if np.any(Lr) else not np.any(L)
    assert rel_fro(E, Er) <= tol if np.any(Er) else not np.any(E)


def threshold(X, frac):
    """mu0 whose first threshold is `frac` of the largest singular value."""
    s = np.linalg.norm(np.fft.rfft(X, axis=2)[:, :, 0], 2)
    return 1.0 / (frac * s)


@pytest.mark.parametrize("n1,n2,n3", [(47, 60, 3), (48, 48, 4), (49, 70, 3), (65, 64, 2),
                                      (100, 97, 3), (130, 129, 3), (384, 385, 2), (385, 400, 2),
                                      (400, 208, 1)])
def test_widths(n1, n2, n3):
    X = synth.lowrank_np(n1, n2, n3, 4, seed=n1, noise=0.05)
    mask = (np.random.default_rng(n2).random(X.shape) < 0.6).astype(np.uint8)
    compare(X, np.asfortranarray(mask), 4, threshold(X, 0.3))


@pytest.mark.parametrize("rank", [1, 25, 26, 27, 31, 32, 60])
@pytest.mark.parametrize("precision", [tp.TP_FP32, tp.TP_BF16X3])
def test_rank_at_the_edge_of_the_kept_vectors(rank, precision):
    X = synth.lowrank_np(90, 80, 4, rank, seed=rank)
    mask = np.ones(X.shape, dtype=np.uint8, order="F")
    compare(X, mask, 3, threshold(X, 0.05), precision)


@pytest.mark.parametrize("batch", [False, True])
def test_noise_at_the_threshold(batch):
    # the largest noise singular values lie on both sides of the threshold
    X = synth.iid_normal((96, 72, 5), seed=7)
    s = np.linalg.svd(np.fft.rfft(X, axis=2)[:, :, 1], compute_uv=False)
    mask = np.ones(X.shape, dtype=np.uint8, order="F")
    compare(X, mask, 2, 1.0 / s[3], batch=batch)


def test_many_iterations_down_to_a_small_threshold():
    X = synth.lowrank_np(70, 64, 6, 5, seed=3, noise=0.01)
    mask = (np.random.default_rng(1).random(X.shape) < 0.5).astype(np.uint8)
    L, E = run(X, np.asfortranarray(mask), 60, 1e-3)
    Lr, Er, _, _ = completion_ref.tcomplete_svt(X.astype(np.float64), mask, 60)
    assert rel_fro(L, Lr) <= 1e-4 and rel_fro(E, Er) <= 1e-4


@pytest.mark.parametrize("scale", [0.0, 1e-6, 1e6])
def test_zero_and_scaled_data(scale):
    X = synth.lowrank_np(60, 56, 4, 3, seed=5)
    mu0 = threshold(X, 0.3) / (scale or 1.0)
    X = np.asfortranarray((X * scale).astype(np.float32))
    mask = np.ones(X.shape, dtype=np.uint8, order="F")
    L, E = run(X, mask, 2, mu0)
    Lr, _, _, _ = completion_ref.tcomplete_svt(X.astype(np.float64), mask, 2, mu0=mu0)
    assert rel_fro(L, Lr) <= 2 * TOL_FP32 if scale else not np.any(L)
    assert not np.any(E)


@pytest.mark.parametrize("short", [0, 256, 1 << 30])
def test_a_workspace_without_the_kept_vectors(short, monkeypatch):
    """256 bytes fewer than asked for: every slice takes the Jacobi; far too
    few are refused."""
    from paper_1704_04362_gb300 import binding
    X = synth.lowrank_np(70, 64, 6, 4, seed=3, noise=0.02)
    mask = np.asfortranarray((np.random.default_rng(1).random(X.shape) < 0.6).astype(np.uint8))
    mu0 = threshold(X, 0.3)
    plain = binding._opts

    def less(op, dims, *args, **kw):
        import ctypes
        o = plain(op, dims, *args, **kw)
        d = (ctypes.c_int64 * len(dims))(*dims)
        need = binding.lib().tp_workspace_query(op, ctypes.addressof(d), len(dims), ctypes.byref(o))
        o.workspace_bytes = max(need - short, 0)
        return o

    monkeypatch.setattr(binding, "_opts", less)
    if short > 256:
        with pytest.raises(Exception):
            run(X, mask, 4, mu0)
        return
    compare(X, mask, 4, mu0)
    compare(X, mask, 4, mu0, batch=True)
