"""The ADMM's thresholding from kept vectors in runs that outgrow it: where its
attempts fail (noise-free data once tau nears the residuals' floor, noisy data
once the noise passes tau) they are spaced out instead of repeated in every
iteration, and the iterates stay those of the float64 oracle (1e-4 after many
iterations, as the other long runs are held); while they succeed, the Jacobi has
nothing to do."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp
from oracle import completion_ref
from paper_1704_04362_gb300 import binding, synth
from tests.util import rel_fro, to_np

pytestmark = pytest.mark.gpu


def data(n1, n2, n3, rank, noise):
    X = synth.lowrank_np(n1, n2, n3, rank, seed=n1, noise=noise)
    mask = (np.random.default_rng(n2).random(X.shape) < 0.5).astype(np.uint8)
    return X, np.asfortranarray(mask)


def device_ms(X, mask, iters):
    """Device time of the run's kernels by name, after a run that warms up."""
    import torch
    Xd, Md = tp.as_tprod_layout(X), tp.as_tprod_layout(mask, torch.uint8)
    tp.tcomplete_svt(Xd, Md, iters)
    torch.cuda.synchronize()
    tp.profile_start()
    tp.tcomplete_svt(Xd, Md, iters)
    torch.cuda.synchronize()
    return {k: v[0] for k, v in tp.profile_stop().items()}


def test_failing_attempts_are_spaced_out():
    X, mask = data(96, 64, 8, 5, 0.0)
    early, before, after = (device_ms(X, mask, n)["svt_top"] for n in (60, 110, 170))
    assert after - before < early   # 2.4 times it with an attempt in every iteration


@pytest.mark.parametrize("n1,n2,n3,rank,noise,iters", [(96, 64, 4, 5, 0.0, 130),
                                                       (90, 80, 4, 6, 0.01, 90)])
def test_iterates_past_the_kept_vectors(n1, n2, n3, rank, noise, iters):
    import torch
    X, mask = data(n1, n2, n3, rank, noise)
    L, E, _, _ = tp.tcomplete_svt(tp.as_tprod_layout(X), tp.as_tprod_layout(mask, torch.uint8), iters)
    Lr, Er, _, _ = completion_ref.tcomplete_svt(X.astype(np.float64), mask, iters)
    assert rel_fro(to_np(L), Lr) <= 1e-4 and rel_fro(to_np(E), Er) <= 1e-4


def test_low_rank_slices_leave_the_jacobi_idle(monkeypatch):
    X, mask = data(144, 100, 8, 5, 0.0)
    kept = device_ms(X, mask, 10)
    plain = binding._opts

    def less(op, dims, *args, **kw):   # no room for the kept vectors: all slices to the Jacobi
        import ctypes
        o = plain(op, dims, *args, **kw)
        d = (ctypes.c_int64 * len(dims))(*dims)
        o.workspace_bytes = binding.lib().tp_workspace_query(
            op, ctypes.addressof(d), len(dims), ctypes.byref(o)) - 256
        return o

    monkeypatch.setattr(binding, "_opts", less)
    without = device_ms(X, mask, 10)
    assert "svt_top" not in without
    assert kept["jacobi_f32"] < 0.2 * without["jacobi_f32"]
