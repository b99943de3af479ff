"""Workloads of the t-product library, each through its public Python entry points.

A case names one of the library's uses (``kind``) and its sizes:

tprod       exact t-product A * B
gram        U^T * U of a tall tensor (the paper's tensor-multiplication experiment)
sampled     rt-product: slices of A and B drawn, rescaled and multiplied
rsvd        randomized low-tubal-rank approximation: factors, then U * S * V^T
sketch      plain rank rule: randomized sketch spectrum, per-frequency ranks
tsvd        truncated t-SVD: factors, then the rank-k product U_k * S_k * V_k^T
complete    nuclear-norm ADMM on one tensor (completion, or the robust form)
batch       the same completion on several tensors of uneven sizes in one call
tcx         t-CX: lateral slices drawn, A projected on their span
stages      the slice norms and the mode-3 transforms that a caller composes

Singular vectors are unique only up to a phase (and a rotation inside a
cluster), so the factorisations return S and the approximation U * S * V^T,
which are unique, instead of U and V; the approximation is what the imaging
applications use.  ``exact`` restates every path in float64 with torch and
numpy routines.
"""
import math

import numpy as np
import torch

import paper_1704_04362_gb300 as tp

PRECISIONS = {"fp32": tp.TP_FP32, "tf32x3": tp.TP_TF32X3, "bf16x3": tp.TP_BF16X3}


def listed():
    return [
        # the smallest call of the tests and of the exact-product workload: launches and host work count
        {"name": "tprod_small", "kind": "tprod", "n1": 64, "n2": 48, "n4": 32, "n3": 16,
         "precision": "fp32"},
        # ordinary exact product in the default precision
        {"name": "tprod_fp32", "kind": "tprod", "n1": 600, "n2": 1600, "n4": 500, "n3": 64,
         "precision": "fp32"},
        # U_r^T * U_r of the paper's tensor-multiplication table: long inner dimension, odd tubes
        {"name": "gram_table1", "kind": "gram", "n": 100000, "r": 300, "n3": 5,
         "precision": "bf16x3"},
        # the headline workload: the largest rt-product, split precision
        {"name": "sampled_bf16x3", "kind": "sampled", "n1": 2000, "n2": 4000, "n4": 1500, "n3": 64,
         "c": 400, "precision": "bf16x3", "prob": "norms", "iid": False},
        # an rt-product of odd sizes whose tube length is no power of two, default precision
        {"name": "sampled_ragged", "kind": "sampled", "n1": 611, "n2": 1203, "n4": 389, "n3": 45,
         "c": 150, "precision": "fp32", "prob": "norms", "iid": False},
        # randomized t-SVD of a mass-spectrometry-imaging tensor (long tubes, many frequencies)
        {"name": "rsvd_msi", "kind": "rsvd", "n1": 128, "n2": 128, "n3": 2000, "k": 40, "p": 10,
         "q": 2, "precision": "bf16x3"},
        # the plain rank rule's sketch of a large tensor with a decaying spectrum
        {"name": "sketch_1024", "kind": "sketch", "n1": 1024, "n2": 1024, "n3": 64, "l": 50, "q": 2},
        # truncated t-SVD of the small exact workload
        {"name": "tsvd_small", "kind": "tsvd", "n1": 64, "n2": 48, "n3": 16, "k": 24},
        # completion of one video of the paper's size from half of its entries
        {"name": "complete_video", "kind": "complete", "n1": 144, "n2": 256, "n3": 80, "iters": 10,
         "robust": False, "precision": "fp32"},
        # several videos of uneven size in one call
        {"name": "complete_batch", "kind": "batch", "count": 6, "sizes": 3, "iters": 10,
         "precision": "fp32"},
        # t-CX of an imaging-like tensor
        {"name": "tcx_256", "kind": "tcx", "n1": 256, "n2": 512, "n3": 32, "c": 64},
        # norms and transforms of the face-stack shape, a tube length that is no power of two
        {"name": "stages_faces", "kind": "stages", "n1": 192, "n2": 1140, "n3": 168},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _smooth(n):
    """The largest product of 2, 3, 5 and 7 up to n (long tubes must factor)."""
    while True:
        m = n
        for f in (2, 3, 5, 7):
            while m % f == 0:
                m //= f
        if m == 1:
            return n
        n -= 1


def draw(rng):
    kind = rng.choice(["tprod", "gram", "sampled", "rsvd", "sketch", "tsvd", "complete", "batch",
                       "tcx", "stages"])
    any_precision = rng.choice(list(PRECISIONS))
    if kind == "tprod":
        return {"kind": kind, "n1": _log_int(rng, 16, 600), "n2": _log_int(rng, 16, 1600),
                "n4": _log_int(rng, 16, 500), "n3": _log_int(rng, 2, 128),
                "precision": any_precision}
    if kind == "gram":
        return {"kind": kind, "n": _log_int(rng, 5000, 100000), "r": rng.randint(100, 300),
                "n3": rng.randint(3, 8), "precision": rng.choice(["bf16x3", "tf32x3"])}
    if kind == "sampled":
        n2 = _log_int(rng, 300, 4000)
        return {"kind": kind, "n1": _log_int(rng, 100, 2000), "n2": n2,
                "n4": _log_int(rng, 100, 1500), "n3": _log_int(rng, 4, 64),
                "c": max(8, int(n2 * rng.uniform(0.05, 0.2))), "precision": any_precision,
                "prob": rng.choice(["norms", "norms", "given"]), "iid": rng.random() < 0.2}
    if kind == "rsvd":
        return {"kind": kind, "n1": rng.randint(64, 160), "n2": rng.randint(64, 160),
                "n3": _smooth(_log_int(rng, 64, 2000)), "k": rng.randint(10, 40),
                "p": rng.randint(5, 10), "q": rng.randint(1, 2), "precision": any_precision}
    if kind == "sketch":
        return {"kind": kind, "n1": _log_int(rng, 96, 1024), "n2": _log_int(rng, 96, 1024),
                "n3": _log_int(rng, 16, 64), "l": rng.randint(17, 50), "q": rng.randint(0, 2)}
    if kind == "tsvd":
        n1, n2 = rng.randint(16, 128), rng.randint(16, 96)
        return {"kind": kind, "n1": n1, "n2": n2, "n3": _log_int(rng, 3, 32),
                "k": rng.randint(4, min(n1, n2) // 2)}
    if kind == "complete":
        robust = rng.random() < 0.4
        return {"kind": kind, "n1": rng.randint(64, 192), "n2": rng.randint(64, 256),
                "n3": rng.randint(16, 80), "iters": rng.randint(6, 12), "robust": robust,
                "precision": any_precision}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 4), "sizes": rng.randint(10, 1 << 20),
                "iters": rng.randint(6, 10), "precision": any_precision}
    if kind == "tcx":
        n2 = _log_int(rng, 96, 512)
        return {"kind": kind, "n1": _log_int(rng, 64, 256), "n2": n2, "n3": _log_int(rng, 8, 64),
                "c": rng.randint(16, 64)}
    return {"kind": kind, "n1": _log_int(rng, 50, 200), "n2": _log_int(rng, 50, 1140),
            "n3": _log_int(rng, 4, 256)}


# ---------------------------------------------------------------- inputs
# Storage order is (n3, n2, n1), rows fastest; a logical tensor is its permutation.

def _logical(x):
    return x.contiguous().permute(2, 1, 0)


def _generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _lowrank(g, n1, n2, n3, r, noise, factor="normal"):
    """t-product of random factors of tubal rank r (unit RMS) plus noise, in storage order."""
    if factor == "normal":
        P, Q = _randn(g, n3, r, n1), _randn(g, n3, n2, r)
    else:   # Gamma(2, 1): the sum of two unit exponentials
        def gamma(*s):
            u = torch.rand((2,) + s, generator=g, device="cuda").clamp_min_(1e-12)
            return -torch.log(u).sum(0)
        P, Q = gamma(n3, r, n1), gamma(n3, n2, r)
    X = torch.fft.irfft(torch.fft.rfft(Q, dim=0) @ torch.fft.rfft(P, dim=0), n=n3, dim=0)
    X /= torch.linalg.vector_norm(X) / math.sqrt(X.numel())
    return X.add_(_randn(g, n3, n2, n1), alpha=noise) if noise else X


def _video_sizes(case):
    """(H, W, T) per tensor, uniform from 64 x 64 x 16 up to 480 x 360 x 120."""
    g = np.random.default_rng(case["sizes"])
    return [(int(g.integers(64, 481)), int(g.integers(64, 361)), int(g.integers(16, 121)))
            for _ in range(case["count"])]


def _video(g, n1, n2, n3):
    X = _lowrank(g, n1, n2, n3, 10, 0.01)
    mask = (torch.rand((n3, n2, n1), generator=g, device="cuda") < 0.5).to(torch.uint8)
    return _logical(X), _logical(mask)


def prepare(case, seed):
    kind = case["kind"]
    g = _generator(seed)
    state = {"case": case, "seed": int(seed)}
    if "precision" in case:
        state["precision"] = PRECISIONS[case["precision"]]
    if kind == "batch":
        state["tensors"] = [_video(_generator(seed, i), *s) for i, s in enumerate(_video_sizes(case))]
        return state
    n3 = case["n3"]
    if kind == "gram":
        n, r = case["n"], case["r"]
        # columns near orthonormal with a heavy-tailed row leverage
        lev = torch.exp(0.5 * _randn(g, 1, 1, n))
        U = _randn(g, n3, r, n) * (lev / math.sqrt(n))
        Ut = torch.roll(torch.flip(U.transpose(1, 2), (0,)), 1, 0)   # t-transpose
        state["U"], state["Ut"] = _logical(U), _logical(Ut)
        return state
    n1, n2 = case["n1"], case["n2"]
    if kind == "tprod":
        state["A"], state["B"] = (_logical(_randn(g, n3, n2, n1)),
                                  _logical(_randn(g, n3, case["n4"], n2)))
    elif kind == "sampled":
        state["A"] = _logical(_lowrank(g, n1, n2, n3, 20, 0.01))
        state["B"] = _logical(_lowrank(g, n2, case["n4"], n3, 20, 0.01))
        if case["prob"] == "given":
            state["p"] = torch.full((n2,), 1.0 / n2, dtype=torch.float64, device="cuda")
    elif kind == "rsvd":
        X = _lowrank(g, n1, n2, n3, 15, 0.0, "gamma")
        spikes = torch.rand(X.shape, generator=g, device="cuda") < 1e-3
        height = -5.0 * torch.log(torch.rand(X.shape, generator=g, device="cuda").clamp_min_(1e-12))
        state["X"] = _logical(X + spikes * height + 5e-3 * _randn(g, *X.shape))
    elif kind == "sketch":
        m, h = min(n1, n2) // 2, n3 // 2 + 1
        a = 2.5 + 0.3 * (2.0 * torch.rand((h, 1), generator=g, device="cuda") - 1.0)
        s = torch.arange(1, m + 1, device="cuda", dtype=torch.float32)[None, :] ** (-a)
        V = torch.fft.rfft(_randn(g, n3, n2, m), dim=0) / math.sqrt(n2)
        U = torch.fft.rfft(_randn(g, n3, m, n1), dim=0) / math.sqrt(n1)
        state["X"] = _logical(torch.fft.irfft((V * s[:, None, :]) @ U, n=n3, dim=0))
    elif kind == "complete" and not case["robust"]:
        state["X"], state["mask"] = _video(g, n1, n2, n3)
    elif kind == "complete":
        X = _lowrank(g, n1, n2, n3, 10, 0.0)
        hit = torch.rand(X.shape, generator=g, device="cuda") < 0.1
        state["X"] = _logical(X + hit * (5.0 * _randn(g, *X.shape)))
    elif kind == "tcx":
        state["X"] = _logical(_lowrank(g, n1, n2, n3, 10, 0.01))
    else:   # tsvd, stages
        state["X"] = _logical(_randn(g, n3, n2, n1))
    return state


# ---------------------------------------------------------------- one pass

def _transpose(V):
    """t-transpose: every frontal slice transposed, slices 2 .. n3 reversed."""
    s = V.permute(2, 0, 1)                                    # (n3, rows, columns)
    return _logical(torch.roll(torch.flip(s, (0,)), 1, 0))


def _facewise(U, S, V, n3):
    """U * S * V^T from the library's transforms (tubes of any length)."""
    (ur, ui), (sr, _), (vr, vi) = tp.rdft3(U), tp.rdft3(S), tp.rdft3(V)
    uh = torch.complex(ur, ui).permute(2, 0, 1)               # (h, n1, k)
    vh = torch.complex(vr, -vi).permute(2, 1, 0)              # (h, k, n2): V^H
    d = torch.diagonal(sr, dim1=0, dim2=1)                    # (h, k)
    xh = (vh.transpose(1, 2) * d[:, None, :]) @ uh.transpose(1, 2)   # (h, n2, n1)
    return tp.irdft3(_logical(xh.real), _logical(xh.imag), n3)


def run(state):
    case = state["case"]
    kind = case["kind"]
    prec = state.get("precision")
    if kind == "tprod":
        return {"C": tp.tprod(state["A"], state["B"], precision=prec)}
    if kind == "gram":
        return {"C": tp.tprod(state["Ut"], state["U"], precision=prec)}
    if kind == "sampled":
        p = state.get("p")
        Z, _, count = tp.tprod_sampled(
            state["A"], state["B"], case["c"], seed=state["seed"], precision=prec, p_given=p,
            prob_mode=tp.TP_PROB_AB if p is None else tp.TP_PROB_GIVEN,
            sample_mode=tp.TP_SAMPLE_IID if case["iid"] else tp.TP_SAMPLE_BERNOULLI)
        return {"Z": Z, "count": count}
    if kind == "rsvd":
        U, S, V = tp.tsvd_randomized(state["X"], case["k"], case["p"], case["q"],
                                     seed=state["seed"], precision=prec)
        return {"S": S, "L": _facewise(U, S, V, case["n3"])}
    if kind == "sketch":
        sig = tp.sketch_spectrum(state["X"], case["l"], case["q"], seed=state["seed"])
        return {"sig": sig, "rank": tp.rank_rule(sig, case["l"] - 2)}
    if kind == "tsvd":
        k = case["k"]
        U, S, V = tp.tsvd(state["X"])
        US = tp.tprod(tp.as_tprod_layout(U[:, :k]), tp.as_tprod_layout(S[:k, :k]))
        return {"S": S, "L": tp.tprod(US, _transpose(V[:, :k]))}
    if kind == "complete":
        if case["robust"]:
            L, E, Y, mu = tp.trpca_admm(state["X"], case["iters"], precision=prec)
        else:
            L, E, Y, mu = tp.tcomplete_svt(state["X"], state["mask"], case["iters"],
                                           precision=prec)
        return {"L": L, "E": E, "Y": Y, "mu": mu}
    if kind == "batch":
        todo = [(X, M, torch.zeros_like(X), torch.zeros_like(X), torch.zeros_like(X),
                 torch.full((1,), 1e-3, dtype=torch.float64, device="cuda"))
                for X, M in state["tensors"]]
        done = tp.tcomplete_svt_batched(todo, case["iters"], precision=prec)
        return [{"L": t[2], "E": t[3], "Y": t[4], "mu": t[5]} for t in done]
    if kind == "tcx":
        Z, _, count = tp.tcx(state["X"], case["c"], seed=state["seed"])
        return {"Z": Z, "count": count}
    Xr, Xi = tp.rdft3(state["X"])
    return {"lateral": tp.slice_norms(state["X"], 0), "horizontal": tp.slice_norms(state["X"], 1),
            "Xr": Xr, "Xi": Xi, "back": tp.irdft3(Xr, Xi, case["n3"])}


# ---------------------------------------------------------------- what a pass cannot do without

def _admm_work(sizes, iters):
    b = f = 0
    for n1, n2, n3 in sizes:
        n, m, w, h = n1 * n2 * n3, min(n1, n2), max(n1, n2), n3 // 2 + 1
        b += n * (4 + 1 + 12)   # data and mask read, the state written
        # per slice and iteration: the product with the leading directions and the rebuild
        f += iters * (h * 2 * 8 * m * w * min(10, m) + 2 * 2.5 * n * math.log2(max(2, n3)))
    return {"bytes": b, "flops": f}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        return _admm_work(_video_sizes(case), case["iters"])
    n3 = case["n3"]
    h = n3 // 2 + 1
    real = 2 - n3 % 2   # real slices
    face = 8 * (h - real) + 2 * real   # flops of one complex multiply-add over the half spectrum
    fft = 2.5 * n3 * math.log2(max(2, n3))
    if kind == "gram":
        n, r = case["n"], case["r"]
        return {"bytes": 4 * n3 * (2 * n * r + r * r),
                "flops": face * n * r * r + fft * (2 * n * r + r * r)}
    n1, n2 = case["n1"], case["n2"]
    if kind == "tprod":
        n4 = case["n4"]
        el = n1 * n2 + n2 * n4 + n1 * n4
        return {"bytes": 4 * n3 * el, "flops": face * n1 * n2 * n4 + fft * el}
    if kind == "sampled":
        n4, c = case["n4"], case["c"]
        read = n1 * n2 + n2 * n4 if case["prob"] == "norms" else c * (n1 + n4)
        return {"bytes": 4 * n3 * (read + n1 * n4),
                "flops": face * n1 * c * n4 + fft * (n1 * c + c * n4 + n1 * n4)
                + (2 * n3 * read if case["prob"] == "norms" else 0)}
    if kind == "rsvd":
        k, l, q = case["k"], case["k"] + case["p"], case["q"]
        el = 2 * n1 * n2 + k * (n1 + n2)
        return {"bytes": 4 * n3 * (2 * n1 * n2 + k * k),
                "flops": face * (n1 * n2 * (l * (2 * q + 2) + k) + (n1 + n2) * l * l * (q + 1))
                + fft * el}
    if kind == "sketch":
        l, q = case["l"], case["q"]
        return {"bytes": 4 * (n1 * n2 * n3 + h * l),
                "flops": face * (n1 * n2 * l * (2 * q + 2) + (n1 + n2) * l * l * (q + 1))
                + fft * n1 * n2}
    if kind == "tsvd":
        m, k = min(n1, n2), case["k"]
        return {"bytes": 4 * n3 * (2 * n1 * n2 + m * m),
                "flops": face * (6 * max(n1, n2) * m * m + n1 * n2 * k)
                + fft * (2 * n1 * n2 + m * (n1 + n2))}
    if kind == "complete":
        return _admm_work([(n1, n2, n3)], case["iters"])
    if kind == "tcx":
        c = min(case["c"], n1, n2)
        return {"bytes": 4 * n3 * 2 * n1 * n2,
                "flops": face * (2 * n1 * c * c + 2 * n1 * n2 * c) + 2 * fft * n1 * n2}
    n = n1 * n2
    return {"bytes": 4 * n * (2 * n3 + 2 * h), "flops": n * (2 * fft + 4 * n3)}


# ---------------------------------------------------------------- the same in 64 bits

def _philox(counter, stream, word3, seed):
    """Words 0 and 1 of Philox4x32-10 (Salmon et al., SC'11) for 64-bit counters."""
    u = np.uint64
    mask = u(0xFFFFFFFF)
    c0, c1 = counter & mask, counter >> u(32)
    c2, c3 = np.full_like(c0, u(stream)), np.full_like(c0, u(word3))
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        a, b = u(0xD2511F53) * c0, u(0xCD9E8D57) * c2
        c0, c1, c2, c3 = (b >> u(32)) ^ c1 ^ u(k0), b & mask, (a >> u(32)) ^ c3 ^ u(k1), a & mask
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1


def _picks(p, c, seed):
    """Bernoulli picks of slices with probability min(1, c p): indices and 1/sqrt(q)."""
    q = np.minimum(1.0, c * p)
    x0, x1 = _philox(np.arange(len(q), dtype=np.uint64), 0, 0, seed)
    u = (x0 >> np.uint64(5) << np.uint64(26)) | (x1 >> np.uint64(6))
    idx = np.nonzero(u < np.floor(q * 2.0 ** 53).astype(np.uint64))[0]
    return torch.from_numpy(idx).cuda(), torch.from_numpy(1.0 / np.sqrt(q[idx])).cuda()


def _store(x):
    """Storage order (n3, n2, n1) of a logical tensor, float64."""
    return x.permute(2, 1, 0).double()


def _product(A, B, n3):
    """t-product of storage-order tensors: the slices are transposes, so B_hat A_hat."""
    return torch.fft.irfft(torch.fft.rfft(B, dim=0) @ torch.fft.rfft(A, dim=0), n=n3, dim=0)


def _orth(Y):
    for _ in range(2):   # Cholesky QR, twice
        R = torch.linalg.cholesky(Y.mH @ Y).mH
        Y = torch.linalg.solve_triangular(R, Y, upper=True, left=False)
    return Y


def _range_svd(Xh, l, q, n3, seed):
    """Randomized range finder of (h, n1, n2) slices; Q, singular values and left
    vectors of Q^H Xh, descending."""
    h, _, n2 = Xh.shape
    x0, x1 = _philox(np.arange(n2 * l * h, dtype=np.uint64), 2, 0, seed)
    s0, s1 = (torch.from_numpy(1.0 - 2.0 * (x >> np.uint64(31)).astype(np.float64)).cuda()
              .view(h, l, n2).transpose(1, 2) for x in (x0, x1))
    omega = torch.complex(s0, s1) / math.sqrt(2.0)
    for f in [0] + ([h - 1] if n3 % 2 == 0 else []):
        omega[f] = s0[f].to(omega.dtype)
    Q = _orth(Xh @ omega)
    for _ in range(q):
        Q = _orth(Xh @ _orth(Xh.mH @ Q))
    B = Q.mH @ Xh
    ev, W = torch.linalg.eigh(B @ B.mH)
    return Q, ev.flip(1).clamp_min(0).sqrt(), W.flip(2), B


def _fdiag(s, n3):
    """f-diagonal tensor (m, m, n3) of the half-spectrum singular values (h, m)."""
    return torch.diag_embed(torch.fft.irfft(s.to(torch.complex128), n=n3, dim=0)).permute(1, 2, 0)


def _shrink(X, tau, n3):
    """Tensor singular value thresholding of a storage-order tensor."""
    Xh = torch.fft.rfft(X, dim=0)
    wide = Xh.shape[1] < Xh.shape[2]
    G = Xh @ Xh.mH if wide else Xh.mH @ Xh
    ev, W = torch.linalg.eigh(G)
    s = ev.clamp_min(0).sqrt()
    P = (W * ((s - tau).clamp_min(0) / s.clamp_min(1e-300)).unsqueeze(1)) @ W.mH
    return torch.fft.irfft(P @ Xh if wide else Xh @ P, n=n3, dim=0)


def _admm(X, mask, iters, n3):
    """Nuclear-norm ADMM (mu0 = 1e-3, rho = 1.1), storage order; mask None is the robust form."""
    lam = 1.0 / math.sqrt(max(X.shape[1], X.shape[2]) * n3)
    if mask is not None:
        X = torch.where(mask, X, torch.zeros_like(X))
    L = E = Y = torch.zeros_like(X)
    mu = 1e-3
    for _ in range(iters):
        L = _shrink(X - E - Y / mu, 1.0 / mu, n3)
        E = X - L - Y / mu
        E = (torch.where(mask, torch.zeros_like(E), E) if mask is not None
             else torch.sign(E) * (E.abs() - lam / mu).clamp_min(0))
        Y = Y + mu * (L + E - X)
        mu = min(1.1 * mu, 1e10)
    L, E, Y = (t.permute(2, 1, 0) for t in (L, E, Y))
    return {"L": L, "E": E, "Y": Y, "mu": torch.tensor([mu], dtype=torch.float64)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" or (kind == "complete" and case["n3"] * case["iters"] > 1000) or (
            kind == "sampled" and case["iid"]):
        return None
    s = prepare(case, seed)
    n3 = case["n3"]
    if kind == "tprod":
        return {"C": _product(_store(s["A"]), _store(s["B"]), n3).permute(2, 1, 0)}
    if kind == "gram":
        return {"C": _product(_store(s["Ut"]), _store(s["U"]), n3).permute(2, 1, 0)}
    if kind == "sampled":
        A, B = s["A"].permute(2, 1, 0), s["B"].permute(2, 1, 0)
        if case["prob"] == "given":
            p = s["p"].cpu().numpy()
        else:
            a = torch.stack([x.double().square().sum(1) for x in A]).sum(0).sqrt()
            b = torch.stack([x.double().square().sum(0) for x in B]).sum(0).sqrt()
            p = (a * b / (a * b).sum()).cpu().numpy()
        idx, d = _picks(p, case["c"], s["seed"])
        Z = _product(A[:, idx, :].double() * d[None, :, None], B[:, :, idx].double() * d, n3)
        return {"Z": Z.permute(2, 1, 0), "count": None}
    if kind == "tcx":
        X = s["X"].permute(2, 1, 0)
        a = X.double().square().sum((0, 2))
        idx, d = _picks((a / a.sum()).cpu().numpy(), case["c"], s["seed"])
        Xh = torch.fft.rfft(X.double(), dim=0).transpose(1, 2)            # (h, n1, n2)
        U, sv, _ = torch.linalg.svd(Xh[:, :, idx] * d, full_matrices=False)
        keep = sv > max(Xh.shape[1], len(idx)) * 2.0 ** -52 * sv[:, :1]
        U = U * keep[:, None, :]
        Z = torch.fft.irfft(U @ (U.mH @ Xh), n=n3, dim=0)
        return {"Z": Z.permute(1, 2, 0), "count": None}
    if kind == "complete":
        M = None if case["robust"] else s["mask"].permute(2, 1, 0).bool()
        return _admm(_store(s["X"]), M, case["iters"], n3)
    X = _store(s["X"])
    if kind == "stages":
        Xh = torch.fft.rfft(X, dim=0).permute(2, 1, 0)
        return {"lateral": X.square().sum((0, 2)), "horizontal": X.square().sum((0, 1)),
                "Xr": Xh.real, "Xi": Xh.imag, "back": X.permute(2, 1, 0)}
    Xh = torch.fft.rfft(X, dim=0).transpose(1, 2)                         # (h, n1, n2)
    if kind == "tsvd":
        U, sv, Vh = torch.linalg.svd(Xh, full_matrices=False)
        k = case["k"]
        L = torch.fft.irfft((U[:, :, :k] * sv[:, None, :k]) @ Vh[:, :k], n=n3, dim=0)
        return {"S": _fdiag(sv, n3), "L": L.permute(1, 2, 0)}
    if kind == "sketch":
        return {"sig": _range_svd(Xh, case["l"], case["q"], n3, s["seed"])[1], "rank": None}
    k = case["k"]
    Q, sv, W, B = _range_svd(Xh, k + case["p"], case["q"], n3, s["seed"])
    W = W[:, :, :k]
    L = torch.fft.irfft((Q @ W) @ (W.mH @ B), n=n3, dim=0)
    return {"S": _fdiag(sv[:, :k], n3), "L": L.permute(1, 2, 0)}
