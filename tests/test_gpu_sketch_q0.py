"""sketch_spectrum with no and one power iteration, against recorded values.

With q = 0 (and, less so, q = 1) the singular values below about 2^-12 of the largest are resolved as
a group only (the core's Gram matrix is float32), so the order of every sum
before it shows in them at 1e-5 of the spectrum's norm.  Callers compare ranks
and spectra between runs, so the orders are part of the result: the recorded
spectra (tests/golden/sketch_q0.txt, GB300, hexadecimal float32) are to be met
to rounding.  Tolerance: 1e-6 of the norm for q = 0, sixteen float32 roundings of
the largest value and a tenth of the smallest change that another order was seen
to make, and 1e-8 for q = 1, where another order makes 5e-8 at least; equal orders
give equal bits.

The inputs are sums of products of uniform numbers with IEEE operations only, so
that they have the same bits on every machine.
"""
import os

import numpy as np
import pytest

import paper_1704_04362_gb300 as tp

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "sketch_q0.txt")
# n1, n2, n3, l and q where it is not 0: slices of at most and of more than 256 rows; tube lengths with
# small factors, prime and a power of two
CASES = [(150, 190, 21, 40), (300, 120, 17, 44), (290, 90, 16, 36), (96, 130, 32, 48),
         (257, 64, 30, 34), (260, 131, 22, 44, 1), (140, 150, 21, 40, 1), (270, 300, 16, 48, 1)]


def decaying(n1, n2, n3):
    """sum over r of r^-2.5 u_r (outer) v_r (outer) c_r, c_r one at its first
    sample and small beyond."""
    g = np.random.Generator(np.random.PCG64(n1 * n2 + n3))
    X = np.zeros((n3, n2, n1))
    for r in range(1, min(n1, n2) // 2 + 1):
        u, v = 2.0 * g.random(n1) - 1.0, 2.0 * g.random(n2) - 1.0
        c = 0.25 * (2.0 * g.random(n3) - 1.0) / n3
        c[0] += 1.0
        a = 1.0 / (np.float64(r * r) * np.sqrt(np.float64(r)))
        X += (a * c)[:, None, None] * (v[:, None] * u[None, :])[None]
    return X.astype(np.float32)   # storage order


def spectrum(case):
    import torch
    X = torch.from_numpy(decaying(*case[:3])).cuda().permute(2, 1, 0)
    q = case[4] if len(case) > 4 else 0
    return tp.sketch_spectrum(X, case[3], q, seed=5).cpu().numpy()


def recorded():
    out = {}
    with open(GOLDEN) as f:
        for line in f:
            if line.startswith("#"):
                continue
            name, words = line.split(":")
            out[tuple(int(x) for x in name.split())] = np.frombuffer(
                bytes.fromhex(words.strip()), dtype="<f4")
    return out


def test_recorded_spectra_decay_past_the_gram_matrix():
    """The recorded values reach the range in which the order of sums shows."""
    for case in CASES:
        if len(case) > 4:
            continue
        s = recorded()[case].reshape(case[2] // 2 + 1, case[3])
        assert (np.diff(s, axis=1) <= 0).all()
        assert s[:, -1].max() < 2.0 ** -12 * s[:, 0].min()


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES)
def test_values_are_the_recorded_ones(case):
    got, ref = spectrum(case).ravel().astype(np.float64), recorded()[case].astype(np.float64)
    assert np.linalg.norm(got - ref) <= (1e-8 if len(case) > 4 else 1e-6) * np.linalg.norm(ref)


@pytest.mark.gpu
@pytest.mark.parametrize("n3", [3, 5, 6, 7, 9, 11, 12, 15])
def test_short_tubes_match_the_oracle(n3):
    """Lengths whose product has one or two groups of outputs (a flat spectrum,
    which every order of the sums resolves; tolerance of the float32 paths)."""
    from oracle import decomp_ref, philox_ref
    from paper_1704_04362_gb300 import synth
    from tests.util import TOL_FP32, rel_fro
    X = synth.lowrank_np(70, 50, n3, 50, seed=n3, factor="normal")
    omega = philox_ref.sketch_signs(50, 17, n3 // 2 + 1, n3, 4)
    ref = decomp_ref.tsvd_randomized_hat(X.astype(np.float64), 17, 0, 0, omega)[1].T
    got = tp.sketch_spectrum(tp.as_tprod_layout(X), 17, 0, seed=4).cpu().numpy()
    assert rel_fro(got, ref) < TOL_FP32
