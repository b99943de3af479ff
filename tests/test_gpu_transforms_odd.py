"""Inverse transforms of odd lengths on both sides of the line between the FFT and
the product, against float64 (1e-6 of the result's norm: float32 sums of up to
40 folded terms, 2^-24 sqrt(40) = 4e-7, doubled); and, by device time, neither
odd composite lengths nor those just above 16 slower than their prime neighbours,
whose arithmetic is the same or more."""
import numpy as np
import pytest

import paper_1704_04362_gb300 as tp

pytestmark = pytest.mark.gpu


def spectrum(rows, n3):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(rows + n3)
    x = torch.randn((n3, rows), generator=g, device="cuda", dtype=torch.float64)
    h = torch.fft.rfft(x, dim=0)
    lay = [v.float().contiguous().view(n3 // 2 + 1, 1, rows).permute(2, 1, 0) for v in (h.real, h.imag)]
    return x, lay


@pytest.mark.parametrize("rows,n3", [(49151, 45), (49152, 45), (49153, 21), (50001, 25), (49160, 47),
                                     (163839, 63), (163840, 63), (163843, 49), (170001, 77),
                                     (60000, 17), (4097, 19), (16384, 23)])
def test_inverse(rows, n3):
    import torch
    x, (re, im) = spectrum(rows, n3)
    got = tp.irdft3(re, im, n3).permute(2, 1, 0).reshape(n3, rows).double()
    assert torch.linalg.vector_norm(got - x) <= 1e-6 * torch.linalg.vector_norm(x)


def inverse_ms(rows, n3):
    import torch
    _, (re, im) = spectrum(rows, n3)
    best = np.inf
    for _ in range(5):
        torch.cuda.synchronize()
        tp.profile_start()
        for _ in range(4):
            tp.irdft3(re, im, n3)
        torch.cuda.synchronize()
        best = min(best, sum(v[0] for v in tp.profile_stop().values()))
    return best


@pytest.mark.parametrize("n3,prime,most", [(39, 41, 1.2), (63, 67, 1.2), (19, 29, 1.1)])
def test_time_of_a_neighbour(n3, prime, most):
    assert inverse_ms(220000, n3) < most * inverse_ms(220000, prime)
