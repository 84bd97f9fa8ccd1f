"""Final sampling of complex64 states searches in float64: states made so that
the exact running sum at the end of the first 256 amplitudes lies 2^-50 above
or below the draw.  At most 16 float64 roundings of values below 1 (2^-54
each, so less than 2^-50 together) stand between that sum and the computed
one, and the key is known exactly."""
import ctypes as C
from fractions import Fraction

import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv

pytestmark = pytest.mark.gpu


def _floor_sqrt32(r):
    """the largest float32 whose square is at most the Fraction r"""
    x = np.float32(float(r) ** 0.5)
    while Fraction(float(x)) ** 2 > r:
        x = np.nextafter(x, np.float32(0))
    return x


def _state(n, u, above, rng):
    x = rng.standard_normal((1 << n, 2)).astype(np.float32)
    x[:256] *= np.float32(np.sqrt(u * (1 - 2.0 ** -18) / (x[:256].astype(np.float64) ** 2).sum()))
    x[256:] *= np.float32(np.sqrt((1 - u) / (x[256:].astype(np.float64) ** 2).sum()))
    x[255] = 0
    x[100, 1] = 0
    rest = Fraction(u) + Fraction(1 if above else -1, 1 << 50)
    rest -= sum(Fraction(float(v)) ** 2 for v in x[:256].reshape(-1))
    for at in ((255, 0), (100, 1), (255, 1)):  # each leaves 2^-23 of what was left
        x[at] = _floor_sqrt32(rest)
        rest -= Fraction(float(x[at])) ** 2
    assert 0 <= rest < Fraction(1, 1 << 60) and float(x[255, 0]) ** 2 > 2.0 ** -30
    return x


@pytest.mark.parametrize("n", [10, 11])
def test_block_totals_keep_float64_precision(n):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(800 + n)
    seed, op, k = 62, 4, 96
    us = [O.uniform(seed, s, op) for s in range(400)]
    shots = [s for s in range(400) if 0.2 < us[s] < 0.9][:k]
    assert len(shots) == k
    above = rng.integers(0, 2, k)
    states = np.stack([_state(n, us[s], a, rng) for s, a in zip(shots, above)])
    dev = torch.from_numpy(states.reshape(-1)).cuda()
    ids = torch.tensor(shots, dtype=torch.int64).cuda()
    keys = torch.full((k,), -1, dtype=torch.int64).cuda()
    rc = sv.lib().sv_final_sample_noalloc(C.c_void_p(dev.data_ptr()), sv.SV_C64, n, k, C.c_void_p(ids.data_ptr()), seed,
                                          op, C.c_void_p(keys.data_ptr()),
                                          C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == sv.SV_OK
    torch.cuda.synchronize()
    assert np.array_equal(keys.cpu().numpy(), np.where(above, 255, 256))
