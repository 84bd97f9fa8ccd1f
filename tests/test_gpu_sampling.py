"""Final sampling of caller-held states at the edges of its chunking: one
chunk, chunks of a warp and of a CTA, and complex64 states that start on an
8-byte boundary only (no 128-bit loads)."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n,k,shift", [(1, 5, 0), (4, 7, 1), (11, 33, 0), (12, 9, 1), (22, 2, 0), (23, 2, 1)])
def test_keys_follow_the_running_sums(n, k, shift, prec):
    torch = pytest.importorskip("torch")
    real = np.float32 if prec == sv.SV_C64 else np.float64
    rng = np.random.default_rng(600 + n)
    x = rng.standard_normal((k, 2 << n)).astype(real)
    x /= np.linalg.norm(x.astype(np.float64), axis=1, keepdims=True).astype(real)
    buf = torch.zeros(2 * shift + x.size, dtype=torch.float32 if real is np.float32 else torch.float64).cuda()
    buf[2 * shift:] = torch.from_numpy(x.reshape(-1))
    ids = torch.arange(k, dtype=torch.int64).cuda() + 3
    keys = torch.full((k,), -1, dtype=torch.int64).cuda()
    seed, op = 61, 5
    rc = sv.lib().sv_final_sample_noalloc(C.c_void_p(buf[2 * shift:].data_ptr()), prec, n, k,
                                          C.c_void_p(ids.data_ptr()), seed, op, C.c_void_p(keys.data_ptr()),
                                          C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == sv.SV_OK
    torch.cuda.synchronize()
    got = keys.cpu().numpy()
    v = x.astype(np.float64).reshape(k, -1, 2)
    cum = np.cumsum((v ** 2).sum(-1), axis=1)
    for s in range(k):
        u = O.uniform(seed, 3 + s, op)
        # the first index whose running sum exceeds u; sums of 2^n terms are
        # good to 2^n roundings of float64 (and float-float's 2^-45)
        lo, hi = (int(np.searchsorted(cum[s], u + d, side="right")) for d in (-4e-13, 4e-13))
        assert min(lo, (1 << n) - 1) <= got[s] <= min(hi, (1 << n) - 1)
