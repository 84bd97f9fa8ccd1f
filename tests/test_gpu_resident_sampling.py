"""A resident run samples its states as sv_final_sample_noalloc does: every
shot's state has a running sum within a few roundings of the shot's draw, so
that chunks of another size or sums in another order would give other keys."""
import ctypes as C
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 11, 12])
def test_resident_keys_are_those_of_the_final_sampling_call(n):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(900 + n)
    seed, shots, final_op = 63, 300, 2 * n
    c = W.Circuit(n)
    for q in range(n - 1):
        c.gate([q], W.u3(*rng.uniform(0, 6.28, 3)))
    # the top qubit is 0, and the sample in the lower half, with probability u
    us = [O.uniform(seed, s, final_op) for s in range(shots)]
    c.param_gate([n - 1], [W.u3(2 * math.acos(math.sqrt(u)), 0.0, 0.0) for u in us])
    for q in range(n):
        c.gate([q], np.diag([1.0, 1j]))
    c.final()
    assert c.n_ops == final_op + 1
    with sv.Batch(n, shots, 1, sv.SV_C128, sv.SV_BATCH, seed) as b:
        b.set_param_sets(np.arange(shots, dtype=np.uint32), shots)
        b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
        keys, launches = b.get_keys().astype(np.int64), b.stats()["launches"]
        states = np.stack([b.get_amplitudes(s) for s in range(shots)])
    assert launches == 1, "the run was not resident"
    dev = torch.from_numpy(np.stack([states.real, states.imag], -1).reshape(-1)).cuda()
    ids = torch.arange(shots, dtype=torch.int64).cuda()
    got = torch.full((shots,), -1, dtype=torch.int64).cuda()
    rc = sv.lib().sv_final_sample_noalloc(C.c_void_p(dev.data_ptr()), sv.SV_C128, n, shots, C.c_void_p(ids.data_ptr()),
                                          seed, final_op, C.c_void_p(got.data_ptr()),
                                          C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == sv.SV_OK
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), keys)
