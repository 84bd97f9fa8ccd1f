"""sv_stats of a shot-branching batch whose runs are resident: the branches of
the last run and the fork copies of every run since the last call, as a batch
on the pass kernels reports them for the same calls."""
import numpy as np
import pytest

from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N = 250
A = W.qft(8, 0.03, seed=541, kraus=True)
B = W.brickwork(8, 6, 0.01, 0.02, seed=542)


def _batch(passes, c=A):
    b = sv.Batch(8, N, max(1, c.n_clbits), sv.SV_C64, sv.SV_BRANCH, 84)
    if passes:
        b.set_option(sv.SV_OPT_MAX_ACTIVE, 4)
    return b


def _run(b, c):
    b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)


def _counts(b):
    st = b.stats()
    return st["live_branches"], st["copy_bytes"]


@pytest.mark.parametrize("seq", [(A, B), (A, A, B), (B, A, A, B, A)], ids=["ab", "aab", "baaba"])
def test_several_circuits_between_two_calls(seq):
    with _batch(False) as r, _batch(True) as p:
        for _ in range(2):
            for c in seq:
                _run(r, c)
                _run(p, c)
            assert _counts(r) == _counts(p)
        assert _counts(r) == (_counts(p)[0], 0)  # no run since
        assert np.array_equal(r.get_keys(), p.get_keys())


def test_resident_runs_and_then_the_pass_kernels():
    with _batch(False) as r, _batch(True) as p:
        for b in (r, p):
            _run(b, A)
            _run(b, A)
        r.set_option(sv.SV_OPT_MAX_ACTIVE, 4)
        for b in (r, p):
            _run(b, B)
        assert _counts(r) == _counts(p)


def test_calls_per_op_after_a_resident_run():
    with _batch(False) as r, _batch(True) as p:
        for b in (r, p):
            _run(b, A)
            b.stats()
            b.apply_gate_batch([0], W.H)
            b.sample_noise_pauli(1, [0], [0.5, 1.0], ["I", "X"])
            b.branch(1)
        assert _counts(r) == _counts(p)
        assert r.stats()["live_branches"] == 2


def test_parameter_sets():
    c = W.param_sweep(8, 3, 5, 0.05, seed=543)
    with _batch(False) as r, _batch(True) as p:
        for sets in (5, 5, 3):  # shots of 5 and of 3 sets
            ps = (np.random.default_rng(sets).integers(0, sets, N)).astype(np.uint32)
            for b in (r, p):
                b.set_param_sets(ps, 5)
                _run(b, c)
        lr, lp = r.stats(), p.stats()
        assert lr["launches"] < 20 < lp["launches"]
        assert (lr["live_branches"], lr["copy_bytes"]) == (lp["live_branches"], lp["copy_bytes"])
        assert np.array_equal(r.get_keys(), p.get_keys())
