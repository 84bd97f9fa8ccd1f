"""Resident runs against the pass kernels where probabilities enter the state:
the sums of a Kraus op or a measurement run over other lanes, so the float32
factor of a choice may differ by one rounding, in some 1e-7 of the choices.
Every shot's state is compared, and shards that run resident are compared with
a union of them that the number of shots keeps on the passes."""
import numpy as np
import pytest

from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(c, n_shots, seed, passes=False, base=0, amps=None):
    with sv.Batch(c.n_qubits, n_shots, max(1, c.n_clbits), sv.SV_C64, sv.SV_BATCH, seed) as b:
        b.set_option(sv.SV_OPT_SHOT_BASE, base)
        if passes:
            b.set_option(sv.SV_OPT_MAX_ACTIVE, 4)
        b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
        resident = b.stats()["launches"] == 1
        shots = range(n_shots) if amps is None else amps
        return b.get_keys(), np.stack([b.get_amplitudes(s) for s in shots]), resident


@pytest.mark.parametrize("make", [lambda: W.qft(9, 0.02, seed=521, kraus=True),
                                  lambda: W.midcircuit_measure(8, 12, 0.02, [1, 3, 4, 7], seed=522),
                                  lambda: W.random_su4(10, 8, 0.05, 0.1, seed=523)], ids=["qft", "mid", "su4"])
def test_states_of_all_shots(make):
    c = make()
    k, a, resident = _run(c, 2000, 81)
    pk, pa, pres = _run(c, 2000, 81, passes=True)
    assert resident and not pres
    assert np.array_equal(k, pk)
    # a shot either took the same factors (the same bits) or is as far off as
    # complex64 states are from each other after a rounding
    differ = (a != pa).any(axis=1)
    assert differ.mean() <= 0.01
    assert np.abs(a - pa).max() <= 1e-5


def test_resident_shards_make_the_union():
    # 14 qubits, passes with reductions: resident up to four CTAs a SM's worth
    # of shots, passes beyond
    c = W.random_su4(14, 2, 0.05, 0.05, seed=524)
    n = 900
    k, a, resident = _run(c, n, 82, amps=range(0, n, 50))
    assert not resident
    parts = [_run(c, n // 3, 82, base=b, amps=range(0, n // 3, 50)) for b in range(0, n, n // 3)]
    assert all(p[2] for p in parts)
    assert np.array_equal(np.concatenate([p[0] for p in parts]), k)
    assert np.abs(np.concatenate([p[1] for p in parts]) - a).max() <= 1e-5
