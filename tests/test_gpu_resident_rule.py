"""Which shot-branching circuits run resident.  The estimate has to see that
few shots branch: whatever the place of the identity in a Pauli table, when
measured outcomes are certain, and when two Kraus ops share a decide.  Each of
these runs 1.05 to 2.6 times as fast on the pass kernels."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _noisy(n, depth, p, last):
    rng = np.random.default_rng(531)
    cum, strings = W.depolarizing_table(p, 1)
    if last:
        cum, strings = list(np.cumsum(np.diff([0.0] + list(cum))[::-1])), list(strings)[::-1]
        cum[-1] = 1.0
    c = W.Circuit(n)
    for layer in range(depth):
        for q in range(n):
            c.gate([q], W.u3(*rng.uniform(0, 6.28, 3)))
            c.pauli([q], cum, strings)
        for a in range(layer % 2, n - 1, 2):
            c.gate([a, a + 1], W.cx())
    c.final()
    return c


def _parity(n, rounds, p):
    # pair parities of a computational state, four at a time
    c, d = W.Circuit(n), n - 4
    c.gate([1], W.X)
    for r in range(rounds):
        for a in range(4):
            for j in (0, 1):
                c.gate([(2 * a + j + r) % d, d + a], W.cx())
                c.depolarizing([(2 * a + j + r) % d, d + a], p)
        c.measure([d, d + 1, d + 2, d + 3], [0, 1, 2, 3], reset=1)
    c.final()
    return c


def _run(c, shots, seed=83):
    with sv.Batch(c.n_qubits, shots, max(1, c.n_clbits), sv.SV_C64, sv.SV_BRANCH, seed) as b:
        b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
        return b.get_keys(), b.stats()["launches"]


@pytest.mark.parametrize("name,make", [("identity_first", lambda: _noisy(14, 6, 1e-4, False)),
                                       ("identity_last", lambda: _noisy(14, 6, 1e-4, True)),
                                       ("certain_outcomes", lambda: _parity(13, 12, 1e-4)),
                                       ("kraus_pairs", lambda: W.random_su4(11, 4, 1e-4, 1e-4, 1))])
def test_few_branches_stay_on_the_passes(name, make):
    c = make()
    keys, launches = _run(c, 4000)
    assert launches > 5
    oc = O.OracleCircuit(c)
    assert np.array_equal(keys[:8], [O.run_shot(oc, 83, s)["key"] for s in range(8)])


@pytest.mark.parametrize("make", [lambda: W.brickwork(12, 8, 1e-3, 1e-2, 1), lambda: W.qft(11, 1e-2, 1, kraus=True),
                                  lambda: _parity(9, 12, 1e-4)])
def test_many_decides_run_resident(make):
    assert _run(make(), 4000)[1] == 1
