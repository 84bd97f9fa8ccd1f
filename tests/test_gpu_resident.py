"""Resident runs (one launch per circuit, the state in shared memory): a
batch without logs or tuning options takes them; an explicit fusion width
keeps the same circuit on the pass kernels.  Both have to give the oracle's
keys, and the same states within the complex64 / complex128 bars."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu
AMP = {sv.SV_C64: 1e-5, sv.SV_C128: 1e-12}

CIRCUITS = {
    "n1": lambda: _tiny(),
    "n3_mid": lambda: W.midcircuit_measure(3, 3, 0.05, [0, 2], seed=501),
    "n4": lambda: W.brickwork(4, 5, 0.05, 0.1, seed=502),
    "n5_kraus": lambda: W.qft(5, 0.05, seed=503, kraus=True),
    "n7_su4": lambda: W.random_su4(7, 4, 0.05, 0.1, seed=504),
    "n8_mid4": lambda: W.midcircuit_measure(8, 3, 0.02, [1, 3, 4, 7], seed=505),
    "n9_qft": lambda: W.qft(9, 0.02, seed=506),
    "n11_su4": lambda: W.random_su4(11, 3, 0.05, 0.05, seed=507),
    "n13_brick": lambda: W.brickwork(13, 3, 0.02, 0.05, seed=508),
    "n13_mid": lambda: W.midcircuit_measure(13, 2, 0.02, [0, 6, 12], seed=509),
    "n14_su4": lambda: W.random_su4(14, 2, 0.05, 0.05, seed=510),
    "forms": lambda: _forms(),
    "forms_mid": lambda: _forms(True),
    "mix": lambda: _two_qubit_mix(),
    "mono": lambda: _monomial(),
}
# complex64 measurements that the pass kernels take on shared-memory tiles
# (other than four qubits) round differently there and stay there
PASSES_C64 = {"n1", "n3_mid", "n13_mid", "forms_mid"}


def _tiny():
    c = W.Circuit(1)
    c.gate([0], W.H)
    c.depolarizing([0], 0.3)
    c.kraus([0], W.amplitude_damping(0.4))
    c.measure([0], [0], reset=1)
    c.gate([0], W.H, cond_clbit=0, cond_val=1)
    c.final()
    return c


def _forms(measure=False):
    # Kraus forms that are not diagonal, and a lone Kraus op between gates
    rng = np.random.default_rng(511)
    c = W.Circuit(6)
    for r in range(4):
        for q in range(6):
            c.gate([q], W.u3(*rng.uniform(0, 6.28, 3)))
        u = W.haar_unitary(2, rng)
        c.kraus([r], [k @ u for k in W.amplitude_damping(0.3)])
        c.gate([r, 5], W.haar_su4(rng))
        if measure:
            c.measure([r], [0], reset=r & 1)
    c.final()
    return c


def _two_qubit_mix():
    # dense and monomial pairs in both orders, two-qubit Kraus terms, strings
    # of four, diagonal and anti-diagonal phases, in passes too short to fold
    rng = np.random.default_rng(513)
    c = W.Circuit(8)
    cum, strings = W.depolarizing_table(0.2, 2)
    ph = np.exp(1j * rng.uniform(0, 6.28, 6))
    for r in range(6):
        a, b = (int(x) for x in rng.permutation(8)[:2])
        c.gate([a, b], W.haar_su4(rng))
        c.gate([b, a], W.cx())
        c.gate([b, a], W.haar_su4(rng))
        c.kraus([b, a], W.pauli_as_kraus(cum, strings))
        c.gate([b], np.diag(ph[:2]) if r % 2 else np.array([[0, ph[2]], [ph[3], 0]]))
        c.gate([b, a], W.cx() @ np.diag(ph[[0, 2, 4, 5]]))
        c.gate([a], W.u3(*rng.uniform(0, 6.28, 3)))
        c.pauli([0, 2, 5, 7], [0.5, 1.0], ["XIYZ", "ZZXI"])
        c.measure([1, 3, 4, 6], [0, 1, 2, 3], reset=r & 1)
    c.final()
    return c


def _monomial():
    # folded passes of complex phases: diagonal, anti-diagonal, permutations
    rng = np.random.default_rng(514)
    c = W.Circuit(7)
    for r in range(8):
        ph = np.exp(1j * rng.uniform(0, 6.28, 4))
        for q in range(7):
            c.gate([q], W.u3(*rng.uniform(0, 6.28, 3)) if r == 0 else
                   (np.diag(ph[:2]) if (q + r) % 2 else np.array([[0, ph[2]], [ph[3], 0]])))
            c.depolarizing([q], 0.1)
        for q in range(6):
            c.gate([q, q + 1], W.cx() @ np.diag(ph))
    c.final()
    return c


def _run(c, prec, mode, n_shots, seed, opts=(), psets=None):
    with sv.Batch(c.n_qubits, n_shots, max(1, c.n_clbits), prec, mode, seed) as b:
        if psets is not None:
            b.set_param_sets(psets, int(psets.max()) + 1)
        for k, v in opts:
            b.set_option(k, v)
        cs = sv.circuit_struct(c.to_arrays())
        b.run_circuit(cs, use_graph=True)
        first = b.get_keys()
        b.run_circuit(cs, use_graph=True)  # the kept launch
        st = b.stats()
        amps = [b.get_amplitudes(s) for s in (0, n_shots - 1)]
        return first, b.get_keys(), amps, st


@pytest.mark.parametrize("prec", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("name", sorted(CIRCUITS))
def test_resident_runs_match_passes_and_oracle(name, prec):
    c = CIRCUITS[name]()
    n = 200
    k1, k2, a, st = _run(c, prec, sv.SV_BATCH, n, 77)
    p1, _, pa, pst = _run(c, prec, sv.SV_BATCH, n, 77, [(sv.SV_OPT_MAX_ACTIVE, 4)])
    if not (prec == sv.SV_C128 and c.n_qubits > 13) and not (prec == sv.SV_C64 and name in PASSES_C64):
        assert st["launches"] < pst["launches"], "the run was not resident"
    assert np.array_equal(k1, k2) and np.array_equal(k1, p1)
    oc = O.OracleCircuit(c)
    assert np.array_equal(k1[:40], [O.run_shot(oc, 77, s)["key"] for s in range(40)])
    if prec == sv.SV_C64:  # the same arithmetic in the same order
        assert all(np.array_equal(x, y) for x, y in zip(a, pa))
    for s, x, y in zip((0, n - 1), a, pa):
        ref = O.run_shot(oc, 77, s, want_state=True)["state"]
        assert np.abs(x - ref).max() <= AMP[prec] and np.abs(y - ref).max() <= AMP[prec]


@pytest.mark.parametrize("prec", [sv.SV_C64, sv.SV_C128])
def test_resident_parameter_sweep(prec):
    c = W.param_sweep(7, 3, 5, 0.05, seed=512)
    ps = np.random.default_rng(1).integers(0, 5, 150).astype(np.uint32)
    k1, _, a, st = _run(c, prec, sv.SV_BATCH, 150, 9, psets=ps)
    oc = O.OracleCircuit(c)
    assert np.array_equal(k1[:40], [O.run_shot(oc, 9, s, pset=int(ps[s]))["key"] for s in range(40)])
    ref = O.run_shot(oc, 9, 0, want_state=True, pset=int(ps[0]))["state"]
    assert np.abs(a[0] - ref).max() <= AMP[prec]


@pytest.mark.parametrize("name,prec", [("n5_kraus", sv.SV_C64), ("n5_kraus", sv.SV_C128), ("n8_mid4", sv.SV_C64),
                                       ("n9_qft", sv.SV_C64), ("n9_qft", sv.SV_C128), ("n13_brick", sv.SV_C64)])
def test_resident_branching_runs_match_passes(name, prec):
    # a shot-branching batch with a slot per shot: the same keys and states,
    # and sv_stats reports the branches and fork copies the run stands for
    c = CIRCUITS[name]()
    n = 300
    k1, k2, a, st = _run(c, prec, sv.SV_BRANCH, n, 78)
    p1, _, pa, pst = _run(c, prec, sv.SV_BRANCH, n, 78, [(sv.SV_OPT_MAX_ACTIVE, 4)])
    assert st["launches"] < 5 < pst["launches"], "the run was not resident"
    assert np.array_equal(k1, k2) and np.array_equal(k1, p1)
    assert st["live_branches"] == pst["live_branches"] and st["copy_bytes"] == pst["copy_bytes"]
    if prec == sv.SV_C64:
        assert all(np.array_equal(x, y) for x, y in zip(a, pa))
    else:
        assert all(np.abs(x - y).max() <= AMP[prec] for x, y in zip(a, pa))


def test_short_of_slots_stays_on_passes():
    # fewer slots than shots: the waiting list, as without resident runs
    c = CIRCUITS["n7_su4"]()
    with sv.Batch(c.n_qubits, 200, 1, sv.SV_C64, sv.SV_BRANCH, 79) as b:
        b.set_option(sv.SV_OPT_SLOT_LIMIT, 20)
        b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
        st, keys = b.stats(), b.get_keys()
    assert st["restarts"] > 0
    oc = O.OracleCircuit(c)
    assert np.array_equal(keys[:20], [O.run_shot(oc, 79, s)["key"] for s in range(20)])
