"""Three- and four-qubit gates with few nonzero entries (the tile kernel leaves
the products with zeros out up to a quarter of the entries): controlled gates,
matrices at that quarter and just past it, on any qubits and tile sizes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu
AMP = {sv.SV_C64: 1e-5, sv.SV_C128: 1e-12}


def _gates(rng):
    swap = np.eye(4)[[0, 2, 1, 3]]
    toffoli, fredkin = np.eye(8)[[0, 1, 2, 7, 4, 5, 6, 3]], np.kron(np.eye(2), np.eye(4))
    fredkin[4:, 4:] = swap
    ph = np.exp(1j * rng.uniform(0, 6.28, 16))
    return [toffoli, fredkin, np.diag(ph[:8]), np.kron(np.eye(4), W.haar_unitary(2, rng)),  # 16 of 64: a quarter
            np.kron(W.haar_su4(rng), np.eye(2)),  # 32 of 64: dense
            np.kron(np.eye(2), toffoli), np.diag(ph), np.eye(16)[rng.permutation(16)] * ph,
            np.kron(np.eye(4), W.haar_su4(rng)),  # 64 of 256: a quarter
            np.kron(W.haar_unitary(8, rng), np.eye(2))]  # 128 of 256


def _circuit(n, seed):
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for q in range(n):
        c.gate([q], W.u3(*rng.uniform(0, 6.28, 3)))
    gates = _gates(rng)
    for i in rng.permutation(len(gates)):
        k = int(np.log2(len(gates[i])))
        c.gate([int(q) for q in rng.permutation(n)[:k]], gates[i])
        c.depolarizing([int(rng.integers(n))], 0.2)
    c.final()
    return c


@pytest.mark.parametrize("prec", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("n,tile", [(4, 0), (5, 5), (7, 0), (9, 5), (12, 0), (13, 6)])
def test_sparse_gates_match_the_oracle(n, tile, prec):
    c, shots, seed = _circuit(n, 570 + n), 30, 88
    oc = O.OracleCircuit(c)
    ref = [O.run_shot(oc, seed, s, want_state=True) for s in range(shots)]
    for mode in (sv.SV_BATCH, sv.SV_BRANCH):
        with sv.Batch(n, shots, 1, prec, mode, seed) as b:
            if tile:
                b.set_option(sv.SV_OPT_TILE_BITS, tile)
            b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
            assert np.array_equal(b.get_keys(), [r["key"] for r in ref])
            for s in (0, 11, shots - 1):
                assert np.abs(b.get_amplitudes(s) - ref[s]["state"]).max() <= AMP[prec]
