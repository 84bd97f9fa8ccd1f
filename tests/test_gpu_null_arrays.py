"""Arrays and counts of measurements on the way to the recorder: a circuit
without measurements may leave the arrays that only they have at NULL, and a
count out of range is refused."""
import ctypes as C

import numpy as np
import pytest

from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("n", [6, 15])
def test_no_measurement_arrays(n, use_graph):
    c = W.brickwork(n, 2, 0.05, 0.05, seed=551)
    full, bare = sv.circuit_struct(c.to_arrays()), sv.circuit_struct(c.to_arrays())
    for f in ("reset", "cl_off", "clbits"):
        setattr(bare, f, C.cast(None, C.POINTER(C.c_int32)))
    keys = []
    for cs in (full, bare):
        with sv.Batch(n, 20, 1, sv.SV_C64, sv.SV_BATCH, 85) as b:
            b.run_circuit(cs, use_graph=use_graph)
            keys.append(b.get_keys())
    assert np.array_equal(*keys)


@pytest.mark.parametrize("nq", [-1, 0, 5, 7])
def test_measured_qubit_count_out_of_range(nq):
    c = W.Circuit(6)
    c.gate([0], W.H)
    c.measure([0, 1, 2, 3], [0, 1, 2, 3])
    c.final()
    a = c.to_arrays()
    a["nq"][1] = nq
    a["qubits"] = np.concatenate([a["qubits"], np.zeros(8, np.int32)])
    a["clbits"] = np.concatenate([a["clbits"], np.zeros(8, np.int32)])
    with sv.Batch(6, 4, 4, sv.SV_C64, sv.SV_BATCH, 86) as b:
        with pytest.raises(sv.SvError):
            b.run_circuit(sv.circuit_struct(a))


def test_measurement_without_classical_bits_is_refused():
    c = W.Circuit(6)
    c.measure([0, 1, 2, 3], [0, 1, 2, 3])
    cs = sv.circuit_struct(c.to_arrays())
    cs.clbits = C.cast(None, C.POINTER(C.c_int32))
    with sv.Batch(6, 4, 4, sv.SV_C64, sv.SV_BATCH, 87) as b:
        with pytest.raises(sv.SvError, match="clbits"):
            b.run_circuit(cs)
