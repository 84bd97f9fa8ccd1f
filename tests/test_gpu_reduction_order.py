"""The sums of a large state do not depend on the memory a batch has: with a
budget that leaves no room for a record per reduction unit, a batch logs the
same running sums, bit for bit, as one with all of the device's memory."""
import numpy as np
import pytest

from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _circuit(n):
    rng = np.random.default_rng(560 + n)
    c = W.Circuit(n)
    for q in range(n):
        c.gate([q], W.u3(*rng.uniform(0.5, 2.5, 3)))
    c.kraus([n - 1], W.amplitude_damping(0.3))
    u = W.haar_unitary(2, rng)
    c.kraus([3], [k @ u for k in W.amplitude_damping(0.3)])  # forms that are not diagonal
    c.measure([0, 5, n - 3, n - 1], [0, 1, 2, 3])
    c.kraus([1], W.amplitude_damping(0.2))
    c.kraus([n - 2], W.amplitude_damping(0.4))
    c.final()
    return c


@pytest.mark.parametrize("mode", [sv.SV_BATCH, sv.SV_BRANCH])
@pytest.mark.parametrize("n", [23, 24, 26])
def test_running_sums_do_not_depend_on_the_budget(n, mode):
    c, shots = _circuit(n), 2
    cs = sv.circuit_struct(c.to_arrays())
    out = []
    # no limit; room for the states and 1024 records of 16 float64 each
    for budget in (0, shots * ((8 << n) + 1024 * 16 * 8)):
        with sv.Batch(n, shots, 4, sv.SV_C64, mode, 87, mem_budget=budget) as b:
            b.set_option(sv.SV_OPT_LOG, 1)
            b.run_circuit(cs, use_graph=True)
            ops = [i for i, o in enumerate(c.ops) if o.kind in (W.KRAUS, W.MEASURE, W.FINAL)]
            out.append([b.get_outcomes(i, thresholds=True) for i in ops] + [b.get_keys()])
            assert b.stats()["restarts"] == 0
    for x, y in zip(*out):
        assert all(np.array_equal(p, q) for p, q in zip(x, y)) if isinstance(x, tuple) else np.array_equal(x, y)
