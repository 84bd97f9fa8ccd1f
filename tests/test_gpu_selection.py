"""Selection at the end of the cumulative table: a complex64 state that has
lost a little norm, a draw past the rounded total, and trailing Kraus terms of
probability zero.  The choice is the last term of nonzero probability, on the
pass kernels and in a resident run (a term of probability zero would leave a
state that is not a number)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu
# cos 1 and sin 1 in float32 have squares that sum to 1 - 7.9e-8: 40 rotations
# by them keep about 1 - 3e-6 of a state's norm
TURNS = 40
SEED, OP = 91, 3 + TURNS
# shots whose draw for OP lies within 1.2e-6 of 1
SHOTS = [589042, 862907, 2895701, 3836964, 4334687, 4578881, 4815992, 6182850]


def _weights(i):
    return np.random.default_rng(700 + i).dirichlet(np.full(8, 3.0))


def _circuit(i):
    rng = np.random.default_rng(720 + i)
    c = W.Circuit(5)
    for q in (0, 1, 4):
        c.gate([q], W.u3(*rng.uniform(0.5, 2.5, 3)))
    for _ in range(TURNS):  # on a qubit of the channel, which waits for them
        c.gate([3], W.u3(2.0, 0.0, 0.0))
    # qubit 2 is |0>: damping it changes nothing, and the eight terms of its
    # decay have probability 0
    keep, decay = (np.kron(np.eye(2), k) for k in W.amplitude_damping(0.3))
    c.kraus([2, 3], [np.sqrt(w) * m for m in (keep, decay) for w in _weights(i)])
    c.final()
    assert c.n_ops == OP + 2
    return c


@pytest.mark.parametrize("opts", [(), ((sv.SV_OPT_MAX_ACTIVE, 4),)], ids=["resident", "passes"])
@pytest.mark.parametrize("i", range(len(SHOTS)))
def test_draw_past_the_total_takes_the_last_possible_term(i, opts):
    assert 0 < 1 - O.uniform(SEED, SHOTS[i], OP) < 1.2e-6
    c = _circuit(i)
    with sv.Batch(5, 1, 1, sv.SV_C64, sv.SV_BATCH, SEED) as b:
        b.set_option(sv.SV_OPT_SHOT_BASE, SHOTS[i])
        for k, v in opts:
            b.set_option(k, v)
        b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
        a, launches = b.get_amplitudes(0), b.stats()["launches"]
    assert (launches == 1) == (not opts)
    p = np.abs(a) ** 2
    assert np.all(np.isfinite(p)) and abs(p.sum() - 1) < 1e-5
    assert p.reshape(2, 2, 2, 4)[:, :, 1].sum() == 0
