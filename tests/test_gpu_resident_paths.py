"""Which launches a circuit takes at the edges of the resident runs' rules, and
that both sides of each edge give the keys of the pass kernels: parameter
sweeps in both modes, more states than CTAs (a CTA's second state) with folded
passes, and the shots beyond which one CTA per SM is too slow."""
import numpy as np
import pytest

from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

pytestmark = pytest.mark.gpu
AMP = {sv.SV_C64: 1e-5, sv.SV_C128: 1e-12}


def _run(c, prec, mode, shots, psets=None, passes=False):
    with sv.Batch(c.n_qubits, shots, max(1, c.n_clbits), prec, mode, 89) as b:
        if psets is not None:
            b.set_param_sets(psets, int(psets.max()) + 1)
        if passes:
            b.set_option(sv.SV_OPT_MAX_ACTIVE, 4)
        b.run_circuit(sv.circuit_struct(c.to_arrays()), use_graph=True)
        amps = np.stack([b.get_amplitudes(s) for s in (0, shots // 2, shots - 1)])
        return b.get_keys(), amps, b.stats()


def _same(c, prec, mode, shots, psets=None):
    k, a, st = _run(c, prec, mode, shots, psets)
    pk, pa, pst = _run(c, prec, mode, shots, psets, passes=True)
    assert pst["launches"] > 1 and np.array_equal(k, pk)
    assert np.abs(a - pa).max() <= AMP[prec]
    return st, pst


@pytest.mark.parametrize("mode", [sv.SV_BATCH, sv.SV_BRANCH])
@pytest.mark.parametrize("prec", [sv.SV_C64, sv.SV_C128])
def test_parameter_sweeps_run_resident(prec, mode):
    c = W.param_sweep(7, 3, 5, 0.05, seed=581)
    st, pst = _same(c, prec, mode, 150, np.random.default_rng(2).integers(0, 5, 150).astype(np.uint32))
    assert st["launches"] == 1
    if mode == sv.SV_BRANCH:
        assert st["live_branches"] == pst["live_branches"] and st["copy_bytes"] == pst["copy_bytes"]


@pytest.mark.parametrize("n,shots", [(6, 9000), (10, 2500), (13, 700)])
def test_folded_passes_of_more_states_than_ctas(n, shots):
    st, _ = _same(W.qft(n, 0.02, seed=582), sv.SV_C64, sv.SV_BATCH, shots)
    assert st["launches"] == 1


@pytest.mark.parametrize("prec,make,over", [(sv.SV_C64, lambda: W.brickwork(14, 3, 0.02, 0.05, seed=583), True),
                                            (sv.SV_C64, lambda: W.random_su4(14, 2, 0.05, 0.05, seed=584), False),
                                            (sv.SV_C128, lambda: W.brickwork(13, 2, 0.02, 0.05, seed=585), False),
                                            (sv.SV_C128, lambda: W.random_su4(13, 2, 0.05, 0.05, seed=586), False)],
                         ids=["c64", "c64_reductions", "c128", "c128_reductions"])
def test_one_cta_per_sm(prec, make, over):
    torch = pytest.importorskip("torch")
    edge = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    c = make()
    assert _same(c, prec, sv.SV_BATCH, edge)[0]["launches"] == 1
    assert (_same(c, prec, sv.SV_BATCH, edge + 1)[0]["launches"] == 1) == over
