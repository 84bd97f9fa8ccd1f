"""The work that is timed: noisy multi-shot runs through the public entry points.

A case names a circuit family of `workloads`, its size, a number of shots, a
precision and a mode.  `run` makes the calls that a user's program makes and
returns what it gets back: the final key of every shot, the distribution of
the density-matrix method and, for some cases, the state of one shot.

Families: brick (U3 / CX bricks with depolarizing noise), qft (Pauli or Kraus
noise), su4 (two-qubit unitaries, depolarizing and amplitude damping), mid
(mid-circuit measurements and conditional gates), sweep (parameter sets), dm
(density matrix), multi (many circuits in one graph), ops (a layer call by
call on a new batch) and sample (final sampling of states the caller holds).
"""
import ctypes
import math

import numpy as np
import torch

from paper_2308_03399_gb300 import sv
from paper_2308_03399_gb300 import workloads as W

MODES = {"batch": sv.SV_BATCH, "branch": sv.SV_BRANCH}
PRECS = {"c64": sv.SV_C64, "c128": sv.SV_C128}


def listed():
    return [
        # launch-bound: a small register and few shots
        {"name": "brick6", "family": "brick", "n": 6, "depth": 6, "shots": 100, "p": 1e-2, "prec": "c64",
         "mode": "batch", "amps": False},
        {"name": "brick10", "family": "brick", "n": 10, "depth": 20, "shots": 1000, "p": 1e-3, "prec": "c64",
         "mode": "batch", "amps": False},
        {"name": "qft13", "family": "qft", "n": 13, "kraus": False, "shots": 4000, "p": 1e-2, "prec": "c64",
         "mode": "batch", "amps": True},
        {"name": "qft12_kraus", "family": "qft", "n": 12, "kraus": True, "shots": 4000, "p": 1e-2, "prec": "c64",
         "mode": "branch", "amps": False},
        {"name": "su4_16", "family": "su4", "n": 16, "depth": 16, "shots": 10000, "p": 1e-2, "gamma": 5e-3,
         "prec": "c64", "mode": "branch", "amps": True},
        {"name": "mid20", "family": "mid", "n": 20, "rounds": 30, "shots": 300, "p": 5e-3, "prec": "c64",
         "mode": "branch", "amps": False},
        {"name": "su4_27", "family": "su4", "n": 27, "depth": 12, "shots": 7, "p": 1e-3, "gamma": 1e-3,
         "prec": "c64", "mode": "branch", "amps": False},
        {"name": "sweep11_c128", "family": "sweep", "n": 11, "layers": 6, "sets": 16, "shots": 1000, "p": 1e-2,
         "prec": "c128", "mode": "batch", "amps": True},
        {"name": "dm9_c128", "family": "dm", "n": 9, "depth": 6, "shots": 4000, "p": 1e-2, "prec": "c128"},
        {"name": "multi8", "family": "multi", "circuits": 8, "lo": 8, "hi": 17, "depth": 12, "shots": 2501,
         "p": 3e-3, "prec": "c64"},
        {"name": "ops12", "family": "ops", "n": 12, "shots": 250, "p": 2e-2, "prec": "c64", "mode": "branch"},
        {"name": "sample15", "family": "sample", "n": 15, "shots": 3001, "prec": "c64"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(["brick", "brick", "qft", "qft", "su4", "su4", "mid", "sweep", "dm", "multi", "ops", "sample"])
    prec = "c64" if rng.random() < 0.75 else "c128"
    mode = rng.choice(["batch", "branch"])
    # amplitude updates of the run, held below those of the largest listed case
    room = 3e11 if prec == "c64" else 1e11
    if f == "brick":
        n, depth = rng.randint(4, 17), rng.randint(4, 30)
        shots = min(_log(rng, 50, 10000), int(room / (2 ** n * n * depth * 3)))
        return {"family": f, "n": n, "depth": depth, "shots": max(3, shots), "p": _log(rng, 10, 1000) * 1e-5,
                "prec": prec, "mode": mode, "amps": n <= 14}
    if f == "qft":
        n, kraus = rng.randint(5, 16), rng.random() < 0.4
        shots = min(_log(rng, 100, 4000), int(room / (2 ** n * n * n * (40 if kraus else 3))))
        return {"family": f, "n": n, "kraus": kraus, "shots": max(3, shots), "p": _log(rng, 100, 3000) * 1e-5,
                "prec": prec, "mode": mode, "amps": n <= 14}
    if f == "su4":
        n, depth = rng.randint(5, 24), rng.randint(4, 16)
        shots = min(_log(rng, 20, 10000), int(room / (2 ** n * n * depth * 3)))
        return {"family": f, "n": n, "depth": depth, "shots": max(2, shots), "p": _log(rng, 100, 1000) * 1e-5,
                "gamma": _log(rng, 100, 1000) * 1e-5, "prec": prec, "mode": mode if n < 17 else "branch",
                "amps": n <= 14}
    if f == "mid":
        n, rounds = rng.randint(6, 20), rng.randint(3, 30)
        shots = min(_log(rng, 20, 5000), int(room / (2 ** n * n * rounds * 4)))
        return {"family": f, "n": n, "rounds": rounds, "shots": max(2, shots), "p": _log(rng, 100, 1000) * 1e-5,
                "prec": prec, "mode": mode if n < 17 else "branch", "amps": n <= 14}
    if f == "sweep":
        n, layers = rng.randint(5, 14), rng.randint(2, 8)
        return {"family": f, "n": n, "layers": layers, "sets": rng.randint(3, 32),
                "shots": min(_log(rng, 64, 2000), int(room / (2 ** n * n * layers * 3))),
                "p": _log(rng, 100, 3000) * 1e-5, "prec": prec, "mode": mode, "amps": True}
    if f == "dm":
        return {"family": f, "n": rng.randint(4, 10), "depth": rng.randint(2, 8), "shots": _log(rng, 100, 8000),
                "p": _log(rng, 100, 3000) * 1e-5, "prec": prec}
    if f == "multi":
        lo = rng.randint(6, 9)
        return {"family": f, "circuits": rng.randint(3, 10), "lo": lo, "hi": rng.randint(lo + 3, 16),
                "depth": rng.randint(6, 16), "shots": _log(rng, 300, 3000), "p": _log(rng, 30, 1000) * 1e-5,
                "prec": prec}
    if f == "ops":
        return {"family": f, "n": rng.randint(5, 15), "shots": _log(rng, 16, 1000), "p": _log(rng, 200, 5000) * 1e-5,
                "prec": prec, "mode": mode}
    n = rng.randint(6, 20)
    return {"family": f, "n": n, "shots": min(_log(rng, 10, 20000), 131072 // max(1, 2 ** n // 2048)), "prec": prec}


# ---- the circuits ------------------------------------------------------------
def _layer(n, p, seed):
    """One layer, each op called by itself: U3 with depolarizing noise on every
    qubit, CX bricks with noise, a fused three-qubit block, amplitude damping,
    a measurement and a conditional flip."""
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for q in range(n):
        c.gate([q], W.u3(*rng.uniform(0, 2 * math.pi, 3)))
        c.depolarizing([q], p)
    for a in range(0, n - 1, 2):
        c.gate([a, a + 1], W.cx())
        c.depolarizing([a, a + 1], p)
    c.gate([0, n // 2, n - 1], W.haar_unitary(8, rng))
    c.kraus([1], W.amplitude_damping(0.1))
    c.measure([0, n - 1], [0, 1])
    c.gate([0], W.X, cond_clbit=0, cond_val=1)
    c.final()
    return c


def _circuit(case, seed):
    f = case["family"]
    if f in ("brick", "dm"):
        return W.brickwork(case["n"], case["depth"], case["p"], min(10 * case["p"], 3e-2), seed)
    if f == "qft":
        return W.qft(case["n"], case["p"], seed, kraus=case["kraus"])
    if f == "su4":
        return W.random_su4(case["n"], case["depth"], case["p"], case["gamma"], seed)
    if f == "mid":
        n = case["n"]
        return W.midcircuit_measure(n, case["rounds"], case["p"], sorted({0, n // 4, n // 2, 3 * n // 4}), seed)
    if f == "sweep":
        return W.param_sweep(case["n"], case["layers"], case["sets"], case["p"], seed)
    return _layer(case["n"], case["p"], seed)


def _psets(case, seed):
    return np.random.default_rng(seed + 1).integers(0, case["sets"], case["shots"]).astype(np.uint32)


def _multi(case, seed):
    """Circuits of sizes spread over lo..hi and the shots of each."""
    rng = np.random.default_rng(case["shots"])
    k = case["circuits"]
    sizes = [case["lo"] + (case["hi"] - case["lo"]) * i // max(1, k - 1) for i in range(k)]
    shots = np.maximum(1, rng.dirichlet(np.full(k, 4.0)) * case["shots"]).astype(int)
    return [(W.brickwork(n, case["depth"] + i % 3, case["p"], min(10 * case["p"], 1e-2), seed + i), int(s))
            for i, (n, s) in enumerate(zip(sizes, shots))]


# ---- prepare and run ---------------------------------------------------------
def prepare(case, seed):
    f = case["family"]
    s = dict(case, seed=seed, prec=PRECS[case["prec"]], c64=case["prec"] == "c64")
    if f == "sample":
        n, k = case["n"], case["shots"]
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(k, 2 << n, generator=g, device="cuda", dtype=torch.float32 if s["c64"] else torch.float64)
        x /= x.norm(dim=1, keepdim=True)
        s["states"] = x
        s["ids"] = torch.arange(k, device="cuda", dtype=torch.int64) + 17
        s["keys"] = torch.zeros(k, device="cuda", dtype=torch.int64)
        return s
    if f == "multi":
        s["stream"] = torch.cuda.Stream()
        s["structs"], s["batches"] = [], []
        for c, k in _multi(case, seed):
            s["structs"].append(sv.circuit_struct(c.to_arrays()))
            s["batches"].append(sv.Batch(c.n_qubits, k, 1, s["prec"], sv.SV_BATCH if c.n_qubits <= 12 else sv.SV_BRANCH,
                                         seed, mem_budget=4 << 30, stream=s["stream"].cuda_stream))
        return s
    c = _circuit(case, seed)
    if f == "ops":
        s["circuit"] = c
        return s
    s["struct"] = sv.circuit_struct(c.to_arrays())
    if f != "dm":
        s["batch"] = sv.Batch(c.n_qubits, case["shots"], max(1, c.n_clbits), s["prec"], MODES[case["mode"]], seed)
        if f == "sweep":
            s["batch"].set_param_sets(_psets(case, seed), case["sets"])
    return s


def _amps(batch, c64):
    a = batch.get_amplitudes(0)
    return a.astype(np.complex64) if c64 else a


def run(s):
    f = s["family"]
    if f == "sample":
        st = sv.lib().sv_final_sample_noalloc(
            ctypes.c_void_p(s["states"].data_ptr()), s["prec"], s["n"], s["shots"],
            ctypes.c_void_p(s["ids"].data_ptr()), s["seed"], 7, ctypes.c_void_p(s["keys"].data_ptr()),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st != sv.SV_OK:
            raise sv.SvError(st, sv.lib().sv_last_error().decode())
        return {"keys": s["keys"]}
    if f == "multi":
        sv.run_circuits(s["batches"], s["structs"], use_graph=True)
        return {"keys": [b.get_keys().view(np.int64) for b in s["batches"]]}
    if f == "dm":
        keys, probs = sv.dm_run(s["struct"], s["shots"], s["prec"], s["seed"])
        return {"keys": keys.view(np.int64), "probs": probs.astype(np.float32) if s["c64"] else probs}
    if f == "ops":
        return _run_ops(s)
    b = s["batch"]
    b.run_circuit(s["struct"], use_graph=True)
    out = {"keys": b.get_keys().view(np.int64)}
    if s["amps"]:
        out["amps"] = _amps(b, s["c64"])
    return out


def _run_ops(s):
    c = s["circuit"]
    with sv.Batch(c.n_qubits, s["shots"], c.n_clbits, s["prec"], MODES[s["mode"]], s["seed"], mem_budget=4 << 30) as b:
        for i, o in enumerate(c.ops):
            if o.kind == W.GATE:
                b.apply_gate_batch(o.qubits, o.mat, o.cond_clbit, o.cond_val)
            elif o.kind == W.PAULI:
                b.sample_noise_pauli(i, o.qubits, o.cum, o.strings)
            elif o.kind == W.KRAUS:
                b.sample_noise_kraus(i, o.qubits, o.kraus)
            elif o.kind == W.MEASURE:
                b.measure_batch(i, o.qubits, o.clbits, o.reset)
        hist = b.counts(len(c.ops) - 1)
        dense = np.zeros(1 << c.n_qubits, np.int64)
        dense[list(hist)] = list(hist.values())
        return {"keys": b.get_keys().view(np.int64), "hist": dense, "amps": _amps(b, s["c64"])}


# ---- what a pass cannot do without -------------------------------------------
def _circuit_work(c, shots, prec, amps):
    """Bytes: the circuit's tables read, the keys (and a state) written.
    Operations: every gate and every Kraus or measurement reduction of every
    shot's state, by the matrix's own structure (dense 8 D - 2 per amplitude,
    diagonal 6, permutations none)."""
    dim, flops, data = float(1 << c.n_qubits), 0.0, 0
    for o in c.ops:
        mats = [o.mat] if o.kind == W.GATE else (o.kraus or [])
        data += sum(16 * m.size for m in mats) + 8 * len(o.cum or [])
        if o.kind in (W.GATE, W.PGATE):
            m = mats[0]
            D = m.shape[0]
            nz = m != 0
            if nz.sum() > D:
                flops += dim * (8 * D - 2)
            elif not np.all(m[nz] == 1):
                flops += dim * 6
        elif o.kind == W.KRAUS:
            flops += dim * (4 + 6)
        elif o.kind == W.MEASURE:
            flops += dim * (4 + 2)
        elif o.kind == W.FINAL:
            flops += dim * 4
    return data + 8.0 * shots + (dim * (8 if prec == "c64" else 16) if amps else 0), flops * shots


def work(case):
    f = case["family"]
    amp = 8 if case["prec"] == "c64" else 16
    if f == "sample":
        size = float(case["shots"]) * (1 << case["n"])
        return {"bytes": size * amp + 16.0 * case["shots"], "flops": 4 * size}
    if f == "multi":
        w = [_circuit_work(c, k, case["prec"], False) for c, k in _multi(case, 0)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    c = _circuit(case, 0)
    if f == "dm":
        # gates on both sides of rho, depolarizing channels as one pass each
        dim = 4.0 ** case["n"]
        flops = sum(dim * ((8 * 2 ** len(o.qubits) - 2) * 2 if o.kind == W.GATE else 8) for o in c.ops)
        data = sum(16 * o.mat.size for o in c.ops if o.kind == W.GATE)
        return {"bytes": data + 8.0 * case["shots"] + 8.0 * (1 << case["n"]), "flops": flops}
    bytes_, flops = _circuit_work(c, case["shots"], case["prec"], f == "ops" or case["amps"])
    return {"bytes": bytes_, "flops": flops}


# ---- the same in 64 bits, in plain torch -------------------------------------
def _uniform(seed, shot, op):
    """Philox4x32-10, key = seed, counter = (shot, op): the top 53 bits of the
    first two words times 2^-53."""
    k = [seed & 0xffffffff, (seed >> 32) & 0xffffffff]
    x = [shot & 0xffffffff, (shot >> 32) & 0xffffffff, op, 0]
    for _ in range(10):
        a, b = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
        x = [(b >> 32) ^ x[1] ^ k[0], b & 0xffffffff, (a >> 32) ^ x[3] ^ k[1], a & 0xffffffff]
        k = [(k[0] + 0x9E3779B9) & 0xffffffff, (k[1] + 0xBB67AE85) & 0xffffffff]
    return (((x[0] << 32) | x[1]) >> 11) * 2.0 ** -53


def _pick(u, probs):
    c, last = 0.0, 0
    for t, p in enumerate(probs):
        c += p
        if p > 0:
            last = t
        if u < c:
            return t
    return last


def _apply(psi, n, qubits, m):
    """m on the listed qubits of psi (an n-axis tensor, qubit q on axis n-1-q)."""
    k = len(qubits)
    axes = [n - 1 - q for q in reversed(qubits)]
    m = torch.as_tensor(np.ascontiguousarray(m), dtype=torch.complex128, device=psi.device).reshape([2] * (2 * k))
    out = torch.tensordot(m, psi, dims=(list(range(k, 2 * k)), axes))
    return torch.movedim(out, list(range(k)), axes)


ONE = {"I": np.eye(2), "X": W.X, "Y": np.array([[0, -1j], [1j, 0]]), "Z": np.diag([1.0, -1.0])}


def _norm2(x):
    return float((x.real.square() + x.imag.square()).sum())


def _state_of_shot(c, seed, shot, pset=0):
    n = c.n_qubits
    psi = torch.zeros([2] * n, dtype=torch.complex128, device="cuda")
    psi.view(-1)[0] = 1
    bits = {}
    for i, o in enumerate(c.ops):
        if o.kind == W.GATE:
            if o.cond_clbit < 0 or bits.get(o.cond_clbit, 0) == o.cond_val:
                psi = _apply(psi, n, o.qubits, o.mat)
        elif o.kind == W.PGATE:
            psi = _apply(psi, n, o.qubits, o.kraus[pset])
        elif o.kind == W.PAULI:
            u = _uniform(seed, shot, i)
            t = next((t for t, x in enumerate(o.cum) if u < x), len(o.cum) - 1)
            for q, ch in zip(o.qubits, o.strings[t]):
                if ch != "I":
                    psi = _apply(psi, n, [q], ONE[ch])
        elif o.kind == W.KRAUS:
            outs = [_apply(psi, n, o.qubits, m) for m in o.kraus]
            ps = [_norm2(x) for x in outs]
            t = _pick(_uniform(seed, shot, i), ps)
            psi = outs[t] / math.sqrt(ps[t])
        elif o.kind == W.MEASURE:
            k = len(o.qubits)
            pr = psi.real.square() + psi.imag.square()
            axes = [n - 1 - q for q in reversed(o.qubits)]
            ps = torch.movedim(pr, axes, list(range(k))).reshape(1 << k, -1).sum(1).tolist()
            t = _pick(_uniform(seed, shot, i), ps)
            m = np.zeros((1 << k, 1 << k))
            m[0 if o.reset else t, t] = 1.0 / math.sqrt(ps[t])
            psi = _apply(psi, n, o.qubits, m)
            for j, b in enumerate(o.clbits):
                bits[b] = (t >> j) & 1
    return psi.reshape(-1).cpu().numpy()


def _distribution(c):
    """The final distribution of a circuit of gates and Pauli noise, from its
    density matrix (row qubits 0..n-1, column qubits n..2n-1)."""
    n = c.n_qubits
    rho = torch.zeros([2] * (2 * n), dtype=torch.complex128, device="cuda")
    rho.view(-1)[0] = 1

    def both(r, qubits, m):
        return _apply(_apply(r, 2 * n, qubits, m), 2 * n, [q + n for q in qubits], np.conj(m))

    for o in c.ops:
        if o.kind == W.GATE:
            rho = both(rho, o.qubits, o.mat)
        elif o.kind == W.PAULI:
            new, prev = 0, 0.0
            for x, s in zip(o.cum, o.strings):
                r = rho
                for q, ch in zip(o.qubits, s):
                    if ch != "I":
                        r = both(r, [q], ONE[ch])
                new, prev = new + (x - prev) * r, x
            rho = new
    return torch.diagonal(rho.reshape(1 << n, 1 << n)).real.cpu().numpy().copy()


def exact(case, seed):
    f = case["family"]
    if f in ("sample", "multi"):
        return None
    if f == "dm":
        return {"keys": None, "probs": _distribution(_circuit(case, seed))}
    if f == "ops":
        return {"keys": None, "hist": None, "amps": _state_of_shot(_circuit(case, seed), seed, 0)}
    if not case["amps"]:
        return None
    pset = int(_psets(case, seed)[0]) if f == "sweep" else 0
    return {"keys": None, "amps": _state_of_shot(_circuit(case, seed), seed, 0, pset)}
