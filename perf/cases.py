"""The work that programs have this simulator do, as cases that can be timed and compared.

Every case goes through the entry points of ``paper_2409_14697_gb300.qs`` the way a program
does: it owns the state's memory (a torch tensor handed to ``qs_create_on``), keeps its gate
records, applies circuits and reads amplitudes and expectation values.  The circuit families
and their parameters are those of ``paper_2409_14697_gb300/inputs.py``, the sizes those of
the benchmark's workloads (30-qubit gate sweep, 12-qubit brickwork, 33-qubit families scaled
to passes of a fraction of a second, the paper's QFT and fully connected QAOA, batched
circuits, reductions).  Serving runs the same circuits and reductions on streams of its own
and is not listed apart.

Kinds:
  circuit  a planned call (the default mode) from |0...0> or on the state the program holds;
           with ``read`` also <Z_q> for every qubit and the squared norm, kept at the
           precision of the state's real type (QAOA's <Z_q> are 0 by symmetry: not read)
  sweep    a gate-by-gate call per gate type on the held state
  reduce   norm, <Z_q> for every qubit and the 1024 largest amplitudes of a held state
  batch    many small circuits as one batched launch, every final state copied to the host
"""
import math

import numpy as np
import torch

from paper_2409_14697_gb300 import inputs, qs

BYTES = {"c64": 8, "c128": 16}
QS_DTYPE = {"c64": qs.QS_C64, "c128": qs.QS_C128}
TORCH_DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
REAL = {"c64": np.float32, "c128": np.float64}
TOP_K = 1024


def listed():
    return [
        # a variational program's inner call: a shallow circuit on few qubits, then <Z>
        {"name": "small10 c64", "kind": "circuit", "family": "brickwork", "n": 10, "depth": 6,
         "dtype": "c64", "read": True},
        # the 12-qubit brickwork circuit of the benchmark, state and <Z> read back
        {"name": "brickwork12 c128", "kind": "circuit", "family": "brickwork", "n": 12, "depth": 20,
         "dtype": "c128", "read": True},
        # the headline workload: gate by gate on a 30-qubit complex128 state, six targets of
        # each of the eight types
        {"name": "sweep30 c128", "kind": "sweep", "n": 30, "per_type": 6, "dtype": "c128"},
        # the same on a complex64 state of odd width, every target
        {"name": "sweep27 c64", "kind": "sweep", "n": 27, "per_type": 27, "dtype": "c64"},
        # deep random circuit on a large complex64 state (sampling experiments)
        {"name": "brickwork28 c64", "kind": "circuit", "family": "brickwork", "n": 28, "depth": 40,
         "dtype": "c64", "read": False},
        # Trotterised time evolution on an odd-sized complex64 state, <Z> read after (16 steps: a
        # repeated angle's FP32 rounding adds up to 4e-5 of the norm over 50)
        {"name": "tfim25 c64", "kind": "circuit", "family": "tfim", "n": 25, "depth": 16,
         "dtype": "c64", "read": True},
        # QAOA on a sparse graph on the largest complex64 state here
        {"name": "qaoa30 c64", "kind": "circuit", "family": "qaoa3", "n": 30, "depth": 4,
         "dtype": "c64", "read": False},
        # the paper's QFT on a held complex128 state
        {"name": "qft28 c128", "kind": "circuit", "family": "qft", "n": 28, "depth": 1,
         "dtype": "c128", "read": False},
        # the paper's fully connected QAOA
        {"name": "qaoafull27 c128", "kind": "circuit", "family": "qaoa_full", "n": 27, "depth": 5,
         "dtype": "c128", "read": False},
        # an ordinary double-precision random circuit
        {"name": "brickwork22 c128", "kind": "circuit", "family": "brickwork", "n": 22, "depth": 20,
         "dtype": "c128", "read": True},
        # reading results of a large state
        {"name": "reduce28 c128", "kind": "reduce", "n": 28, "dtype": "c128"},
        # many small circuits at once
        {"name": "batch128 c64", "kind": "batch", "count": 128, "n_lo": 8, "n_hi": 16, "d_lo": 10, "d_hi": 60,
         "dtype": "c64"},
    ]


# Planned families: (smallest n, largest n of complex64, of complex128, depths).  The largest
# are chosen so that a drawn case costs no more than the listed ones.
_FAMILIES = {
    "brickwork": (8, 27, 24, (2, 40)),
    "tfim": (8, 26, 23, (4, 16)),
    "qaoa3": (8, 29, 25, (1, 4)),
    "qft": (8, 29, 28, (1, 1)),
    "qaoa_full": (8, 27, 26, (1, 5)),
}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "circuit", "circuit", "sweep", "reduce", "batch"])
    dtype = rng.choice(["c64", "c128"])
    if kind == "circuit":
        family = rng.choice(sorted(_FAMILIES))
        lo, hi64, hi128, (d0, d1) = _FAMILIES[family]
        n = rng.randint(lo, hi64 if dtype == "c64" else hi128)
        return {"kind": kind, "family": family, "n": n, "depth": _log_int(rng, d0, d1), "dtype": dtype,
                "read": rng.random() < 0.5 and not family.startswith("qaoa")}
    if kind == "sweep":
        return {"kind": kind, "n": rng.randint(8, 29), "per_type": _log_int(rng, 2, 6), "dtype": dtype}
    if kind == "reduce":
        return {"kind": kind, "n": rng.randint(11, 28), "dtype": dtype}
    n_lo = rng.randint(6, 10)
    d_lo = rng.randint(4, 20)
    return {"kind": "batch", "count": _log_int(rng, 16, 128), "n_lo": n_lo, "n_hi": n_lo + rng.randint(0, 6),
            "d_lo": d_lo, "d_hi": d_lo + rng.randint(0, 40), "dtype": dtype}


# ---- inputs -----------------------------------------------------------------------

def _circuit(case, seed):
    n, depth, r = case["n"], case["depth"], inputs.rng(100, seed)
    family = case["family"]
    if family == "brickwork":
        return inputs.brickwork(n, depth, seed=seed)
    if family == "tfim":
        return inputs.tfim(n, depth, dt=float(r.uniform(0.02, 0.08)), h=float(r.uniform(0.5, 1.5)))
    if family == "qaoa3":
        return inputs.qaoa_3regular(n, depth, seed=seed)
    if family == "qaoa_full":
        return inputs.qaoa_complete(n, depth, seed=seed)
    return inputs.qft(n)


def _from_zero(case):
    """The QFT acts on a state the program holds; the other families start from |0...0>."""
    return case["kind"] == "circuit" and case["family"] != "qft"


def _sweep(case, seed):
    """One gate list per type; the targets start at a seeded qubit and go round the register."""
    n, out = case["n"], []
    for name in inputs.SWEEP_GATES:
        r = inputs.rng(101, seed, len(out))
        gates, first, step = [], int(r.integers(n)), max(1, n // case["per_type"])
        for i in range(case["per_type"]):
            q = (first + i * step) % n
            qubits = (q,) if inputs.arity(name) == 1 else (q, (q + 1) % n)
            gates.append((name, qubits, tuple(float(a) for a in r.uniform(0, 2 * math.pi, inputs.n_params(name)))))
        out.append(gates)
    return out


def _batch(case):
    """(qubits, layers) of every circuit: one workload per case, its angles by the seed."""
    r = inputs.rng(102, case["count"], case["n_lo"], case["n_hi"], case["d_lo"], case["d_hi"])
    return [(int(r.integers(case["n_lo"], case["n_hi"] + 1)), int(r.integers(case["d_lo"], case["d_hi"] + 1)))
            for _ in range(case["count"])]


def _batch_circuits(case, seed):
    return [(n, inputs.brickwork(n, d, seed=1000 * (seed % 1000003) + i)) for i, (n, d) in enumerate(_batch(case))]


def _gaussian(n, dtype, seed):
    """Independent normal real and imaginary parts, scaled to unit norm."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    psi = torch.empty(1 << n, dtype=TORCH_DTYPE[dtype], device="cuda")
    v = torch.view_as_real(psi)
    v.normal_(generator=g)
    total = 0.0
    for part in v.view(-1).split(1 << 26):
        total += float(part.double().square().sum())
    v.mul_(1.0 / math.sqrt(total))
    return psi


class _Held:
    """What a program holds: the tensor with the amplitudes and the handle over it."""

    def __init__(self, psi, n, dtype):
        self.psi = psi
        self.h = qs.qs_create_on(n, QS_DTYPE[dtype], psi.data_ptr(), psi.numel() * psi.element_size(),
                                 torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        qs.qs_destroy(self.h)


class _HeldBatch:
    def __init__(self, circuits, dtype):
        self.sizes = [1 << n for n, _ in circuits]
        self.b = qs.qs_batch_create(circuits, QS_DTYPE[dtype])
        self.host = torch.empty(sum(self.sizes), dtype=TORCH_DTYPE[dtype], pin_memory=True)

    def __del__(self):
        qs.qs_batch_destroy(self.b)


def prepare(case, seed):
    kind, dtype = case["kind"], case["dtype"]
    if kind == "batch":
        return {"kind": kind, "held": _HeldBatch(_batch_circuits(case, seed), dtype)}
    n = case["n"]
    if _from_zero(case):
        psi = torch.empty(1 << n, dtype=TORCH_DTYPE[dtype], device="cuda")
    else:
        psi = _gaussian(n, dtype, seed)
    state = {"kind": kind, "held": _Held(psi, n, dtype)}
    if kind == "circuit":
        state.update(records=qs.gate_records(_circuit(case, seed)), options=qs.options(),
                     zero=_from_zero(case), read=case["read"], real=REAL[dtype])
    elif kind == "sweep":
        state.update(records=[qs.gate_records(g) for g in _sweep(case, seed)], options=qs.options(mode=qs.QS_MODE_GATE))
    else:
        state["k"] = min(TOP_K, 1 << n)
    return state


# ---- one pass ---------------------------------------------------------------------

def run(state):
    kind, held = state["kind"], state["held"]
    if kind == "circuit":
        if state["zero"]:
            qs.qs_reset(held.h)
        qs.qs_apply_circuit(held.h, state["records"], state["options"])
        if not state["read"]:
            return {"state": held.psi}
        expz, norm = qs.qs_expectation_z(held.h)
        return {"state": held.psi, "expz": expz.astype(state["real"]), "norm": state["real"](norm)}
    if kind == "sweep":
        for records in state["records"]:
            qs.qs_apply_circuit(held.h, records, state["options"])
        return {"state": held.psi}
    if kind == "reduce":
        norm = qs.qs_norm(held.h)
        expz, _ = qs.qs_expectation_z(held.h)
        index, amplitude = qs.qs_top_amplitudes(held.h, state["k"])
        return {"norm": norm, "expz": expz, "index": index.view(np.int64), "amplitude": amplitude}
    qs.qs_batch_run(held.b)
    qs.qs_batch_synchronize(held.b)
    lib, at, size = qs.load(), held.host.data_ptr(), held.host.element_size()
    for i, count in enumerate(held.sizes):
        if lib.qs_batch_amplitudes(held.b, i, 0, count, at) != qs.QS_OK:
            raise qs.QsError(qs.QS_ERR_CUDA, lib.qs_last_error().decode())
        at += count * size
    return {"states": held.host}


# ---- what a pass cannot do without --------------------------------------------------

# Real operations per amplitude that a gate changes and the share of the amplitudes that it
# changes: complex 2x2 rows, phases, moves.
_GATE_WORK = {"h": (4, 1), "x": (0, 1), "rz": (6, 1), "rx": (6, 1), "u3": (14, 1), "cnot": (0, 0.5), "cz": (0, 0.25),
              "swap": (0, 0.5), "cu3": (14, 0.5), "cp": (6, 0.25), "rzz": (6, 1)}


def _gate_flops(names, n):
    return sum(_GATE_WORK[g][0] * _GATE_WORK[g][1] for g in names) * 2.0 ** n


def work(case):
    B, kind = BYTES[case["dtype"]], case["kind"]
    if kind == "batch":
        sizes = _batch(case)
        return {"bytes": sum(B * 2.0 ** n for n, _ in sizes),
                "flops": sum(_gate_flops(["u3"] * (n * d), n) for n, d in sizes)}
    n = case["n"]
    size = B * 2.0 ** n
    if kind == "circuit":  # the state written once, and read once unless it starts from |0...0>
        return {"bytes": size * (1 if _from_zero(case) else 2), "flops": _gate_flops([g[0] for g in _circuit(case, 1)], n)}
    if kind == "sweep":  # gate by gate: each gate by itself reads and writes what it changes
        names = [g[0] for gates in _sweep(case, 1) for g in gates]
        return {"bytes": sum(2 * size * _GATE_WORK[g][1] for g in names), "flops": _gate_flops(names, n)}
    # norm, <Z_q> and the largest amplitudes are separate calls: each reads the state once
    return {"bytes": 3 * size, "flops": (4 + n) * 2.0 ** n}


# ---- the same in 64 bits with plain torch -----------------------------------------------

def _matrix(name, p):
    """2x2 matrices as ((a, b), (c, d)); for controlled gates the target's."""
    e = lambda x: complex(math.cos(x), math.sin(x))  # noqa: E731
    if name == "h":
        s = math.sqrt(0.5)
        return (s, s), (s, -s)
    if name in ("x", "cnot"):
        return (0, 1), (1, 0)
    if name == "rx":
        c, s = math.cos(p[0] / 2), math.sin(p[0] / 2)
        return (c, -1j * s), (-1j * s, c)
    if name == "rz":
        return (e(-p[0] / 2), 0), (0, e(p[0] / 2))
    if name in ("u3", "cu3"):
        t, ph, la = p
        c, s = math.cos(t / 2), math.sin(t / 2)
        return (c, -e(la) * s), (e(ph) * s, e(ph + la) * c)
    raise ValueError(name)


def _apply(psi, name, q, p):
    if len(q) == 1 or name in ("cnot", "cu3"):
        target = q[-1]
        v = psi.view(-1, 2, 1 << target)
        a, b = v[:, 0], v[:, 1]
        if len(q) == 2:  # the halves where the control is 1
            c = q[0]
            if c > target:
                w = psi.view(-1, 2, 1 << (c - target - 1), 2, 1 << target)[:, 1]
                a, b = w[:, :, 0], w[:, :, 1]
            else:
                w = psi.view(-1, 2, 1 << (target - c - 1), 2, 1 << c)
                a, b = w[:, 0, :, 1], w[:, 1, :, 1]
        (m00, m01), (m10, m11) = _matrix(name, p)
        if m01 == 0 and m10 == 0:
            a.mul_(m00)
            b.mul_(m11)
            return
        old = a.clone()
        a.mul_(m00).add_(b, alpha=m01)
        b.mul_(m11).add_(old, alpha=m10)
        return
    lo, hi = min(q), max(q)
    w = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
    if name == "cz":
        w[:, 1, :, 1].neg_()
    elif name == "cp":
        w[:, 1, :, 1].mul_(complex(math.cos(p[0]), math.sin(p[0])))
    elif name == "rzz":
        same = complex(math.cos(p[0] / 2), -math.sin(p[0] / 2))
        w[:, 0, :, 0].mul_(same)
        w[:, 1, :, 1].mul_(same)
        w[:, 0, :, 1].mul_(same.conjugate())
        w[:, 1, :, 0].mul_(same.conjugate())
    elif name == "swap":
        old = w[:, 0, :, 1].clone()
        w[:, 0, :, 1].copy_(w[:, 1, :, 0])
        w[:, 1, :, 0].copy_(old)
    else:
        raise ValueError(name)


def _zero_state(n):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    return psi


def _readings(psi, n):
    """<Z_q> for every q and the squared norm: halves of the probabilities, pair by pair."""
    prob = torch.view_as_real(psi).square().sum(-1)
    expz = [0.0] * n
    for q in reversed(range(n)):  # the highest qubit is split off first
        half = prob.view(2, -1)
        expz[q] = float(half[0].sum() - half[1].sum())
        prob = half[0] + half[1]
    return np.array(expz), float(prob)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for n, gates in _batch_circuits(case, seed):
            psi = _zero_state(n)
            for name, q, p in gates:
                _apply(psi, name, q, p)
            out.append(psi)
        return {"states": torch.cat(out)}
    n = case["n"]
    if _from_zero(case):
        psi = _zero_state(n)
    else:
        psi = _gaussian(n, case["dtype"], seed).to(torch.complex128)
    if kind == "reduce":
        expz, norm = _readings(psi, n)
        return {"norm": norm, "expz": expz, "index": None, "amplitude": None}
    gates = _circuit(case, seed) if kind == "circuit" else [g for part in _sweep(case, seed) for g in part]
    for name, q, p in gates:
        _apply(psi, name, q, p)
    if kind == "circuit" and case["read"]:
        expz, norm = _readings(psi, n)
        return {"state": psi, "expz": expz, "norm": norm}
    return {"state": psi}
