"""Timed cases of the state-vector simulator: what a program that uses it has it do.

Every case goes through the public entry points of ``paper_2406_14084_gb300.qs``.  Circuit
cases start from a computational basis state, apply a circuit and hand back all amplitudes
in logical qubit order; readout cases start from a given state and hand back what was read.
Angles, basis states, qubit choices, input states and uniforms come from the seed alone.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2406_14084_gb300 import qs
from paper_2406_14084_gb300 import workloads as W
from paper_2406_14084_gb300.workloads import Gate

QS_DTYPE = {"c64": qs.QS_C64, "c128": qs.QS_C128}
TORCH_DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
AMP_BYTES = {"c64": 8, "c128": 16}


# ------------------------------------------------------------------------------ the cases

def listed():
    return [
        # the inner call of a variational loop: new angles every time, so one call plans, runs
        # and reads the energy of a small hardware-efficient ansatz (latency and host work)
        {"name": "vqe12_c64", "kind": "vqe", "n": 12, "layers": 4, "dtype": "c64"},
        # the paper's correctness configuration: 200 mixed gates on 20 qubits, planned once
        {"name": "random20_c128", "kind": "circuit", "family": "random", "n": 20, "size": 200, "dtype": "c128",
         "mode": "plain"},
        # QAOA on the complete graph (the paper's second application), diagonal-heavy
        {"name": "qaoa23_c64", "kind": "circuit", "family": "qaoa", "n": 23, "size": 4, "dtype": "c64", "mode": "plain"},
        # the QFT at the paper's precision (the headline circuit), few gates per pass
        {"name": "qft28_c128", "kind": "circuit", "family": "qft", "n": 28, "size": 1, "dtype": "c128", "mode": "plain"},
        # dense random layers at the paper's precision: every pass full of rotations
        {"name": "layered25_c128", "kind": "circuit", "family": "layered", "n": 25, "size": 20, "dtype": "c128",
         "mode": "plain"},
        # the same at single precision, a large state
        {"name": "layered28_c64", "kind": "circuit", "family": "layered", "n": 28, "size": 20, "dtype": "c64",
         "mode": "plain"},
        # complex128 states with double-float arithmetic (options.arith)
        {"name": "layered26_c128_df", "kind": "circuit", "family": "layered", "n": 26, "size": 12, "dtype": "c128",
         "mode": "df"},
        # 6-qubit blocks on the tensor cores (options.tc)
        {"name": "layered27_c64_tc", "kind": "circuit", "family": "layered", "n": 27, "size": 12, "dtype": "c64",
         "mode": "tc"},
        # many uneven variational circuits in one batch, energies only
        {"name": "batch64_c64", "kind": "batch", "count": 64, "nmin": 10, "nmax": 20, "dtype": "c64"},
        # readouts of one large state: norm, 3-qubit marginals, ZZ-chain energy, 4096 samples
        {"name": "readout28_c64", "kind": "readout", "n": 28, "shots": 4096, "dtype": "c64"},
        # the histogram of a 10-qubit register (phase estimation, arithmetic circuits)
        {"name": "marginals27_c64", "kind": "marginals", "n": 27, "nq": 10, "dtype": "c64"},
        # the energy of a Heisenberg chain: XX + YY + ZZ on every bond and a field
        {"name": "heisenberg26_c64", "kind": "heisenberg", "n": 26, "dtype": "c64"},
    ]


def draw(rng: random.Random):
    kind = rng.choice(["vqe", "random", "qaoa", "qft", "layered", "layered", "df", "tc", "batch", "readout", "marginals",
                       "heisenberg"])
    dtype = rng.choice(["c64", "c128"])
    wide = 1 if dtype == "c64" else 0  # one more qubit at half the bytes
    if kind == "vqe":
        return {"kind": "vqe", "n": rng.randint(6, 16), "layers": rng.randint(1, 8), "dtype": dtype}
    if kind == "random":
        return {"kind": "circuit", "family": "random", "n": rng.randint(14, 24), "size": rng.randint(40, 300),
                "dtype": dtype, "mode": "plain"}
    if kind == "qaoa":
        return {"kind": "circuit", "family": "qaoa", "n": rng.randint(15, 23), "size": rng.randint(1, 4), "dtype": dtype,
                "mode": "plain"}
    if kind == "qft":
        return {"kind": "circuit", "family": "qft", "n": rng.randint(15, 27 + wide), "size": 1, "dtype": dtype,
                "mode": "plain"}
    if kind == "layered":
        return {"kind": "circuit", "family": "layered", "n": rng.randint(15, 24 + 3 * wide), "size": rng.randint(2, 20),
                "dtype": dtype, "mode": "plain"}
    if kind == "df":
        return {"kind": "circuit", "family": "layered", "n": rng.randint(18, 26), "size": rng.randint(2, 12),
                "dtype": "c128", "mode": "df"}
    if kind == "tc":
        return {"kind": "circuit", "family": "layered", "n": rng.randint(18, 27), "size": rng.randint(2, 12),
                "dtype": "c64", "mode": "tc"}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(8, 64), "nmin": rng.randint(8, 12), "nmax": rng.randint(13, 19),
                "dtype": dtype}
    if kind == "readout":
        return {"kind": "readout", "n": rng.randint(16, 27 + wide), "shots": rng.randint(100, 4096), "dtype": dtype}
    if kind == "marginals":
        return {"kind": "marginals", "n": rng.randint(16, 26), "nq": rng.randint(1, 14), "dtype": dtype}
    return {"kind": "heisenberg", "n": rng.randint(14, 25), "dtype": dtype}


# ------------------------------------------------------------------------------ inputs

def _circuit(case, seed):
    n, size, family = case["n"], case["size"], case["family"]
    if family == "random":
        return W.random_circuit(n, size, seed)
    if family == "qaoa":
        return W.qaoa_complete(n, size, seed)
    if family == "qft":
        return W.qft(n)
    return W.layered(n, size, seed)


def _batch_circuits(case, seed):
    """Uneven circuits whose sizes are the case's (the same for every seed); angles from the seed."""
    sizes = W.SplitMix64(1004 + case["count"])
    span = case["nmax"] - case["nmin"] + 1
    out = []
    for i in range(case["count"]):
        n, layers = case["nmin"] + sizes.below(span), 2 + sizes.below(11)
        out.append((n, W.vqe_circuit(n, layers, seed * 4099 + i)))
    return out


def _options(case):
    mode = case.get("mode", "plain")
    o = {"dtype": QS_DTYPE[case["dtype"]]}
    if mode == "df":
        o["arith"] = qs.QS_ARITH_DF
    elif mode == "tc":
        o["tc"] = qs.QS_TC_BF16X3
    return qs.options(**o)


def _input_state(case, seed):
    """What a variational circuit for a chain in a field leaves behind: a product state of tilted
    spins with a correlated rest (a complex Gaussian tenth of the weight), of norm about 1."""
    n, dtype = case["n"], TORCH_DTYPE[case["dtype"]]
    rng = W.SplitMix64(seed + 11)
    a = torch.ones(1, dtype=dtype, device="cuda")
    for _ in range(n):  # qubit 0 first: each further qubit doubles the index range
        t, f = (0.1 + 0.9 * rng.uniform()) * math.pi / 6, (rng.uniform() - 0.5) * math.pi / 2
        a = torch.cat((a * math.cos(t), a * (math.sin(t) * complex(math.cos(f), math.sin(f)))))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    noise = torch.randn(1 << n, dtype=dtype, device="cuda", generator=gen)
    return a.mul_(math.sqrt(0.9)).add_(noise, alpha=math.sqrt(0.1) * 2.0 ** (-n / 2))


def _heisenberg(n, seed):
    rng = W.SplitMix64(seed)
    terms = []
    for i in range(n - 1):
        j = 0.5 + rng.uniform()
        pair = (1 << i) | (1 << (i + 1))
        terms += [(j, pair, 0), (j, pair, pair), (j, 0, pair)]
    terms += [(rng.uniform() - 0.5, 0, 1 << i) for i in range(n)]
    return terms


def _marginal_qubits(case, seed):
    return W.SplitMix64(seed + 77).distinct(case["n"], case["nq"])


class _Held:
    """What a program keeps: the state's memory and handle, its plan or batch; given back with it."""

    def __init__(self, **kw):
        self.state = self.plan = self.batch = None
        self.__dict__.update(kw)

    def __del__(self):
        try:
            if self.plan is not None:
                qs.qs_plan_destroy(self.plan)
            if self.state is not None:
                qs.qs_destroy(self.state)
            if self.batch is not None:
                qs.qs_batch_destroy(self.batch)
        except Exception:
            pass


def _on_device(case, amps):
    return qs.qs_create_from_buffer(case["n"], QS_DTYPE[case["dtype"]], amps.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)


def prepare(case, seed):
    kind, n = case["kind"], case.get("n")
    number = np.float32 if case["dtype"] == "c64" else np.float64
    if kind == "batch":
        circuits = _batch_circuits(case, seed)
        o = _options(case)
        o.graph = 1
        return _Held(kind=kind, number=number, batch=qs.qs_batch_create(circuits, o), count=len(circuits),
                     terms=W.zz_chain_hamiltonian(case["nmax"]))
    if kind in ("circuit", "vqe"):
        amps = torch.empty(1 << n, dtype=TORCH_DTYPE[case["dtype"]], device="cuda")
        h = _Held(kind=kind, number=number, amps=amps, state=_on_device(case, amps), options=_options(case))
        if kind == "circuit":
            h.x0 = W.random_basis(n, seed)
            h.plan = qs.qs_fuse(_circuit(case, seed), n, h.options)
        else:
            h.gates = W.vqe_circuit(n, case["layers"], seed)
            h.terms = W.zz_chain_hamiltonian(n)
        return h
    amps = _input_state(case, seed)
    h = _Held(kind=kind, number=number, amps=amps, state=_on_device(case, amps))
    if kind == "readout":
        r = W.SplitMix64(seed + 5)
        h.qubits = r.distinct(n, 3)
        h.terms = W.zz_chain_hamiltonian(n)
        h.u = np.array([r.uniform() for _ in range(case["shots"])])
    elif kind == "marginals":
        h.qubits = _marginal_qubits(case, seed)
    else:
        h.terms = _heisenberg(n, seed)
    return h


# ------------------------------------------------------------------------------ one pass

def run(h):
    if h.kind == "circuit":
        qs.qs_set_basis(h.state, h.x0)
        qs.qs_apply_plan(h.state, h.plan)
        qs.qs_canonicalize(h.state)  # amplitudes in logical order
        return h.amps
    num = h.number  # a number read from a complex64 state carries the state's precision
    if h.kind == "vqe":
        qs.qs_set_basis(h.state, 0)
        qs.qs_apply_circuit(h.state, h.gates, h.options)
        e = qs.qs_expect_pauli_sum(h.state, h.terms)
        return {"state": h.amps, "energy": num(e.real)}
    if h.kind == "batch":
        return num(qs.qs_apply_batch(h.batch, h.terms, h.count))
    if h.kind == "readout":
        return {"norm": num(qs.qs_norm2(h.state)), "probs": num(qs.qs_probs(h.state, h.qubits)),
                "energy": num(qs.qs_expect_pauli_sum(h.state, h.terms).real), "samples": qs.qs_sample(h.state, h.u)}
    if h.kind == "marginals":
        return num(qs.qs_probs(h.state, h.qubits))
    return num(qs.qs_expect_pauli_sum(h.state, h.terms).real)


# ------------------------------------------------------------------------------ what a pass cannot do without

def _gate_flops(g: Gate) -> float:
    """Real operations per amplitude of one gate on its own, its zeros and ones left out."""
    if g.kind in ("X", "CX", "SWAP"):
        return 0.0
    if g.kind == "H":
        return 4.0
    if g.kind == "RY":
        return 6.0
    if g.kind in ("CZ", "CP"):
        return 1.5
    if g.kind in ("S", "T"):
        return 3.0
    if g.kind in ("RZ", "RZZ"):
        return 6.0
    return 14.0  # a complex 2x2 matrix


def work(case):
    kind = case["kind"]
    if kind == "batch":
        flops = sum(math.ldexp(sum(_gate_flops(g) for g in gates) + 4, n) for n, gates in _batch_circuits(case, 0))
        return {"bytes": 8 * case["count"], "flops": flops}
    amps = 1 << case["n"]
    size = amps * AMP_BYTES[case["dtype"]]
    if kind == "circuit":
        # written once: the input is one basis index
        return {"bytes": size, "flops": amps * sum(_gate_flops(g) for g in _circuit(case, 1))}
    if kind == "vqe":
        gates = W.vqe_circuit(case["n"], case["layers"], 1)
        return {"bytes": size, "flops": amps * (sum(_gate_flops(g) for g in gates) + 4.0)}
    return {"bytes": size, "flops": 4.0 * amps}  # read once


# ------------------------------------------------------------------------------ the same in 64 bits

def _matrix(g: Gate):
    """The 2x2 matrix of a gate kind that is not diagonal, in 64 bits."""
    p = g.params
    if g.kind == "H":
        r = math.sqrt(0.5)
        return [[r, r], [r, -r]]
    if g.kind in ("X", "CX"):
        return [[0, 1], [1, 0]]
    if g.kind == "RX":
        c, s = math.cos(p[0] / 2), math.sin(p[0] / 2)
        return [[c, -1j * s], [-1j * s, c]]
    if g.kind == "RY":
        c, s = math.cos(p[0] / 2), math.sin(p[0] / 2)
        return [[c, -s], [s, c]]
    if g.kind == "U3":
        c, s = math.cos(p[0] / 2), math.sin(p[0] / 2)
        ph, la = p[1], p[2]
        return [[c, -np.exp(1j * la) * s], [np.exp(1j * ph) * s, np.exp(1j * (ph + la)) * c]]
    return None


def _phase(t):
    return complex(math.cos(t), math.sin(t))


def _apply(a, g: Gate):
    if g.kind in ("S", "T", "RZ"):
        q = g.targets[0]
        v = a.view(-1, 2, 1 << q)
        if g.kind == "RZ":
            v[:, 0] *= _phase(-g.params[0] / 2)
        v[:, 1] *= 1j if g.kind == "S" else _phase(math.pi / 4 if g.kind == "T" else g.params[0] / 2)
        return
    if g.kind in ("CZ", "CP", "RZZ", "SWAP", "CX"):
        qa, qb = (g.targets if len(g.targets) == 2 else (g.targets[0], g.controls[0]))
        lo, hi = min(qa, qb), max(qa, qb)
        v = a.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        if g.kind == "CZ":
            v[:, 1, :, 1] *= -1
        elif g.kind == "CP":
            v[:, 1, :, 1] *= _phase(g.params[0])
        elif g.kind == "RZZ":
            e0, e1 = _phase(-g.params[0] / 2), _phase(g.params[0] / 2)
            v[:, 0, :, 0] *= e0
            v[:, 1, :, 1] *= e0
            v[:, 0, :, 1] *= e1
            v[:, 1, :, 0] *= e1
        elif g.kind == "SWAP":
            t = v[:, 0, :, 1].clone()
            v[:, 0, :, 1] = v[:, 1, :, 0]
            v[:, 1, :, 0] = t
        else:  # CX: the target flips where the control (qb) is 1
            one, two = (v[:, 1, :, 0], v[:, 1, :, 1]) if qb == hi else (v[:, 0, :, 1], v[:, 1, :, 1])
            t = one.clone()
            one.copy_(two)
            two.copy_(t)
        return
    m = _matrix(g)
    v = a.view(-1, 2, 1 << g.targets[0])
    lo = v[:, 0] * m[0][0] + v[:, 1] * m[0][1]
    v[:, 1] = v[:, 0] * m[1][0] + v[:, 1] * m[1][1]
    v[:, 0] = lo


def _exact_circuit(n, gates, x0):
    a = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    a[x0] = 1
    for g in gates:
        _apply(a, g)
    return a


def _exact_qft(n, x0):
    """2^{-n/2} exp(2 pi i x y / 2^n) at the bit-reversed index of y (no final swaps)."""
    i = torch.arange(1 << n, dtype=torch.int64, device="cuda")
    y = torch.zeros_like(i)
    for q in range(n):
        y |= ((i >> q) & 1) << (n - 1 - q)
    turn = ((y * x0) & ((1 << n) - 1)).double() * (2.0 * math.pi / (1 << n))
    return torch.polar(torch.full_like(turn, 2.0 ** (-n / 2)), turn)


def _exact_energy(a, n, terms):
    """Real part of <a| sum_t c_t P_t |a>, P|x> = i^{#Y} (-1)^{popcount(x & z)} |x ^ xmask>."""
    x = torch.arange(1 << n, dtype=torch.int64, device=a.device)
    total = 0.0
    groups = {}
    for c, xm, zm in terms:
        groups.setdefault(xm, []).append((c, zm))
    for xm, part in groups.items():
        v = (a.conj()[x ^ xm] * a) if xm else (a.real.square() + a.imag.square()).to(a.dtype)
        for c, zm in part:
            s = torch.zeros_like(x)
            for q in range(n):
                if zm >> q & 1:
                    s ^= (x >> q) & 1
            w = torch.where(s == 1, -v, v).sum().item()
            total += (c * (1j ** bin(xm & zm).count("1")) * w).real
    return total


def _exact_probs(p, n, qubits):
    x = torch.arange(1 << n, dtype=torch.int64, device=p.device)
    m = torch.zeros_like(x)
    for j, q in enumerate(qubits):
        m |= ((x >> q) & 1) << j
    return torch.zeros(1 << len(qubits), dtype=torch.float64, device=p.device).scatter_add_(0, m, p).cpu().numpy()


def exact(case, seed):
    kind, n = case["kind"], case.get("n")
    if kind == "circuit":
        if case["family"] == "qft":
            return _exact_qft(n, W.random_basis(n, seed))
        return _exact_circuit(n, _circuit(case, seed), W.random_basis(n, seed))
    if kind == "vqe":
        a = _exact_circuit(n, W.vqe_circuit(n, case["layers"], seed), 0)
        return {"state": a, "energy": _exact_energy(a, n, W.zz_chain_hamiltonian(n))}
    if kind == "batch":
        out = []
        for m, gates in _batch_circuits(case, seed):
            out.append(_exact_energy(_exact_circuit(m, gates, 0), m, W.zz_chain_hamiltonian(m)))
        return np.array(out)
    a = _input_state(case, seed).to(torch.complex128)
    if kind == "heisenberg":
        return _exact_energy(a, n, _heisenberg(n, seed))
    p = a.real.square() + a.imag.square()
    if kind == "marginals":
        return _exact_probs(p, n, _marginal_qubits(case, seed))
    qubits = W.SplitMix64(seed + 5).distinct(n, 3)
    return {"norm": p.sum().item(), "probs": _exact_probs(p, n, qubits),
            "energy": _exact_energy(a, n, W.zz_chain_hamiltonian(n)), "samples": None}
