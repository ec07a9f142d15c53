"""What a program built on this library has it do, as cases that can be timed.

Every case is one pass through the public calls of
``paper_2105_01533_gb300.sps``: a circuit applied to a state, and the state
(with what else the program reads) brought back into the program's own device
tensors. Families, and what they stand for:

  mix      a random circuit of X / CNOT / Toffoli, Z / S / T / controlled Rz and
           some H from |0..0>, then one probability and the state sorted by label
           (the 24-qubit plain workload and the circuits of the batched one)
  gates    every gate code with up to two controls on 12 to 20 qubits after a
           layer of H: branching passes on growing states, real and complex
           matrices; read back as a dense statevector
  hop      one Trotter step of a fermion Hamiltonian under Jordan-Wigner: Pauli
           exponentials X Z..Z X and Y Z..Z Y, Z Z, and a layer of Rz, on a
           particle-number sector that goes on from step to step
  adder    the reversible-arithmetic workload: superpose, add, phase, un-add,
           with a registered readout; from a reset
  arith    the same arithmetic on a state that the program loaded (any number of
           entries): compute in one call, uncompute in the next
  measure  superpose and add, read the marginal of every result bit, measure
           some of them with collapse
  fill     the number-conserving workload from a reset: the sector fills in the
           first layers and then keeps its labels
  sector   layers of it on a full sector resumed from a saved state; the state
           goes on from pass to pass
  batch    independent circuits in one persistent launch, every state read back

Circuits come from the seeded generators of ``workloads``; sizes are those of
this repository's benchmark and tests, or lie between them.
"""

from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2105_01533_gb300 import sps
from paper_2105_01533_gb300 import workloads as W

EPS = 1e-14   # prune threshold of every workload of the benchmark


def listed():
    return [
        # the smallest call: a short circuit whose state never leaves one block
        dict(name="mix20-short", family="mix", qubits=20, gates=200, log2cap=8),
        # the plain workload: 2,000 gates, at most 4,096 nonzeros
        dict(name="mix24", family="mix", qubits=24, gates=2000, log2cap=12),
        # the widest circuits of the batched workload, run alone: 128-bit labels
        dict(name="mix100", family="mix", qubits=100, gates=5000, log2cap=16),
        # dense states up to 2^20 entries, every gate code, one pass per branching gate
        dict(name="gates20", family="gates", qubits=20, gates=96, controls=1),
        # 24 modes, 6 particles (134,596 labels), 12 hopping terms a step
        dict(name="hop24", family="hop", qubits=24, modes=6, terms=12),
        # 65,536 entries, everything in L2: launches and host time count
        dict(name="adder67-w16", family="adder", bits=32, width=16),
        # the benchmark's headline: 16.8 M entries, larger than L2
        dict(name="adder67-w24", family="adder", bits=32, width=24),
        # 64-bit labels, an odd number of loaded entries
        dict(name="arith59", family="arith", bits=28, entries=5000011),
        # 1 M entries, 32 marginals, 4 measurements
        dict(name="measure67", family="measure", bits=32, width=20, measured=4),
        # 64 modes, 4 particles (635,376 labels) from a reset
        dict(name="givens64-fill", family="fill", qubits=64, modes=4, layers=32),
        # 64 modes, 6 particles (74,974,368 labels), a state of 2.4 GB
        dict(name="givens64-m6", family="sector", qubits=64, modes=6, layers=2),
        # circuits of the batched workload, all states read back
        dict(name="batch256", family="batch", circuits=256, depth=2000, log2cap=13),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["mix", "gates", "hop", "adder", "arith", "measure", "fill", "sector",
                         "batch"])
    if family == "mix":
        return dict(family=family, qubits=rng.randint(20, 100), gates=_log_uniform(rng, 200, 5000),
                    log2cap=rng.randint(8, 16))
    if family == "gates":
        return dict(family=family, qubits=rng.randint(12, 20), gates=_log_uniform(rng, 40, 160),
                    controls=rng.randint(1, 2))
    if family == "hop":
        return dict(family=family, qubits=rng.randint(16, 26), modes=rng.randint(2, 6),
                    terms=rng.randint(4, 16))
    if family == "adder":
        return dict(family=family, bits=rng.randint(26, 40), width=rng.randint(6, 24))
    if family == "arith":
        return dict(family=family, bits=rng.randint(25, 40),
                    entries=_log_uniform(rng, 3000, 16000000))
    if family == "measure":
        return dict(family=family, bits=rng.randint(24, 40), width=rng.randint(10, 22),
                    measured=rng.randint(1, 6))
    if family == "fill":
        return dict(family=family, qubits=rng.randint(24, 80), modes=rng.randint(2, 4),
                    layers=rng.randint(12, 48))
    if family == "sector":
        qubits = rng.randint(24, 100)
        modes = max(k for k in range(2, 7) if math.comb(qubits, k) <= 20000000)
        return dict(family=family, qubits=qubits, modes=rng.randint(2, modes),
                    layers=rng.randint(1, 6))
    return dict(family=family, circuits=_log_uniform(rng, 24, 256),
                depth=_log_uniform(rng, 300, 2000), log2cap=rng.randint(8, 13))


# ---- inputs -----------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _amplitudes(n, seed):
    """n amplitudes of one norm-1 state, complex Gaussian."""
    a = torch.randn(2, n, dtype=torch.float64, device="cuda", generator=_gen(seed))
    a /= torch.linalg.vector_norm(a)
    return a[0], a[1]


def _sector_labels(qubits, modes):
    """(hi, lo) words of every label of `qubits` bits with `modes` ones, sorted
    by their value as whole numbers."""
    hi = torch.zeros(1, dtype=torch.int64, device="cuda")
    lo = torch.zeros(1, dtype=torch.int64, device="cuda")
    top = torch.zeros(1, dtype=torch.int64, device="cuda")   # highest set bit + 1
    for k in range(modes):   # labels with k + 1 ones from those with k: add a higher bit
        count = qubits - (modes - 1 - k) - top
        rep = torch.repeat_interleave(torch.arange(len(top), device="cuda"), count)
        start = torch.cumsum(count, 0) - count
        bit = top[rep] + torch.arange(len(rep), device="cuda") - start[rep]
        one = torch.ones_like(bit)
        lo = lo[rep] | torch.where(bit < 64, one << (bit % 64), 0)
        hi = hi[rep] | torch.where(bit >= 64, one << (bit % 64), 0)
        top = bit + 1
    order = torch.argsort(lo ^ (-1 << 63), stable=True)
    order = order[torch.argsort(hi[order], stable=True)] if qubits > 64 else order
    return hi[order], lo[order]


class _State:
    """A program's handle: the library's state, its circuit, and the tensors
    that it reads the state back into."""

    def __init__(self, qubits, capacity):
        self.sv = sps.SparseState(qubits, capacity)
        self.wide = qubits > 63
        self.cap = capacity
        self.words = torch.zeros(2, capacity, dtype=torch.int64, device="cuda")
        self.amps = torch.zeros(2, capacity, dtype=torch.float64, device="cuda")
        self.out = torch.zeros(64, dtype=torch.float64, device="cuda")

    def read(self):
        """The state in the library's order: (hi, lo, re, im), hi None with
        64-bit labels."""
        hi = self.words[0] if self.wide else None
        n = sps.sps_get_amplitudes(self.sv.handle, hi, self.words[1], self.amps[0], self.amps[1],
                                   self.cap)
        return (hi[:n] if self.wide else None, self.words[1, :n], self.amps[0, :n],
                self.amps[1, :n])

    def read_sorted(self, one_word):
        """The state as a table of `capacity` rows sorted by label, rows that
        hold no entry with label -1 and amplitude 0; one_word: the low words
        alone tell the labels apart."""
        n = len(self.read()[1])
        if n < self.cap:
            self.words[:, n:] = -1
            self.amps[:, n:] = 0.0
        (hi, lo), (re, im) = self.words, self.amps
        if one_word or not self.wide:
            lo, order = torch.sort(lo)
        else:
            order = torch.argsort(lo)
            order = order[torch.argsort(hi[order], stable=True)]
            lo = lo[order]
        got = {"lo": lo, "re": re[order], "im": im[order]}
        if self.wide:
            got["hi"] = hi[order]
        return got

    def slot(self, i):
        return self.out.data_ptr() + 8 * i


def _bit(q):
    return (1 << q, 0) if q < 64 else (0, 1 << (q - 64))


def _mix_gates(case, seed):
    budget = max(0, case["log2cap"] - 8)
    return W.random_mix_fast(1000003 * seed + 17, case["qubits"], case["gates"], budget)


def _all_gates(case, seed):
    """H on all but four qubits, then every gate code, 30% of them branching."""
    n = case["qubits"]
    return np.concatenate([W.to_array([W.H(q) for q in range(n - 4)]),
                           W.random_all_gates(seed + 5, n, case["gates"],
                                              max_controls=case["controls"])])


def _hop_terms(case, seed):
    """(x, z, theta) strings of one Trotter step and the Rz layer after them."""
    rng = W.SplitMix64(seed * 7919 + 3)
    n, strings = case["qubits"], []
    for _ in range(case["terms"]):
        p, q = sorted(rng.distinct(n, 2))
        th = 0.1 + 0.4 * rng.uniform()
        ends = (1 << p) | (1 << q)
        between = (1 << q) - (1 << (p + 1))
        strings.append((ends, between, th))
        strings.append((ends, between | ends, th))
        a, b = rng.distinct(n, 2)
        strings.append((0, (1 << a) | (1 << b), rng.angle()))
    return strings, W.to_array([W.Rz(q, rng.angle()) for q in range(n)])


def _adder_parts(case, seed):
    """(superpose, load and add and phase, un-add) of the adder workload."""
    width = case.get("width", 1)
    wl = W.adder_workload(seed=seed + 1, nbits=case["bits"], width=width)
    split = len(wl.gates) - (6 * case["bits"] + 1)
    return wl, wl.gates[:width], wl.gates[width:split], wl.gates[split:]


def _adder_readout(case):
    """The benchmark's readout: the low (at most 16) bits of register a are 0."""
    return (1 << min(16, case["width"])) - 1, 0


def _layers(case, seed):
    """The workload's layers without the X gates that start it, and those."""
    g = W.givens_workload(seed=seed + 2, nqubits=case["qubits"], modes=case["modes"],
                          layers=case["layers"])
    return g[:case["modes"]], g[case["modes"]:]


def _arith_labels(case, seed):
    """Distinct labels with any value in registers a and b, other qubits 0."""
    bits, n = case["bits"], case["entries"]
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    odd = 2 * (W.SplitMix64(seed).below(1 << (bits - 1))) + 1
    a = (i * odd + 12345) & ((1 << bits) - 1)
    b = torch.randint(0, 1 << bits, (n,), dtype=torch.int64, device="cuda", generator=_gen(seed))
    lo = a | (b << bits)
    hi = b >> (64 - bits) if 2 * bits > 64 else torch.zeros_like(b)
    return hi, lo


def _load(st, hi, lo, seed):
    re, im = _amplitudes(len(lo), seed)
    sps.sps_set_amplitudes(st.sv.handle, hi if st.wide else None, lo, re, im, len(lo))


def _measure_draws(case, seed):
    """(qubit offset in the result register, r) of each measurement."""
    rng = W.SplitMix64(seed + 77)
    return [(k, 0.05 + 0.9 * rng.uniform()) for k in range(case["measured"])]


def _batch_circuits(case, seed):
    return W.batched_workload_fast(case["circuits"], first_seed=1 + seed * case["circuits"],
                                   depth=(200, case["depth"]), log2_cap=(8, case["log2cap"]))


def prepare(case, seed):
    family = case["family"]
    if family == "mix":
        st = _State(case["qubits"], 1 << case["log2cap"])
        st.gates = _mix_gates(case, seed)
    elif family == "gates":
        st = _State(case["qubits"], 1 << case["qubits"])
        st.gates = _all_gates(case, seed)
        st.dense = torch.zeros(2, 1 << case["qubits"], dtype=torch.float64, device="cuda")
    elif family == "hop":
        n = math.comb(case["qubits"], case["modes"])
        st = _State(case["qubits"], 2 * n)
        st.strings, st.gates = _hop_terms(case, seed)
        _load(st, *_sector_labels(case["qubits"], case["modes"]), seed)
    elif family == "adder":
        wl, _, _, _ = _adder_parts(case, seed)
        st = _State(wl.layout.nqubits, 1 << case["width"])
        st.gates = wl.gates
        st.mask, st.value = _adder_readout(case), (0, 0)
        st.sv.set_readout(st.mask, st.value)
    elif family == "arith":
        wl, _, st_fwd, st_back = _adder_parts(case, seed)
        st = _State(wl.layout.nqubits, case["entries"])
        st.forward, st.back = st_fwd, st_back
        _load(st, *_arith_labels(case, seed), seed)
    elif family == "measure":
        wl, sup, fwd, _ = _adder_parts(case, seed)
        st = _State(wl.layout.nqubits, 1 << case["width"])
        st.gates = np.concatenate([sup, fwd])
        st.result = wl.layout.b
        st.draws = _measure_draws(case, seed)
    elif family == "fill":
        st = _State(case["qubits"], math.comb(case["qubits"], case["modes"]) + 4096)
        st.gates = np.concatenate(_layers(case, seed))
    elif family == "sector":
        st = _State(case["qubits"], math.comb(case["qubits"], case["modes"]) + 4096)
        st.gates = _layers(case, seed)[1]
        _load(st, *_sector_labels(case["qubits"], case["modes"]), seed)
    else:
        circuits = _batch_circuits(case, seed)
        st = sps.Batch()
        for c in circuits:
            st.add(c.nqubits, c.cap, c.gates, EPS)
        rows = 1 << case["log2cap"]   # a table of every circuit's entries, in its own row
        st.words = torch.zeros(2, len(circuits), rows, dtype=torch.int64, device="cuda")
        st.amps = torch.zeros(2, len(circuits), rows, dtype=torch.float64, device="cuda")
    return _Case(case, st)


class _Case:
    def __init__(self, case, st):
        self.family, self.case, self.st = case["family"], case, st


# ---- one pass -----------------------------------------------------------------------
def run(state):
    return _RUN[state.family](state.case, state.st)


def _run_mix(case, st):
    st.sv.reset()
    st.sv.apply(st.gates, EPS)
    st.sv.probability_async((3, 0), (1, 0), st.slot(0))   # qubit 0 is 1 and qubit 1 is 0
    got = st.read_sorted(case["qubits"] <= 63)
    got["p"] = st.out[:1]
    return got


def _run_gates(case, st):
    st.sv.reset()
    st.sv.apply(st.gates, EPS)
    _, lo, re, im = st.read()
    st.dense.zero_()
    st.dense[0].scatter_(0, lo, re)
    st.dense[1].scatter_(0, lo, im)
    return st.dense


def _run_hop(case, st):
    for x, z, theta in st.strings:
        st.sv.pauli_exp((x, 0), (z, 0), (0, 0), theta, EPS)
    st.sv.apply(st.gates, EPS)
    return st.read_sorted(True)


def _run_adder(case, st):
    st.sv.reset()
    st.sv.apply(st.gates, EPS)
    st.sv.probability_async(st.mask, st.value, st.slot(0))
    hi, lo, re, im = st.read()
    if case["width"] < 20:
        # register a's wavefunction: the amplitude of each of its values
        a = lo & ((1 << case["width"]) - 1)
        re, im = torch.empty_like(re).scatter_(0, a, re), torch.empty_like(im).scatter_(0, a, im)
        return {"re": re, "im": im, "p": st.out[:1]}
    # (a state this large comes from one launch, in the order of register a)
    got = {"lo": lo, "re": re, "im": im, "p": st.out[:1]}
    if hi is not None:
        got["hi"] = hi
    return got


def _run_arith(case, st):
    st.sv.apply(st.forward, EPS)
    st.sv.apply(st.back, EPS)
    hi, lo, re, im = st.read()
    got = {"lo": lo, "re": re, "im": im}
    if hi is not None:
        got["hi"] = hi
    return got


def _run_measure(case, st):
    st.sv.reset()
    st.sv.apply(st.gates, EPS)
    for k, q in enumerate(st.result):
        st.sv.probability_async(_bit(q), _bit(q), st.slot(k))
    marginals = len(st.result)
    for k, (q, r) in enumerate(st.draws):
        st.sv.measure_async(st.result[q], r, st.slot(marginals + 2 * k))
    got = st.read_sorted(True)
    got["p"] = st.out[:marginals + 2 * len(st.draws)]
    return got


def _run_fill(case, st):
    st.sv.reset()
    st.sv.apply(st.gates, EPS)
    return st.read_sorted(case["qubits"] <= 64)


def _run_sector(case, st):
    st.sv.apply(st.gates, EPS)
    hi, lo, re, im = st.read()
    got = {"lo": lo, "re": re, "im": im}
    if hi is not None and case["qubits"] > 64:
        got["hi"] = hi
    return got


def _run_batch(case, st):
    st.run_graph()
    st.sync()
    lib, got, rows = sps.load_library(), ctypes.c_uint64(0), st.words.shape[2]
    base = [t.data_ptr() for t in (*st.words, *st.amps)]
    for i in range(st.n):
        status = lib.sps_batch_get_amplitudes(st.handle, i, *[p + 8 * rows * i for p in base],
                                              rows, ctypes.byref(got))
        if status != sps.SPS_OK:
            raise sps.SpsError(status, "sps_batch_get_amplitudes")
    return {"labels": st.words, "amplitudes": st.amps}


_RUN = {"mix": _run_mix, "gates": _run_gates, "hop": _run_hop, "adder": _run_adder,
        "arith": _run_arith, "measure": _run_measure, "fill": _run_fill, "sector": _run_sector,
        "batch": _run_batch}


# ---- what a pass cannot do without ------------------------------------------------------
def work(case):
    """Bytes: the entries given (labels 8 or 16 bytes, amplitudes 16) read
    once, the entries returned written once. Operations: FP64 products and sums
    of the branching gates (14 an entry and gate with a complex matrix, 6 with
    a real one) and of one phase an entry (6)."""
    f = case["family"]
    if f == "batch":
        entries = case["circuits"] * (2.0 ** case["log2cap"] - 256) / math.log(
            2.0 ** (case["log2cap"] - 8)) if case["log2cap"] > 8 else case["circuits"] * 256.0
        return {"bytes": 32 * entries, "flops": 12 * entries}
    bits = case.get("qubits") or 2 * case["bits"] + 3
    entry = 24 if bits <= 63 else 32
    if f == "mix":
        n = 2.0 ** case["log2cap"]
        return {"bytes": entry * n, "flops": 18 * n}
    if f == "gates":
        n = 2.0 ** case["qubits"]
        return {"bytes": 16 * n, "flops": 0.3 * case["gates"] * 7 * n}
    if f == "adder":
        n = 2.0 ** case["width"]
        return {"bytes": entry * n, "flops": 6 * n}
    if f == "measure":
        n = 2.0 ** case["width"]
        return {"bytes": entry * n / 2 ** case["measured"], "flops": 3 * n}
    if f == "arith":
        return {"bytes": 2 * entry * case["entries"], "flops": 6 * case["entries"]}
    n = math.comb(case["qubits"], case["modes"])
    differ = 2.0 * case["modes"] * (case["qubits"] - case["modes"]) / (
        case["qubits"] * (case["qubits"] - 1.0))   # a pair of modes differs
    if f == "hop":
        return {"bytes": 2 * entry * n, "flops": case["terms"] * n * (2 * 4 + 6) + 6 * n}
    gates = case["layers"] * (case["qubits"] // 2)
    return {"bytes": (1 if f == "fill" else 2) * entry * n, "flops": 6 * differ * gates * n}


# ---- the same in plain torch, gate by gate in 64 bits --------------------------------------
def _words(mask):
    """A 128-bit mask as two signed 64-bit words (hi, lo)."""
    lo, hi = int(mask) & W._M64, int(mask) >> 64
    return tuple(v - (1 << 64) if v >> 63 else v for v in (hi, lo))


class _Plain:
    """Labels and amplitudes, one gate at a time, with the pruning rule."""

    def __init__(self, hi, lo, amp):
        self.hi, self.lo, self.amp = hi, lo, amp

    @classmethod
    def zero(cls):
        z = torch.zeros(1, dtype=torch.int64, device="cuda")
        return cls(z, z.clone(), torch.ones(1, dtype=torch.complex128, device="cuda"))

    def has(self, mask):
        """Labels with every bit of the mask set."""
        h, l = _words(mask)
        on = None
        if l:
            on = (self.lo & l) == l
        if h:
            on = ((self.hi & h) == h) if on is None else on & ((self.hi & h) == h)
        return torch.ones_like(self.lo, dtype=torch.bool) if on is None else on

    def parity(self, mask):
        """+-1 by the parity of the label's bits under the mask."""
        h, l = _words(mask)
        x = (self.lo & l) ^ (self.hi & h)
        for s in (32, 16, 8, 4, 2, 1):
            x = x ^ (x >> s)
        return (1 - 2 * (x & 1)).to(torch.float64)

    def flip(self, on, mask):
        h, l = _words(mask)
        if l:
            self.lo = torch.where(on, self.lo ^ l, self.lo)
        if h:
            self.hi = torch.where(on, self.hi ^ h, self.hi)

    def scale(self, on, z):
        self.amp = torch.where(on, self.amp * z, self.amp)

    def prune(self):
        a = self.amp
        keep = (a != 0) & (a.real * a.real + a.imag * a.imag >= EPS * EPS)
        self.hi, self.lo, self.amp = self.hi[keep], self.lo[keep], a[keep]

    def pairs(self, active, x, mask, m, to1=1.0, to0=1.0):
        """m = [[m00, m01], [m10, m11]] on the pairs (label with x = 0, that
        label with the mask flipped); to1, to0: further factors of m10 and m01
        for each label that they start from."""
        h, l = _words(mask)
        rest = ~active
        lo, hi, amp, x = self.lo[active], self.hi[active], self.amp[active], x[active]
        lo, hi = torch.where(x, lo ^ l, lo), torch.where(x, hi ^ h, hi)
        order = torch.argsort(lo)
        if bool((hi != hi[:1]).any()):
            order = order[torch.argsort(hi[order], stable=True)]
        lo, hi, amp, x = lo[order], hi[order], amp[order], x[order]
        first = torch.ones_like(x)
        first[1:] = (lo[1:] != lo[:-1]) | (hi[1:] != hi[:-1])
        pair = torch.cumsum(first, 0) - 1
        n = int(first.sum())
        a = torch.zeros(4, n, dtype=torch.complex128, device="cuda")
        f1 = to1[active][order] if isinstance(to1, torch.Tensor) else torch.ones_like(lo)
        f0 = to0[active][order] if isinstance(to0, torch.Tensor) else torch.ones_like(lo)
        a[0, pair[~x]], a[1, pair[x]] = amp[~x], amp[x]
        a[2, pair[~x]], a[3, pair[x]] = (amp * f1)[~x], (amp * f0)[x]
        lo, hi = lo[first], hi[first]
        self.amp = torch.cat([self.amp[rest], m[0][0] * a[0] + m[0][1] * a[3],
                              m[1][0] * a[2] + m[1][1] * a[1]])
        self.lo = torch.cat([self.lo[rest], lo, lo ^ l])
        self.hi = torch.cat([self.hi[rest], hi, hi ^ h])
        self.prune()

    def gate(self, g):
        op, t, th = int(g["op"]), int(g["t0"]), float(g["theta"])
        on = self.has(int(g["cmask"][0]) | int(g["cmask"][1]) << 64)
        c, s = math.cos(th / 2), math.sin(th / 2)
        one = 1 << t
        if op == W.OP_X:
            return self.flip(on, one)
        bit = self.has(one)
        if op == W.OP_GIVENS:
            q = self.has(1 << int(g["t1"]))
            c, s = math.cos(th), math.sin(th)
            return self.pairs(on & (bit != q), bit, one | 1 << int(g["t1"]), [[c, -s], [s, c]])
        if op in (W.OP_H, W.OP_RX, W.OP_RY):
            r = math.sqrt(0.5)
            m = {W.OP_H: [[r, r], [r, -r]], W.OP_RX: [[c, -1j * s], [-1j * s, c]],
                 W.OP_RY: [[c, -s], [s, c]]}[op]
            return self.pairs(on, bit, one, m)
        if op == W.OP_Y:
            self.scale(on & ~bit, 1j)
            self.scale(on & bit, -1j)
            return self.flip(on, one)
        if op == W.OP_RZ:
            self.scale(on & ~bit, complex(c, -s))
            return self.scale(on & bit, complex(c, s))
        r = math.sqrt(0.5)
        z = {W.OP_Z: -1, W.OP_S: 1j, W.OP_SDG: -1j, W.OP_T: complex(r, r),
             W.OP_TDG: complex(r, -r), W.OP_P: complex(math.cos(th), math.sin(th))}[op]
        return self.scale(on & bit, z)

    def pauli(self, x, z, theta):
        """exp(-i theta/2 P), P|j> = i^nY (-1)^|j & z| |j ^ x>."""
        c, s = math.cos(theta / 2), math.sin(theta / 2)
        if not x:
            self.amp = self.amp * (c - 1j * s * self.parity(z))
            return
        ph = -1j * s * 1j ** bin(x & z).count("1")
        sel = self.has(x & -x)
        par = self.parity(z)
        self.pairs(torch.ones_like(sel), sel, x, [[c, ph], [ph, c]], par, par)

    def circuit(self, gates):
        for g in gates:
            self.gate(g)
        return self

    def by_label(self, rows):
        """The amplitudes of a table of that many rows sorted by label, as
        _State.read_sorted lays it out."""
        spare = torch.full((rows - len(self.lo),), -1, dtype=torch.int64, device="cuda")
        hi, lo = torch.cat([self.hi, spare]), torch.cat([self.lo, spare])
        order = torch.argsort(lo)
        order = order[torch.argsort(hi[order], stable=True)]
        return torch.cat([self.amp, torch.zeros_like(spare, dtype=self.amp.dtype)])[order]


def _answer(amp, **more):
    return {"lo": None, "re": amp.real.contiguous(), "im": amp.imag.contiguous(), **more}


def _abs2(a):
    return a.real * a.real + a.imag * a.imag


def exact(case, seed):
    f = case["family"]
    if f == "batch":
        return None   # half a million gates one by one take minutes
    if f == "mix":
        s = _Plain.zero().circuit(_mix_gates(case, seed))
        p = _abs2(s.amp[(s.lo & 3) == 1]).sum().reshape(1)
        return _answer(s.by_label(1 << case["log2cap"]), p=p,
                       **({"hi": None} if case["qubits"] > 63 else {}))
    if f == "gates":
        s = _Plain.zero().circuit(_all_gates(case, seed))
        dense = torch.zeros(1 << case["qubits"], dtype=torch.complex128, device="cuda")
        dense[s.lo] = s.amp
        return torch.stack([dense.real, dense.imag])
    if f == "adder":
        wl, _, _, _ = _adder_parts(case, seed)
        s = _Plain.zero().circuit(wl.gates)
        p = _abs2(s.amp[(s.lo & _adder_readout(case)[0]) == 0]).sum().reshape(1)
        a = s.lo & ((1 << case["width"]) - 1)
        amp = torch.empty_like(s.amp)
        amp[a] = s.amp
        got = _answer(amp, p=p)
        if case["width"] < 20:
            del got["lo"]
        elif wl.layout.nqubits > 63:
            got["hi"] = None
        return got
    if f == "arith":
        wl, _, fwd, back = _adder_parts(case, seed)
        hi, lo = _arith_labels(case, seed)
        re, im = _amplitudes(len(lo), seed)
        s = _Plain(hi, lo, torch.complex(re, im)).circuit(fwd).circuit(back)
        return _answer(s.amp, **({"hi": None} if wl.layout.nqubits > 63 else {}))
    if f == "measure":
        wl, sup, fwd, _ = _adder_parts(case, seed)
        s = _Plain.zero().circuit(np.concatenate([sup, fwd]))
        p = [_abs2(s.amp[s.has(1 << q)]).sum().item() for q in wl.layout.b]
        for k, r in _measure_draws(case, seed):
            on = s.has(1 << wl.layout.b[k])
            p1, p0 = _abs2(s.amp[on]).sum().item(), _abs2(s.amp[~on]).sum().item()
            one = r * (p0 + p1) < p1
            kept = p1 if one else p0
            on = on if one else ~on
            s.hi, s.lo, s.amp = s.hi[on], s.lo[on], s.amp[on] / math.sqrt(kept)
            p += [float(one), kept / (p0 + p1)]
        p = torch.tensor(p, dtype=torch.float64, device="cuda")
        s.hi = torch.full_like(s.hi, -1)   # the result is sorted by the low words
        return _answer(s.by_label(1 << case["width"]), p=p,
                       **({"hi": None} if wl.layout.nqubits > 63 else {}))
    if f == "fill":
        s = _Plain.zero().circuit(np.concatenate(_layers(case, seed)))
        if case["qubits"] <= 64:
            s.hi = torch.full_like(s.hi, -1)   # sorted by the low words
        return _answer(s.by_label(math.comb(case["qubits"], case["modes"]) + 4096),
                       **({"hi": None} if case["qubits"] > 63 else {}))
    hi, lo = _sector_labels(case["qubits"], case["modes"])
    re, im = _amplitudes(len(lo), seed)
    if f == "hop":
        s = _Plain(hi, lo, torch.complex(re, im))
        strings, rz = _hop_terms(case, seed)
        for x, z, theta in strings:
            s.pauli(x, z, theta)
        s.circuit(rz)
        return _answer(s.by_label(2 * len(lo)))
    # sector: labels stay, so a gate's pairs are found by searching for them
    s = _Plain(hi, lo, torch.complex(re, im))
    if case["qubits"] > 64:
        if len(lo) > 2000000:
            return None
        start = torch.argsort(lo)
        start = start[torch.argsort(hi[start], stable=True)]
        s.circuit(_layers(case, seed)[1])
        amp = torch.empty_like(s.amp)
        amp[start] = s.by_label(len(lo))
        return _answer(amp, hi=None)
    order = torch.argsort(lo)
    keys = lo[order]
    for g in _layers(case, seed)[1]:
        if int(g["op"]) != W.OP_GIVENS:
            s.gate(g)
            continue
        one, two = 1 << int(g["t0"]), 1 << int(g["t1"])
        c, sn = math.cos(float(g["theta"])), math.sin(float(g["theta"]))
        i = torch.nonzero(s.has(two) & ~s.has(one))[:, 0]
        j = order[torch.searchsorted(keys, lo[i] ^ _words(one | two)[1])]
        ai, aj = s.amp[i], s.amp[j]
        s.amp[i], s.amp[j] = c * ai - sn * aj, sn * ai + c * aj
    return _answer(s.amp)
