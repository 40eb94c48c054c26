"""What a user of this simulator runs, as cases that can be timed and compared.

Kinds:
  gates     a gate list applied from |0...0> without a plan (one kernel per gate)
  fused     the same through a greedy fusion plan the program keeps; complex128 or
            complex64; random circuits or U3 + CZ brickwork layers
  readout   <Z_i> of every qubit, the marginal of a few qubits and the squared norm
  energy    the expectation of the transverse-field Ising Hamiltonian
  sample    measurement shots of a state
  gradient  energy and gradient of a hardware-efficient ansatz (torch.autograd)
  batch     energies and gradients of many ansatz instances of mixed sizes
  noisy     one noise trajectory: depolarizing on every gate, damping on every CZ
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2212_14201_gb300 as q
from paper_2212_14201_gb300.autograd import Expectation

H, X, Y, Z, S, T, RX, RY, RZ, U3, CNOT, CZ, CR = 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 13, 14
ONE = (H, X, Y, Z, S, T, RX, RY, RZ, U3)
TWO = (CNOT, CZ, CR)
ANGLED = (RX, RY, RZ, U3, CR)
DEPOLARIZING, DAMPING = 3, 0


def listed():
    return [
        # the smallest program: a 12-qubit circuit of 200 gates, all launch latency
        {"name": "gates_n12", "kind": "gates", "program": "random", "n": 12, "gates": 200},
        # a large state without a plan: two layers of the brickwork, a sweep per gate
        {"name": "gates_n26", "kind": "gates", "program": "layers", "n": 26, "depth": 2},
        # an everyday circuit: 20 qubits, as in the published library comparisons
        {"name": "random_n20", "kind": "fused", "program": "random", "n": 20, "gates": 300, "bits": 128},
        # the same kind of circuit on a state larger than the caches
        {"name": "random_n27", "kind": "fused", "program": "random", "n": 27, "gates": 400, "bits": 128},
        # the benchmark's own circuit at full size
        {"name": "layers_n30", "kind": "fused", "program": "layers", "n": 30, "depth": 20, "bits": 128},
        # single precision, for users who trade accuracy for speed
        {"name": "layers_c64_n28", "kind": "fused", "program": "layers", "n": 28, "depth": 16, "bits": 64},
        # reading a state out: all <Z_i>, a register of 7 qubits, the norm
        {"name": "readout_n26", "kind": "readout", "n": 26, "qubits": 7},
        # the energy of a 25-site chain
        {"name": "energy_n25", "kind": "energy", "n": 25},
        # a million shots
        {"name": "sample_n26", "kind": "sample", "n": 26, "shots": 1000000},
        # one optimiser step's energy and gradient of a 22-qubit ansatz
        {"name": "gradient_n22", "kind": "gradient", "n": 22, "layers": 4},
        # a sweep over parameter sets and chain lengths
        {"name": "batch_128", "kind": "batch", "sets": 128, "lo": 10, "hi": 18, "layers": 8},
        # a noise trajectory of a brickwork circuit
        {"name": "noisy_n22", "kind": "noisy", "n": 22, "depth": 6},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("gates", "fused", "fused", "fused", "readout", "energy", "sample", "gradient", "batch", "noisy"))
    if kind == "gates":
        if rng.random() < 0.5:
            return {"kind": kind, "program": "random", "n": rng.randint(5, 24), "gates": _log(rng, 20, 600)}
        return {"kind": kind, "program": "layers", "n": rng.randint(8, 27), "depth": rng.randint(1, 4)}
    if kind == "fused":
        bits = rng.choice((128, 128, 64))
        if rng.random() < 0.5:
            return {"kind": kind, "program": "random", "n": rng.randint(10, 28), "gates": _log(rng, 50, 500), "bits": bits}
        return {"kind": kind, "program": "layers", "n": rng.randint(10, 28), "depth": rng.randint(2, 20), "bits": bits}
    if kind == "readout":
        n = rng.randint(8, 28)
        return {"kind": kind, "n": n, "qubits": rng.randint(1, min(n - 1, 12))}
    if kind == "energy":
        return {"kind": kind, "n": rng.randint(6, 27)}
    if kind == "sample":
        return {"kind": kind, "n": rng.randint(6, 28), "shots": _log(rng, 100, 1000000)}
    if kind == "gradient":
        return {"kind": kind, "n": rng.randint(6, 24), "layers": rng.randint(1, 6)}
    if kind == "batch":
        lo = rng.randint(6, 12)
        return {"kind": kind, "sets": _log(rng, 4, 160), "lo": lo, "hi": lo + rng.randint(2, 6), "layers": rng.randint(2, 8)}
    return {"kind": kind, "n": rng.randint(10, 23), "depth": rng.randint(2, 8)}


# ---- inputs ---------------------------------------------------------------------------

def _pack(records):
    """(type, q0, q1, angles, parameter) tuples as the library's gate records."""
    g = np.zeros(len(records), dtype=q.GATE_DTYPE)
    for k, (t, a, b, p, idx) in enumerate(records):
        g[k]["type"], g[k]["q0"], g[k]["q1"], g[k]["p"], g[k]["param_idx"] = t, a, b, p, idx
    return g


def _random_gates(n, count, rs):
    """Random circuit: 40 % two-qubit gates, the rest one-qubit gates of every type."""
    out = []
    for _ in range(count):
        t = int(rs.choice(TWO)) if rs.random_sample() < 0.4 else int(rs.choice(ONE))
        a, b = (int(v) for v in rs.choice(n, 2, replace=False))
        p = tuple(rs.uniform(0, 2 * np.pi, 3)) if t in ANGLED else (0.0, 0.0, 0.0)
        if t != U3:
            p = (p[0], 0.0, 0.0)
        out.append((t, a, b if t in TWO else -1, p, -1))
    return out


def _layers(n, depth, rs):
    """U3 on every qubit, then CZ on alternating neighbour pairs, `depth` times."""
    out = []
    for d in range(depth):
        out += [(U3, a, -1, tuple(rs.uniform(0, 2 * np.pi, 3)), -1) for a in range(n)]
        out += [(CZ, a, a + 1, (0.0, 0.0, 0.0), -1) for a in range(d % 2, n - 1, 2)]
    return out


def _ansatz(n, layers):
    """RY and RZ on every qubit, then a CNOT ring, `layers` times; one parameter a rotation."""
    out, k = [], 0
    for _ in range(layers):
        for t in (RY, RZ):
            for a in range(n):
                out.append((t, a, -1, (0.0, 0.0, 0.0), k))
                k += 1
        out += [(CNOT, (a + 1) % n, a, (0.0, 0.0, 0.0), -1) for a in range(n)]
    return out, k


def _ising(n, field=0.7):
    """Open transverse-field Ising chain: (coefficient, X mask, Z mask)."""
    zz = [(1.0, 0, 3 << a) for a in range(n - 1)]
    return zz + [(field, 1 << a, 0) for a in range(n)]


def _records(case, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    if case.get("program") == "random":
        return _random_gates(case["n"], case["gates"], rs)
    return _layers(case["n"], case["depth"], rs)


def _state(n, seed):
    """A normalised random state (what a deep circuit leaves), as interleaved re, im."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(2 << n, dtype=torch.float64, device="cuda", generator=g)
    return v.mul_(1.0 / torch.linalg.vector_norm(v).item())


def _sizes(case):
    span = case["hi"] - case["lo"] + 1
    return [case["lo"] + (7 * k) % span for k in range(case["sets"])]


def _angles(count, seed):
    return np.random.RandomState(seed % (1 << 31)).uniform(0, 2 * np.pi, count)


def _list(case, seed):
    """The register that is read out."""
    return [int(v) for v in np.random.RandomState(seed % (1 << 31)).permutation(case["n"])[:case["qubits"]]]


class _Kept:
    """Library handles a program keeps, given back when it drops them."""

    def __init__(self):
        self._free = []

    def keep(self, handle, free):
        self._free.append((handle, free))
        return handle

    def __del__(self):
        for handle, free in reversed(self._free):
            free(handle)


def prepare(case, seed):
    s = _Kept()
    s.kind = kind = case["kind"]
    n = case.get("n")
    if kind in ("gates", "fused"):
        s.gates, s.plan = _pack(_records(case, seed)), None
        s.bits = case.get("bits", 128)
        if kind == "fused":
            s.plan = s.keep(q.qs_plan_create(n, s.gates, q.PLAN_GREEDY), q.qs_plan_free)
        if s.bits == 64:
            s.handle = s.keep(q.qs_alloc_c64(n, torch.cuda.current_stream()), q.qs_free)
            s.out = torch.empty(2 << n, dtype=torch.float32, device="cuda")
        else:
            s.sv = q.StateVector(n)
    elif kind in ("readout", "energy", "sample"):
        s.sv = q.StateVector(n)
        s.sv.set_state(_state(n, seed))
        if kind == "readout":
            s.qubits = _list(case, seed)
        elif kind == "energy":
            s.terms = np.array(_ising(n), dtype=q.PAULI_DTYPE)
        else:
            s.seed, s.shots = seed, case["shots"]
    elif kind == "gradient":
        records, count = _ansatz(n, case["layers"])
        s.energy = Expectation(n, _pack(records), np.array(_ising(n), dtype=q.PAULI_DTYPE))
        s.params = torch.from_numpy(_angles(count, seed)).requires_grad_(True)
    elif kind == "batch":
        sizes = _sizes(case)
        programs = {m: _ansatz(m, case["layers"]) for m in set(sizes)}
        packed = {m: _pack(r) for m, (r, _) in programs.items()}
        terms = {m: np.array(_ising(m), dtype=q.PAULI_DTYPE) for m in programs}
        counts = [programs[m][1] for m in sizes]
        s.batch = s.keep(q.qs_batch_create(sizes, [packed[m] for m in sizes], counts, [terms[m] for m in sizes]),
                         q.qs_batch_free)
        s.params = _angles(sum(counts), seed)
        s.energies, s.grads = np.empty(len(sizes)), np.empty(sum(counts))
    else:
        s.sv = q.StateVector(n)
        s.gates, s.seed = _pack(_records(case, seed)), seed
        s.rules = np.array([(DEPOLARIZING, -1, -1, -1, 0.01, 0, 0, 0), (DAMPING, CZ, -1, -1, 0.02, 0, 0, 0)],
                           dtype=q.NOISE_DTYPE)
    return s


def run(s):
    if s.kind in ("gates", "fused"):
        if s.bits == 64:
            q.qs_set_zero(s.handle)
            q.qs_apply(s.handle, s.gates, None, s.plan)
            return q.qs_get_state(s.handle, s.out)
        q.qs_set_zero(s.sv.handle)
        s.sv.apply(s.gates, None, s.plan)
        return s.sv.amps
    if s.kind == "readout":
        return {"z": s.sv.expect_z(), "p": s.sv.probs(s.qubits), "norm": s.sv.probs([])}
    if s.kind == "energy":
        return s.sv.expect(s.terms)
    if s.kind == "sample":
        return s.sv.sample(s.seed, s.shots).view(np.int64)
    if s.kind == "gradient":
        s.params.grad = None
        e = s.energy(s.params)
        e.backward()
        return {"energy": e.detach(), "grad": s.params.grad}
    if s.kind == "batch":
        q.qs_batch_run(s.batch, s.params, s.energies, s.grads)
        return {"energies": s.energies, "grads": s.grads}
    q.qs_set_zero(s.sv.handle)
    draws = q.qs_run_noisy(s.sv.handle, s.gates, s.rules, seed=s.seed)
    return {"amps": s.sv.amps, "draws": draws}


def _flops(records, n):
    """Real operations of a gate list on 2^n amplitudes, each gate as its own kind."""
    per = {H: 4, RX: 6, RY: 6, U3: 14, RZ: 6, T: 3, CR: 1.5}
    return sum(per.get(r[0], 0) for r in records) * float(1 << n)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        by, fl = 0.0, 0.0
        for m in _sizes(case):
            records, count = _ansatz(m, case["layers"])
            by += 16.0 * count + 8
            fl += 4.0 * _flops(records, m)
        return {"bytes": by, "flops": fl}
    n = case["n"]
    N = float(1 << n)
    if kind in ("gates", "fused", "noisy"):
        return {"bytes": (8.0 if case.get("bits") == 64 else 16.0) * N, "flops": _flops(_records(case, 0), n)}
    if kind == "readout":
        return {"bytes": 16.0 * N, "flops": 4.0 * N + n * N}
    if kind == "energy":
        return {"bytes": 16.0 * N, "flops": 6.0 * n * N}
    if kind == "sample":
        return {"bytes": 16.0 * N + 8.0 * case["shots"], "flops": 4.0 * N}
    records, count = _ansatz(n, case["layers"])
    return {"bytes": 16.0 * count + 8, "flops": 4.0 * _flops(records, n)}


# ---- the same results from plain torch in 64 bits -----------------------------------------

def _matrix(t, p):
    th, ph, lam = p
    c, s = math.cos(th / 2), math.sin(th / 2)
    e = lambda a: complex(math.cos(a), math.sin(a))  # noqa: E731
    r = math.sqrt(0.5)
    return {H: (r, r, r, -r), X: (0, 1, 1, 0), Y: (0, -1j, 1j, 0), Z: (1, 0, 0, -1), S: (1, 0, 0, 1j),
            T: (1, 0, 0, complex(r, r)), RX: (c, -1j * s, -1j * s, c), RY: (c, -s, s, c),
            RZ: (e(-th / 2), 0, 0, e(th / 2)), U3: (c, -e(lam) * s, e(ph) * s, e(ph + lam) * c),
            CNOT: (0, 1, 1, 0), CZ: (1, 0, 0, -1), CR: (1, 0, 0, e(th))}[t]


def _gate(psi, n, m, t, c=None):
    """The 2x2 matrix m on qubit t of psi (..., 2^n), where qubit c (if any) is 1; in place."""
    v = psi.view(-1, 2, 1 << t)
    if c is not None:
        hi, lo = max(t, c), min(t, c)
        v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        v = v.select(1 if c == hi else 3, 1).movedim(1 if t == hi else 2, 1)
    a, b = v[:, 0], v[:, 1]
    if m[1] == 0 and m[2] == 0:
        if m[0] != 1:
            a.mul_(m[0])
        if m[3] != 1:
            b.mul_(m[3])
        return
    new = a * m[0] + b * m[1] if m[0] != 0 else b * m[1]
    if m[3] != 0:
        b.mul_(m[3]).add_(a, alpha=m[2])
    else:
        b.copy_(a).mul_(m[2])
    a.copy_(new)


def _program(records, n):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    for t, a, b, p, _ in records:
        _gate(psi, n, _matrix(t, p), b if t in TWO else a, a if t in TWO else None)
    return psi


def _flip(psi, n, t):
    """X on qubit t of psi (S, 2^n)."""
    return psi.view(psi.shape[0], -1, 2, 1 << t).flip(2).reshape(psi.shape)


def _ising_times(psi, n):
    x = torch.arange(1 << n, device="cuda")
    zz = torch.full((1 << n,), float(n - 1), dtype=torch.float64, device="cuda")
    for a in range(n - 1):
        zz -= 2.0 * ((x >> a ^ x >> a + 1) & 1)
    out = psi * zz
    for a in range(n):
        out += 0.7 * _flip(psi, n, a)
    return out


def _energy_and_gradient(n, layers, params):
    """Energies and gradients of the ansatz for params (S, P), by the adjoint recursion."""
    records, count = _ansatz(n, layers)
    S = params.shape[0]
    p = torch.from_numpy(params).cuda()
    psi = torch.zeros(S, 1 << n, dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1

    def rotate(v, t, a, th):
        w = v.view(S, -1, 2, 1 << a)
        x, y = w[:, :, 0], w[:, :, 1]
        c, s = torch.cos(th / 2).view(-1, 1, 1), torch.sin(th / 2).view(-1, 1, 1)
        if t == RY:
            return torch.stack((c * x - s * y, s * x + c * y), 2).view(S, -1)
        return torch.stack((torch.complex(c, -s) * x, torch.complex(c, s) * y), 2).view(S, -1)

    def cnot(v, c, a):
        hi, lo = max(a, c), min(a, c)
        w = v.view(S, -1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        i, j = (2, 3) if c == hi else (4, 2)
        one = w.select(i, 1)
        one.copy_(one.flip(j))
        return v

    for t, a, b, _, k in records:
        psi = cnot(psi, a, b) if t == CNOT else rotate(psi, t, a, p[:, k])
    lam = _ising_times(psi, n)
    energy = (psi.conj() * lam).sum(1).real
    grad = torch.empty(S, count, dtype=torch.float64, device="cuda")
    for t, a, b, _, k in reversed(records):
        if t == CNOT:
            psi, lam = cnot(psi, a, b), cnot(lam, a, b)
            continue
        u, v = psi.view(S, -1, 2, 1 << a), lam.view(S, -1, 2, 1 << a)
        if t == RY:
            grad[:, k] = (v[:, :, 1].conj() * u[:, :, 0] - v[:, :, 0].conj() * u[:, :, 1]).sum((1, 2)).real
        else:
            grad[:, k] = (v[:, :, 0].conj() * u[:, :, 0] - v[:, :, 1].conj() * u[:, :, 1]).sum((1, 2)).imag
        psi, lam = rotate(psi, t, a, -p[:, k]), rotate(lam, t, a, -p[:, k])
    return energy.cpu().numpy(), grad.cpu().numpy()


def _uniform(seed, k):
    """Draw k of a trajectory: SplitMix64 in counter form, mapped to [0, 1)."""
    mask = (1 << 64) - 1
    z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return ((z ^ (z >> 31)) >> 11) * 2.0 ** -53


def _trajectory(records, n, seed, p=0.01, gamma=0.02):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    k = 0

    def pick(w):
        nonlocal k
        u, c = _uniform(seed, k) * sum(w), 0.0
        k += 1
        for j, x in enumerate(w):
            c += x
            if u < c:
                return j
        return len(w) - 1

    for t, a, b, ang, _ in records:
        _gate(psi, n, _matrix(t, ang), b if t in TWO else a, a if t in TWO else None)
        touched = sorted((a, b)) if t in TWO else [a]
        for x in touched:
            j = pick([1 - 0.75 * p] + [p / 4] * 3)
            if j:
                _gate(psi, n, _matrix((X, Y, Z)[j - 1], (0, 0, 0)), x)
        for x in touched if t == CZ else ():
            v = torch.view_as_real(psi).view(-1, 2, 2 << x).square().sum((0, 2)).tolist()
            w = [v[0] + (1 - gamma) * v[1], gamma * v[1]]
            j = pick(w)
            f = 1 / math.sqrt(w[j])
            _gate(psi, n, ((f, 0, 0, f * math.sqrt(1 - gamma)), (0, f * math.sqrt(gamma), 0, 0))[j], x)
    return psi, k


def _real(psi):
    return torch.view_as_real(psi).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("gates", "fused"):
        records = _records(case, seed)
        if len(records) << case["n"] > 800 << 28:  # half a minute and more
            return None
        return _real(_program(records, case["n"]))
    if kind in ("readout", "energy"):
        n = case["n"]
        psi = torch.view_as_complex(_state(n, seed).view(-1, 2))
        if kind == "energy":
            v = psi.view(1, -1)
            return float((v.conj() * _ising_times(v, n)).sum().real)
        pr = _real(psi).view(-1, 2).square().sum(1)
        z = [float(pr.view(-1, 2, 1 << a).sum((0, 2)).diff()) for a in range(n)]
        qubits = _list(case, seed)
        m = pr
        for a in sorted(set(range(n)) - set(qubits), reverse=True):
            m = m.view(-1, 2, 1 << a).sum(1)
        kept = sorted(qubits, reverse=True)
        m = m.view((2,) * len(qubits)).permute([kept.index(a) for a in reversed(qubits)]).reshape(-1)
        return {"z": -np.array(z), "p": m.cpu().numpy(), "norm": np.array([float(pr.sum())])}
    if kind == "gradient":
        count = _ansatz(case["n"], case["layers"])[1]
        e, g = _energy_and_gradient(case["n"], case["layers"], _angles(count, seed)[None])
        return {"energy": torch.tensor(e[0]), "grad": torch.from_numpy(g[0])}
    if kind == "batch":
        sizes = _sizes(case)
        counts = [2 * m * case["layers"] for m in sizes]
        angles = np.split(_angles(sum(counts), seed), np.cumsum(counts)[:-1])
        energies, grads = np.empty(len(sizes)), [None] * len(sizes)
        for m in set(sizes):
            at = [k for k, x in enumerate(sizes) if x == m]
            e, g = _energy_and_gradient(m, case["layers"], np.stack([angles[k] for k in at]))
            for i, k in enumerate(at):
                energies[k], grads[k] = e[i], g[i]
        return {"energies": energies, "grads": np.concatenate(grads)}
    if kind == "noisy":
        psi, draws = _trajectory(_records(case, seed), case["n"], seed)
        return {"amps": _real(psi), "draws": draws}
    return None
