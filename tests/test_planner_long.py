"""Planning long programs on the host: the greedy passes are those of a scan over all
remaining gates, and the time grows with the number of gates, not with its square."""
import time

import numpy as np
import pytest

import workloads as w

DIAG = {w.GATE_CODES[k] for k in ("I", "Z", "S", "T", "RZ", "P", "CZ", "CR")}
TWO = {w.GATE_CODES[k] for k in ("CNOT", "CZ", "CR")}
MAX_GATES = 224  # of a pass
SCAN = 2048      # gates a scan leaves before it ends


@pytest.fixture(scope="module")
def q():
    import paper_2212_14201_gb300 as q
    q.build()
    return q


def full_scans(n, gates, m, scan=None):
    """Execution order of the greedy passes, each a scan of the whole remaining list, or
    of its gates up to `scan` left ones."""
    info = []
    for r in gates:
        two, diag = int(r["type"]) in TWO, int(r["type"]) in DIAG
        t = 1 << int(r["q1"] if two else r["q0"])
        c = int(r["ctrl_mask"]) | (1 << int(r["q0"]) if two else 0)
        info.append((0 if diag else t, (t if diag else 0) | c))
    remaining, order = list(range(len(gates))), []
    while remaining:
        Q, bn, bd, took, rest = (1 << min(n, 3)) - 1, 0, 0, 0, []
        for at, k in enumerate(remaining):
            if scan is not None and len(rest) >= scan:
                rest += remaining[at:]
                break
            N, D = info[k]
            no = bool(N & (bn | bd)) or bool(D & bn) or took >= MAX_GATES
            if not no and N & ~Q:
                if bin(Q).count("1") < m:
                    Q |= N
                else:
                    no = True
            if no:
                rest.append(k)
                bn, bd = bn | N, bd | D
            else:
                order.append(k)
                took += 1
        remaining = rest
    return order


def sparse(n, ng, seed):
    """CNOTs from one control into the others, T on it now and then, and a qubit that only
    the last gate uses: the scan's blocked set never covers all qubits."""
    rng = w.SplitMix64(seed)
    out = []
    for k in range(ng - 1):
        t = rng.below(n - 2)
        out.append(w.gate("T", n - 2) if k % 97 == 0 else w.gate("CNOT", n - 2, t) if k % 3 else w.gate("H", t))
    return w.pack(out + [w.gate("H", n - 1)])


def idle(n, ng, seed):
    """Random gates on n - 1 qubits, and one gate on the last qubit at the very end."""
    return np.concatenate([w.random_circuit(n - 1, ng - 1, seed, two_qubit_prob=0.4), w.pack([w.gate("Z", n - 1)])])


PROGRAMS = {"random": lambda n, ng, seed: w.random_circuit(n, ng, seed, two_qubit_prob=0.4), "sparse": sparse, "idle": idle}


def order_of(q, n, g, m):
    p = q.qs_plan_create_variant(n, g, m, 0)
    try:
        return np.concatenate([idx for _, _, idx in q.qs_plan_passes(p)]).tolist()
    finally:
        q.qs_plan_free(p)


@pytest.mark.parametrize("n,ng,m", [(4, 700, 4), (13, 900, 12), (20, 1500, 12), (20, 1500, 5), (34, 1500, 13)])
@pytest.mark.parametrize("kind", list(PROGRAMS))
def test_passes_are_those_of_full_scans(q, n, ng, m, kind):
    g = PROGRAMS[kind](n, ng, 3 + n)
    assert order_of(q, n, g, m) == full_scans(n, g, m)


def test_scans_end_after_enough_gates_left(q):
    g = idle(20, 6000, 1)
    got = order_of(q, 20, g, 12)
    assert got == full_scans(20, g, 12, SCAN)
    assert got != full_scans(20, g, 12)   # the last gate is too far for the first pass


@pytest.mark.parametrize("kind", list(PROGRAMS))
def test_time_is_linear_in_the_gates(q, kind):
    n, sizes = 20, (10000, 100000)
    t = []
    for ng in sizes:
        g = PROGRAMS[kind](n, ng, 5)
        best = 1e9
        for _ in range(3):
            t0 = time.perf_counter()
            p = q.qs_plan_create(n, g, q.PLAN_GREEDY, 5)
            best = min(best, time.perf_counter() - t0)
            q.qs_plan_free(p)
        t.append(best)
    # ten times the gates: 10 when linear, 100 when every pass scans what is left
    assert t[1] < 30 * t[0], t
