"""Which qubits a table of joint populations covers (the reduction records of the timing
log: k is the number of qubits read): one where every rotation moves the populations of
its own qubit before its channel, many where a layer of diagonal gates follows; results
against the oracle."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
TOL = 1e-12
N = 13


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


def layers(entangler):
    rng = w.SplitMix64(8)
    out = []
    for d in range(3):
        out += [w.gate("RY", k, theta=rng.angle()) for k in range(N)]
        if entangler:
            out += [w.gate(entangler, k, k + 1) for k in range(d % 2, N - 1, 2)]
    return w.pack(out)


def widths(q, orc, gates, rules):
    ref, nd = orc.run_noisy(N, gates, rules, seed=5)
    h = q.qs_alloc(N)
    try:
        q.qs_timing_enable(h, True)
        assert q.qs_run_noisy(h, gates, rules, seed=5) == nd
        out = [r["k"] for r in q.qs_timing_fetch(h) if r["kind"] == q._lib.K_REDUCE]
        assert np.max(np.abs(q.qs_get_state(h) - orc.as_complex(ref))) < TOL
    finally:
        q.qs_free(h)
    return out


def test_rotations_read_their_own_qubit(q, orc):
    rules = w.noise_rules([w.noise_rule("DECOHERENCE", "RY", t1=30.0, t2=20.0, tgate=1.0)])
    got = widths(q, orc, layers(None), rules)
    assert len(got) == 3 * N and set(got) == {1}


@pytest.mark.parametrize("entangler", ["CZ", "CNOT"])
def test_layers_of_entanglers_share_a_table(q, orc, entangler):
    rules = w.noise_rules([w.noise_rule("DAMPING", entangler, 1e-4)])
    got = widths(q, orc, layers(entangler), rules)
    per_layer = N - 1   # qubits that the entanglers of a layer touch
    if entangler == "CZ":
        # eleven qubits, then the twelfth with the other qubit of its gate
        assert sorted(got) == [2] * 3 + [11] * 3
    else:
        # a CNOT moves its target after the table of the gate before was read
        assert max(got) > 1 and len(got) <= 3 * per_layer


def test_large_states_read_seven_qubits(q, orc):
    """From 20 qubits on a narrow table is read with other qubits and folded."""
    n = 20
    g = w.pack([w.gate("RY", k, theta=0.3 + 0.1 * k) for k in range(n)] + [w.gate("CZ", 0, 1), w.gate("H", 1)])
    rules = w.noise_rules([w.noise_rule("DAMPING", "RY", 0.05), w.noise_rule("PHASE_DAMPING", "CZ", 0.05)])
    ref, nd = orc.run_noisy(n, g, rules, seed=6)
    h = q.qs_alloc(n)
    try:
        q.qs_timing_enable(h, True)
        assert q.qs_run_noisy(h, g, rules, seed=6) == nd
        got = [r["k"] for r in q.qs_timing_fetch(h) if r["kind"] == q._lib.K_REDUCE]
        assert len(got) >= n and set(got) == {7}
        assert np.max(np.abs(q.qs_get_state(h) - orc.as_complex(ref))) < TOL
    finally:
        q.qs_free(h)
