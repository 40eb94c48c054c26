"""Trajectories whose channels need populations, on more qubits than one table of
joint populations holds (11), with jumps frequent enough to end many tables early:
layers of rotations and entanglers with damping, decoherence and Pauli noise, against
the oracle (draw count exactly, amplitudes 1e-12)."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


def layers(n, entangler, depth, seed):
    rng = w.SplitMix64(seed)
    out = []
    for d in range(depth):
        out += [w.gate("RY", k, theta=rng.angle()) for k in range(n)]
        out += [w.gate(entangler, k, k + 1) for k in range(d % 2, n - 1, 2)]
        out += [w.gate("T", k) for k in range(0, n, 3)]
    return w.pack(out)


@pytest.mark.parametrize("n,entangler,p", [(2, "CZ", 0.3), (11, "CZ", 0.02), (12, "CZ", 0.3), (13, "CNOT", 0.1),
                                           (15, "CZ", 0.05)])
def test_joint_populations(q, orc, n, entangler, p):
    rules = w.noise_rules([
        w.noise_rule("DAMPING", entangler, p), w.noise_rule("PHASE_DAMPING", "T", p),
        w.noise_rule("DECOHERENCE", "RY", t1=30.0, t2=20.0, tgate=1.0), w.noise_rule("DEPOLARIZING", entangler, 0.05)])
    g = layers(n, entangler, 3, 50 + n)
    for seed in range(3):
        st, nd = orc.run_noisy(n, g, rules, seed=seed)
        h = q.qs_alloc(n)
        try:
            got_nd = q.qs_run_noisy(h, g, rules, seed=seed)
            got = q.qs_get_state(h)
        finally:
            q.qs_free(h)
        assert got_nd == nd
        assert np.max(np.abs(got - orc.as_complex(st))) < TOL
