"""Temporaries of calls that return small results stay with the state: after the first
call, neither small whole distributions nor trajectories whose table covers every qubit
allocate (an armed allocation fault does not fire)."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    yield q
    q.qs_fault_set(q.FAULT_NONE)


@pytest.mark.parametrize("n", [1, 4, 11])
def test_whole_distribution(q, orc, n):
    g = w.random_circuit(n, 40, 3)
    order = [int(v) for v in np.random.default_rng(n).permutation(n)]
    h = q.qs_alloc(n)
    try:
        q.qs_apply(h, g)
        want = q.qs_probs(h, order)
        assert np.max(np.abs(want - orc.marginal(orc.run(n, g), n, order))) < 1e-12
        q.qs_fault_set(q.FAULT_ALLOC, 0, -1)
        assert np.array_equal(q.qs_probs(h, order), want)
        assert q.qs_fault_get()["fired"] == 0
    finally:
        q.qs_fault_set(q.FAULT_NONE)
        q.qs_free(h)


@pytest.mark.parametrize("n", [4, 8, 11])
def test_trajectory(q, orc, n):
    g = w.layered_u3_cz(n, 3, 4)
    rules = w.noise_rules([w.noise_rule("DAMPING", "CZ", 0.02)])
    ref, nd = orc.run_noisy(n, g, rules, seed=4)
    h = q.qs_alloc(n)
    try:
        q.qs_run_noisy(h, g, rules, seed=4)
        q.qs_set_zero(h)
        q.qs_fault_set(q.FAULT_ALLOC, 0, -1)
        assert q.qs_run_noisy(h, g, rules, seed=4) == nd
        assert q.qs_fault_get()["fired"] == 0
        q.qs_fault_set(q.FAULT_NONE)
        assert np.max(np.abs(q.qs_get_state(h) - orc.as_complex(ref))) < 1e-12
    finally:
        q.qs_fault_set(q.FAULT_NONE)
        q.qs_free(h)
