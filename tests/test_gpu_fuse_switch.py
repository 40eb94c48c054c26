"""The fuse switch of programs, trajectories and partial amplitudes: off is one kernel per
gate (launches counted), on is fewer launches; the same results against the oracle."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
N, NG = 11, 160
TOL = 1e-12


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


def launches(q, call):
    before = q.qs_launch_count()
    out = call()
    return out, q.qs_launch_count() - before


def with_state(q, call):
    h = q.qs_alloc(N)
    try:
        r = call(h)
        return r, q.qs_get_state(h)
    finally:
        q.qs_free(h)


@pytest.mark.parametrize("fuse", [False, True])
def test_trajectory(q, orc, fuse):
    g = w.random_circuit(N, NG, 5, two_qubit_prob=0.4)
    rules = w.noise_rules([w.noise_rule("BITFLIP", None, 0.02)])
    ref, draws = orc.run_noisy(N, g, rules, seed=3)
    (nd, psi), count = launches(q, lambda: with_state(q, lambda h: q.qs_run_noisy(h, g, rules, seed=3, fuse=fuse)))
    assert nd == draws and np.max(np.abs(psi - orc.as_complex(ref))) < TOL
    assert count > NG if not fuse else count < NG // 2


@pytest.mark.parametrize("fuse", [False, True])
def test_program(q, orc, fuse):
    prog, g = w.random_program(N, 4)
    ref, cb0, rec0 = orc.run_program(N, prog, g, seed=2)
    ((cb, rec), psi), count = launches(q, lambda: with_state(q, lambda h: q.qs_run_program(h, prog, g, fuse=fuse, seed=2)))
    assert np.array_equal(cb, cb0) and np.max(np.abs(rec - rec0)) < TOL
    assert np.max(np.abs(psi - orc.as_complex(ref))) < TOL
    # its longest run of gates alone
    ng = np.where(prog["op"] == 0, prog["gate_end"] - prog["gate_begin"], 0).astype(int)
    one, first = prog[[int(np.argmax(ng))]].copy(), int(ng.max())
    assert first > 20
    _, per_run = launches(q, lambda: with_state(q, lambda h: q.qs_run_program(h, one, g, fuse=fuse)))
    _, without = launches(q, lambda: with_state(q, lambda h: None))
    assert per_run - without == first if not fuse else per_run - without < first
    assert count > per_run


@pytest.mark.parametrize("fuse", [False, True])
def test_partial_amplitudes(q, orc, fuse):
    lo, hi = (w.random_circuit(N, NG, s, two_qubit_prob=0.4) for s in (6, 7))
    hi["q0"] += N
    hi["q1"] = np.where(hi["q1"] >= 0, hi["q1"] + N, -1)
    g = np.concatenate([lo, hi])   # no gate across the split: one path
    idx = [0, 5, (1 << 2 * N) - 1]
    (amps, paths), count = launches(q, lambda: q.qs_partial_amplitudes(2 * N, g, N, idx, fuse=fuse))
    ref = np.array([orc.as_complex(orc.run(N, lo))[i & ((1 << N) - 1)] * orc.as_complex(orc.run(N, w.random_circuit(
        N, NG, 7, two_qubit_prob=0.4)))[i >> N] for i in idx])
    assert paths == 1 and np.max(np.abs(amps - ref)) < TOL
    identities = int(np.sum(g["type"] == 0))
    assert count >= 2 * NG - identities if not fuse else count < NG
