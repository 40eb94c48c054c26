"""Gate lists without a plan round no more amplitudes than a kernel per gate does: X, Y, Z,
S, CNOT, CZ and Toffoli only move, swap and negate components, so a list of them gives the
start's bits back in another order whatever the magnitudes (a Q60 pass would round to
2^-60), and phases or controlled gates leave the amplitudes that they do not multiply as
they are.  Exact comparison, against the oracle and the plan of one kernel per gate."""
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
    return q


def wide_state(n, seed):
    """Components from 1 down to 2^-90, norm 1."""
    rng = np.random.default_rng(seed)
    v = rng.standard_normal(2 << n) * 2.0 ** -rng.integers(0, 90, 2 << n)
    return v / np.linalg.norm(v)


def moves(n, ng, seed, names=("X", "Y", "Z", "S", "CNOT", "CZ")):
    rng = w.SplitMix64(seed)
    out = []
    for _ in range(ng):
        name = names[rng.below(len(names))]
        t = rng.below(n)
        o = (t + 1 + rng.below(n - 1)) % n if n > 1 else t
        if name in w.TWO_QUBIT:
            if n > 1:
                out.append(w.gate(name, o, t, theta=rng.angle()))
            continue
        cm = 1 << o if n > 1 and rng.below(4) == 0 else 0
        out.append(w.gate(name, t, theta=rng.angle(), dagger=rng.below(2), ctrl_mask=cm))
    return w.pack(out)


def run(q, n, g, psi, plan_mode=None):
    h = q.qs_alloc(n)
    p = None if plan_mode is None else q.qs_plan_create(n, g, plan_mode, 1)
    try:
        q.qs_set_state(h, psi)
        q.qs_apply(h, g, None, p)
        return q.qs_get_state(h)
    finally:
        q.qs_free(h)
        if p is not None:
            q.qs_plan_free(p)


@pytest.mark.parametrize("n,ng", [(1, 9), (3, 40), (9, 200), (10, 200), (12, 300), (15, 200), (19, 60), (20, 60), (24, 30)])
def test_unit_factors_move_bits(q, orc, n, ng):
    psi = wide_state(n, n)
    g = moves(n, ng, 70 + n)
    got = run(q, n, g, psi.view(np.complex128))
    assert np.array_equal(got, orc.as_complex(orc.apply_circuit(psi.copy(), n, g)))


@pytest.mark.parametrize("n,ng", [(3, 30), (12, 80), (21, 20)])
def test_amplitudes_outside_the_arithmetic_stay(q, n, ng):
    psi = wide_state(n, 100 + n).view(np.complex128)
    g = np.concatenate([moves(n, ng, 80 + n, ("X", "CNOT", "T", "CR", "P")), w.pack([w.gate("H", 0, ctrl_mask=2)])])
    assert np.array_equal(run(q, n, g, psi), run(q, n, g, psi, q.PLAN_PLAIN))
