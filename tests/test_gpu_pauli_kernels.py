"""Pauli sums on states of 12 qubits and more, where field terms and |a|^2 terms have
kernels of their own: chains, more |a|^2 terms than a launch holds, X masks that are
not single basis coordinates, terms with Y and Z beside them, against the oracle."""
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


def mixed(n):
    full = (1 << n) - 1
    rows = [(0.02 * (k + 1), 0, (k * 7919 + 3) & full) for k in range(27)]
    rows += [(0.1, 1 << b, 0) for b in (0, 3, 4, min(11, n - 2), n - 1)]
    rows += [(0.05, (1 << b) | (1 << (n - 2)), 0) for b in (1, 5)]
    rows += [(0.2, 1 << 6, 1 << 6), (0.2, 1 << 6, 1 << 2), (-0.3, 0b11, 0b11), (0.04, full, 0)]
    return np.array(rows, dtype=w.PAULI_DTYPE)


@pytest.mark.parametrize("n", [11, 12, 13, 15, 16, 17, 20])
@pytest.mark.parametrize("kind", ["tfim", "mixed", "random"])
def test_expectation(q, orc, n, kind):
    terms = {"tfim": lambda: w.tfim(n, 0.7), "mixed": lambda: mixed(n), "random": lambda: w.random_paulis(n, 30, n)}[kind]()
    st = w.random_state_fast(n, 11 + n)
    st /= np.linalg.norm(st)
    scale = max(1.0, float(np.sum(np.abs(terms["coef"]))))
    h = q.qs_alloc(n)
    try:
        q.qs_set_state(h, st.view(np.complex128))
        assert abs(q.qs_expect_pauli(h, terms) - orc.expect_pauli(st, n, terms)) < TOL * scale
    finally:
        q.qs_free(h)
    h = q.qs_alloc_c64(n)
    try:
        q.qs_set_state(h, st.view(np.complex128).astype(np.complex64))
        wide = q.qs_get_state(h).astype(np.complex128).view(np.float64)
        assert abs(q.qs_expect_pauli(h, terms) - orc.expect_pauli(wide, n, terms)) < TOL * scale
    finally:
        q.qs_free(h)


@pytest.mark.parametrize("x", [0, 5, (1 << 17) - 1])
def test_basis_state(q, x):
    """A basis state: +-coef for every Z term, exactly; 0 for every X term."""
    n = 17
    st = np.zeros(1 << n, dtype=np.complex128)
    st[x] = 1.0
    h = q.qs_alloc(n)
    try:
        q.qs_set_state(h, st)
        for zm in (0, 1, 0b110, 1 << 9, (1 << 16) | 1, (1 << n) - 1):
            one = np.array([(1.0, 0, zm)], dtype=w.PAULI_DTYPE)
            assert q.qs_expect_pauli(h, one) == (-1.0) ** bin(x & zm).count("1")
        for b in (0, 4, 12, 16):
            assert q.qs_expect_pauli(h, np.array([(1.0, 1 << b, 0)], dtype=w.PAULI_DTYPE)) == 0.0
    finally:
        q.qs_free(h)
