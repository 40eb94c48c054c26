"""Marginals over four and more qubits (rows of 32 amplitudes, listed high qubits
fixed per warp) against the oracle: no unlisted high qubit, no listed high qubit,
listed qubits on both sides of the row, orders that are not ascending, one row per
warp and many, chunks that split the rows, and complex64 states."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
# sums of non-negative terms adding to 1: each of at most 2^19 additions rounds by 2^-53
TOL = 2.0 ** 19 * 2.0 ** -53


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


@pytest.mark.parametrize("n,qubits", [
    (5, [4, 0, 2, 1]), (6, [5, 0, 3, 1]), (7, [6, 5, 4, 3, 2, 1]), (9, [5, 6, 7, 8]), (9, [0, 1, 2, 3, 4]),
    (13, [12, 0, 7, 3]), (14, list(range(13, 0, -1))), (17, [2, 16, 5, 9, 0, 11, 14]),
    (19, [18, 17, 16, 15, 14, 13, 12, 11, 10, 9, 8, 7]), (19, [3, 8, 13, 18])])
def test_marginal_rows(q, orc, n, qubits):
    st = w.random_state_fast(n, 7 * n + len(qubits))
    st /= np.linalg.norm(st)
    h = q.qs_alloc(n)
    try:
        q.qs_set_state(h, st.view(np.complex128))
        got = q.qs_probs(h, qubits)
    finally:
        q.qs_free(h)
    assert np.max(np.abs(got - orc.marginal(st, n, qubits))) < TOL
    h = q.qs_alloc_c64(n)
    try:
        q.qs_set_state(h, st.view(np.complex128).astype(np.complex64))
        wide = q.qs_get_state(h).astype(np.complex128).view(np.float64)
        got = q.qs_probs(h, qubits)
    finally:
        q.qs_free(h)
    assert np.max(np.abs(got - orc.marginal(wide, n, qubits))) < TOL
