"""Short Pauli sums of mixed kinds: a few |a|^2 and field terms share the launch of the
terms that need a tile (launches counted in the log, at the edges of the rule), with the
same values as apart; against the oracle."""
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


def terms(n, nz, nx, other):
    """nz Z terms (nz + 1 sums with the total), nx X terms, and Y X on two qubits."""
    t = [(0.3 + k, 0, 1 << k) for k in range(nz)] + [(0.7 - 0.1 * k, 1 << (n - 1 - k), 0) for k in range(nx)]
    if other:
        t.append((-0.4, 3 << (n // 2), 1 << (n // 2)))
    return np.array(t, dtype=w.PAULI_DTYPE)


# n, Z terms, X terms, the other term, launches without the finish
EDGES = [(11, 1, 1, True, 1), (12, 1, 1, True, 1), (14, 2, 3, True, 1), (14, 3, 6, True, 1), (18, 8, 1, True, 1),
         (14, 1, 0, True, 1), (14, 0, 3, True, 1), (14, 0, 0, True, 1), (14, 1, 1, False, 2),
         (20, 7, 1, True, 1), (20, 8, 1, True, 2), (20, 1, 5, True, 1), (20, 1, 6, True, 2), (20, 8, 6, True, 3),
         (26, 1, 1, False, 1), (26, 1, 2, False, 2), (26, 2, 1, False, 2), (26, 1, 1, True, 1)]


@pytest.mark.parametrize("bits", [128, 64])
@pytest.mark.parametrize("n,nz,nx,other,launches", EDGES)
def test_launches_and_values(q, orc, bits, n, nz, nx, other, launches):
    g = w.layered_u3_cz(n, 2, 5)
    t = terms(n, nz, nx, other)
    h = (q.qs_alloc if bits == 128 else q.qs_alloc_c64)(n)
    try:
        q.qs_apply(h, g)
        q.qs_expect_pauli(h, t)   # the norm bound is known afterwards
        q.qs_timing_enable(h, True)
        got = q.qs_expect_pauli(h, t)
        recs = q.qs_timing_fetch(h)
        assert len(recs) == launches + 1
        one_by_one = sum(float(c["coef"]) * q.qs_expect_pauli(h, np.array([(1.0, c["xmask"], c["zmask"])], dtype=w.PAULI_DTYPE))
                         for c in t)
        # exact sums, each rounded to double; coefficients below 3.5
        assert abs(got - one_by_one) < 3.5 * len(t) * 2.0 ** -50
        if n <= 20:
            st = q.qs_get_state(h).astype(np.complex128).view(np.float64)
            assert abs(got - orc.expect_pauli(st, n, t)) < 1e-12
    finally:
        q.qs_free(h)
