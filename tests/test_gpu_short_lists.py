"""The shortest lists without a plan: one kernel per gate where a pass would take longer,
passes from one gate more on (launches counted at the edges of the rule), and the same
results against the oracle either way."""
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


def gates(n, ng, diag):
    out = []
    for k in range(ng):
        t = n - 1 - k
        out.append(w.gate("RZ", t, theta=0.4 + k) if diag else w.gate("RY", t, theta=0.4 + k))
    return w.pack(out)


# bits, qubits, diagonal, fewest gates that run as a pass (0: no list this short is one)
EDGES = [(128, 6, False, 3), (128, 17, False, 3), (128, 18, False, 4), (128, 23, False, 4), (128, 24, False, 2),
         (128, 17, True, 3), (128, 18, True, 4), (128, 24, True, 3),
         (64, 6, False, 3), (64, 23, False, 3), (64, 24, False, 2),
         (64, 11, True, 3), (64, 12, True, 4), (64, 23, True, 4), (64, 24, True, 3), (64, 25, True, 2)]


@pytest.mark.parametrize("bits,n,diag,fewest", EDGES)
def test_edges_of_the_rule(q, orc, bits, n, diag, fewest):
    h = (q.qs_alloc if bits == 128 else q.qs_alloc_c64)(n)
    try:
        for ng in (fewest - 1, fewest):
            g = gates(n, ng, diag)
            q.qs_set_zero(h)
            before = q.qs_launch_count()
            q.qs_apply(h, g)
            count = q.qs_launch_count() - before
            # a pass: its kernel, and one more where it has a phase table
            assert count == ng if ng < fewest else count in (1, 2)
            got = q.qs_get_state(h).astype(np.complex128)
            err = np.max(np.abs(got - orc.as_complex(orc.run(n, g))))
            assert err < (1e-12 if bits == 128 else 8 * ng * 2.0 ** -24)
    finally:
        q.qs_free(h)
