"""The timing log brackets every kernel queued for the state, and the launch counter counts
each once: the finishing kernels of Pauli sums and gradients have records, and the record
of a tile pass opens before the pass's phase tables are built."""
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


@pytest.fixture
def logged(q):
    states = []

    def make(n):
        h = q.qs_alloc(n)
        states.append(h)
        q.qs_timing_enable(h, True)
        return h
    yield make
    q.qs_fault_set(q.FAULT_NONE)
    for h in states:
        q.qs_free(h)


@pytest.mark.parametrize("n", [6, 13])
def test_pauli_sum(q, logged, n):
    """One record per kernel: passes, then the finish over their partials."""
    h = logged(n)
    q.qs_expect_pauli(h, w.tfim(n))   # the norm bound is known afterwards
    q.qs_timing_fetch(h)
    before = q.qs_launch_count()
    q.qs_expect_pauli(h, w.tfim(n))
    launched = q.qs_launch_count() - before
    recs = q.qs_timing_fetch(h)
    assert all(r["kind"] == q._lib.K_REDUCE for r in recs)
    assert len(recs) == launched
    assert [r["items"] for r in recs].count(0.0) == 1 and recs[-1]["items"] == 0.0


def test_gradient(q, logged):
    n = 12
    g, npar = w.hea_ansatz(n, 2)
    h = logged(n)
    q.qs_timing_fetch(h)
    before = q.qs_launch_count()
    q.qs_adjoint_grad(h, g, w.uniform_angles(npar, 1), w.tfim(n))
    launched = q.qs_launch_count() - before
    recs = q.qs_timing_fetch(h)
    tables = launched - len(recs)   # one record covers a pass's tables and its tile kernel
    assert 0 <= tables <= sum(r["kind"] == q._lib.K_TILE for r in recs)
    assert any(r["kind"] == q._lib.K_ADJOINT and r["items"] == 0.0 for r in recs)


def test_tables_inside_the_record_of_their_pass(q, logged):
    n = 14
    g = w.layered_u3_cz(n, 6, 2)
    h = logged(n)
    p = q.qs_plan_create(n, g, q.PLAN_GREEDY, 5)
    try:
        q.qs_timing_fetch(h)
        q.qs_fault_set(q.FAULT_LAUNCH, 0, 1)   # the first launch: the first pass's tables
        with pytest.raises(q.QsimError) as ei:
            q.qs_apply(h, g, None, p)
        assert "phase tables" in str(ei.value)
        assert [r["kind"] for r in q.qs_timing_fetch(h)] == [q._lib.K_TILE]
    finally:
        q.qs_plan_free(p)
