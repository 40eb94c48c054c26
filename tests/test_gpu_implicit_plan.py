"""Gate lists applied without a plan (greedy passes planned inside the call): around
every change of tile width and of op form, against the oracle; per gate where the
timing log is on; and inside a captured CUDA graph."""
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


@pytest.mark.parametrize("n,ng", [(1, 40), (2, 60), (3, 2), (5, 120), (10, 300), (11, 300), (15, 250), (16, 250),
                                  (17, 250), (18, 250), (19, 120), (20, 120), (23, 40), (24, 40)])
def test_without_a_plan(q, orc, n, ng):
    g = w.random_circuit(n, ng, 300 + n, two_qubit_prob=0.4 if n > 1 else None)
    ref = orc.as_complex(orc.run(n, g))
    h = q.qs_alloc(n)
    try:
        q.qs_apply(h, g)
        assert np.max(np.abs(q.qs_get_state(h) - ref)) < TOL
        q.qs_set_zero(h)
        q.qs_timing_enable(h, True)
        q.qs_apply(h, g)
        assert len([r for r in q.qs_timing_fetch(h) if r["kind"] == q._lib.K_TILE]) == 0
        assert np.max(np.abs(q.qs_get_state(h) - ref)) < TOL
    finally:
        q.qs_free(h)
    h = q.qs_alloc_c64(n)
    try:
        q.qs_apply(h, g)
        assert np.linalg.norm(q.qs_get_state(h).astype(np.complex128) - ref) <= 8 * ng * 2.0 ** -24
    finally:
        q.qs_free(h)


@pytest.mark.parametrize("n", [6, 14, 24])
def test_captured(q, n):
    import torch
    g = w.random_circuit(n, 60, 17, two_qubit_prob=0.4)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        h = q.qs_alloc(n, st)
        try:
            q.qs_apply(h, g)
            want = q.qs_get_state(h)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                q.qs_set_zero(h)
                q.qs_apply(h, g)
            for _ in range(2):
                graph.replay()
            st.synchronize()
            assert np.array_equal(q.qs_get_state(h), want)
        finally:
            q.qs_free(h)
