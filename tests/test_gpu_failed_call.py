"""A call of several kernels that fails part way (host-side fault injection: the check
after a launch reports an error, the kernel itself was queued) leaves amplitudes, not the
Q60 integers that tile passes keep between them: whichever check fails, the buffer is a
normalised complex128 state, because every kernel queued before it is unitary."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
N = 14


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    yield q
    q.qs_fault_set(q.FAULT_NONE)


def calls(q):
    brick = w.layered_u3_cz(N, 6, 2)
    hea, npar = w.hea_ansatz(N, 2)
    theta = w.uniform_angles(npar, 3)

    def greedy(h):
        p = q.qs_plan_create(N, brick, q.PLAN_GREEDY, 5)
        try:
            q.qs_apply(h, brick, None, p)
        finally:
            q.qs_plan_free(p)
    return {"plan": greedy, "no_plan": lambda h: q.qs_apply(h, brick),
            "gradient": lambda h: q.qs_adjoint_grad(h, hea, theta, w.tfim(N))}


@pytest.mark.parametrize("name", ["plan", "no_plan", "gradient"])
def test_amplitudes_after_a_failed_call(q, name):
    call = calls(q)[name]
    h = q.qs_alloc(N)
    try:
        failed = 0
        for after in range(200):
            q.qs_set_zero(h)
            q.qs_fault_set(q.FAULT_LAUNCH, after, 1)
            try:
                call(h)
            except q.QsimError as e:
                assert e.code == -3, str(e)
            fired = q.qs_fault_get()["fired"]
            q.qs_fault_set(q.FAULT_NONE)
            psi = q.qs_get_state(h)
            assert np.all(np.isfinite(psi.view(np.float64))), after
            # 70 to 120 ops at 2^-60 sqrt(2^15) each, and 2^-53 per conversion: far below
            assert abs(float(np.vdot(psi, psi).real) - 1.0) < 1e-12, after
            assert abs(q.qs_probs(h, [])[0] - 1.0) < 1e-12, after
            if not fired:
                break
            failed += 1
        assert 3 <= failed < 200
    finally:
        q.qs_fault_set(q.FAULT_NONE)
        q.qs_free(h)
