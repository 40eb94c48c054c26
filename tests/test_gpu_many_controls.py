"""Gates with more controls than 15, whatever runs them: passes, one kernel per gate (a
plan, the timing log, a single gate, FP64, complex64) and both backward sweeps of the
adjoint gradient, against the oracle."""
import numpy as np
import pytest

import workloads as w
from _tol import grad_close, h1_of

pytestmark = pytest.mark.gpu
TOL = 1e-12
N = 20


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


def ctrl(t, count):
    return sum(1 << b for b in [b for b in range(N) if b != t][-count:])


def program():
    out = [w.gate("RY", a, theta=2.8 + 0.01 * a) for a in range(N)]   # most weight where controls are 1
    for t, c in ((0, 15), (1, 16), (7, 17), (19, 18), (5, 19)):
        out += [w.gate("X", t, ctrl_mask=ctrl(t, c)), w.gate("RY", t, theta=1.1, ctrl_mask=ctrl(t, c)),
                w.gate("P", t, theta=0.7, ctrl_mask=ctrl(t, c)), w.gate("U3", t, theta=0.4, phi=0.9, lam=2.1, ctrl_mask=ctrl(t, c))]
    return w.pack(out)


@pytest.mark.parametrize("how", ["no_plan", "log", "plain", "greedy", "fp64", "single", "c64"])
def test_apply(q, orc, how):
    g = program()
    ref = orc.as_complex(orc.run(N, g))
    h = (q.qs_alloc_c64 if how == "c64" else q.qs_alloc)(N)
    p = q.qs_plan_create(N, g, q.PLAN_GREEDY if how == "greedy" else q.PLAN_PLAIN, 5)
    try:
        if how == "log":
            q.qs_timing_enable(h, True)
        if how == "fp64":
            q.qs_set_arith(h, q.ARITH_FP64)
        if how == "single":
            for k in range(len(g)):
                q.qs_apply(h, g[k:k + 1])
        else:
            q.qs_apply(h, g, None, p if how in ("plain", "greedy", "c64") else None)
        got = q.qs_get_state(h).astype(np.complex128)
    finally:
        q.qs_free(h)
        q.qs_plan_free(p)
    if how == "c64":
        assert np.linalg.norm(got - ref) <= 8 * len(g) * 2.0 ** -24
    else:
        assert np.max(np.abs(got - ref)) < TOL


@pytest.mark.parametrize("fused", [True, False])
def test_gradient(q, orc, fused):
    g = program()
    angled = np.flatnonzero(np.isin(g["type"], [w.GATE_CODES["RY"], w.GATE_CODES["P"]]))
    g["param_idx"][angled] = np.arange(len(angled))
    th, terms = g["p"][angled, 0].copy(), w.tfim(N)
    e0, g0 = orc.adjoint_grad(N, g, th, terms)
    h = q.qs_alloc(N)
    q.qs_set_adjoint_fused(fused)
    try:
        e, grad = q.qs_adjoint_grad(h, g, th, terms)
    finally:
        q.qs_set_adjoint_fused(True)
        q.qs_free(h)
    assert abs(e - e0) < TOL * h1_of(terms)
    assert grad_close(grad, g0, N, len(g), h1_of(terms))
