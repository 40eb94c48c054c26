"""The kernels that run one gate each, through QS_PLAN_PLAIN (a list without a plan runs in
passes): against the oracle with controls, in Q60, FP64 and complex64, and at full size
against the fused passes, amplitude by amplitude.  The log shows that no tile kernel ran."""
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


def apply_plain(q, h, n, g, params=None):
    p = q.qs_plan_create(n, g, q.PLAN_PLAIN, 1)
    q.qs_timing_enable(h, True)
    q.qs_timing_fetch(h)
    try:
        q.qs_apply(h, g, params, p)
        kinds = {r["kind"] for r in q.qs_timing_fetch(h)}
    finally:
        q.qs_timing_enable(h, False)
        q.qs_plan_free(p)
    assert kinds <= {q._lib.K_PHASE1, q._lib.K_DIAG, q._lib.K_ANTI, q._lib.K_REAL, q._lib.K_GENERAL}


def controlled(n, ng, seed):
    """Every gate type with zero to three extra controls."""
    rng = w.SplitMix64(seed)
    out = []
    for k in range(ng):
        name = (w.ONE_QUBIT + ("P",))[rng.below(len(w.ONE_QUBIT) + 1)]
        t = rng.below(n)
        cm = 0
        for _ in range(min(n - 1, k % 4)):
            c = (t + 1 + rng.below(n - 1)) % n
            cm |= 1 << c
        out.append(w.gate(name, t, theta=rng.angle(), phi=rng.angle(), lam=rng.angle(), dagger=rng.below(2), ctrl_mask=cm))
    return w.pack(out)


@pytest.mark.parametrize("kind", ["q60", "fp64", "c64"])
@pytest.mark.parametrize("n,ng", [(1, 20), (2, 40), (5, 120), (9, 200), (14, 150), (20, 60)])
def test_against_oracle(q, orc, n, ng, kind):
    for g in (controlled(n, ng, n), w.random_circuit(n, ng, n, two_qubit_prob=0.4 if n > 1 else None)):
        ref = orc.as_complex(orc.run(n, g))
        h = (q.qs_alloc_c64 if kind == "c64" else q.qs_alloc)(n)
        try:
            if kind != "c64":
                q.qs_set_arith(h, q.ARITH_FIXED if kind == "q60" else q.ARITH_FP64)
            apply_plain(q, h, n, g)
            got = q.qs_get_state(h).astype(np.complex128)
        finally:
            q.qs_free(h)
        if kind == "c64":  # 8 u per op in 2-norm, as for the passes
            assert np.linalg.norm(got - ref) <= 8 * ng * 2.0 ** -24
        else:
            assert np.max(np.abs(got - ref)) < TOL


@pytest.mark.parametrize("n,kind", [(30, "layers"), (32, "random")])
def test_full_size_against_fused(q, n, kind):
    """The benchmark's brickwork at n = 30 and random gates at n = 32: every amplitude
    within 1e-12 of the greedy plan's (whose n = 30 state is checked against the oracle)."""
    import torch
    g = w.layered_u3_cz(n, 20, 1) if kind == "layers" else w.random_circuit(n, 300, 2, two_qubit_prob=0.4)
    greedy = q.qs_plan_create(n, g, q.PLAN_GREEDY, 5)
    h = q.qs_alloc(n, torch.cuda.current_stream())
    fused = plain = None
    try:
        q.qs_set_arith(h, q.ARITH_FIXED)
        q.qs_apply(h, g, None, greedy)
        fused = torch.empty(2 << n, dtype=torch.float64, device="cuda")
        q.qs_get_state(h, fused)
        q.qs_set_zero(h)
        apply_plain(q, h, n, g)
        assert abs(q.qs_probs(h, [])[0] - 1.0) < TOL
        plain = torch.empty(2 << n, dtype=torch.float64, device="cuda")
        q.qs_get_state(h, plain)
        worst = max(float((a - b).abs().max()) for a, b in zip(fused.split(1 << 28), plain.split(1 << 28)))
        assert worst < TOL / 2 ** 0.5   # per component
    finally:
        q.qs_free(h)
        q.qs_plan_free(greedy)
        del fused, plain
        torch.cuda.empty_cache()
