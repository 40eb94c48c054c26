"""Pending diagonal operators of a trajectory on complex64 states: the factors are pairs of
floats, so an operator costs one rounding of each component, and a long run of damping
channels stays within one such rounding per operator and gate of the double oracle."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


@pytest.mark.parametrize("n,channels", [(1, "each"), (2, "each"), (9, "each"), (12, "layer"), (13, "layer"), (18, "each")])
def test_complex64_operators(q, orc, n, channels):
    """each: a damping after every rotation (operators one at a time); layer: after the
    T gates of a layer (up to eleven together).  8 u per gate as for plain circuits, 2 u
    per operator."""
    rng = w.SplitMix64(n)
    out = []
    for _ in range(2):
        out += [w.gate("RY", k, theta=rng.angle()) for k in range(n)] + [w.gate("T", k) for k in range(n)]
    g = w.pack(out)
    rule = w.noise_rule("DAMPING", "RY" if channels == "each" else "T", 0.003)
    rules = w.noise_rules([rule])
    ref, nd = orc.run_noisy(n, g, rules, seed=2)
    h = q.qs_alloc_c64(n)
    try:
        assert q.qs_run_noisy(h, g, rules, seed=2) == nd
        got = q.qs_get_state(h).astype(np.complex128)
    finally:
        q.qs_free(h)
    assert np.linalg.norm(got - orc.as_complex(ref)) <= (8 * len(g) + 2 * nd) * U32
