"""Backward sweeps whose ops are grouped: pairs of RY (even and odd counts, with and
without gradients, shared parameters) and runs of X and CNOT (controls inside the
tile, outside it, none; chains in both orders), for the single-state gradient and the
batch, against the oracle's adjoint gradient."""
import numpy as np
import pytest

import workloads as w
from _tol import grad_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    assert torch.cuda.is_available()
    import paper_2212_14201_gb300 as q
    q.build()
    return q


def program(n, seed):
    rng = w.SplitMix64(seed)
    out, k = [], 0
    for layer in range(3):
        for a in range(n - (layer == 1)):
            if (a + layer) % 4 == 3:
                out.append(w.gate("RY", a, theta=rng.angle()))
            else:
                out.append(w.gate("RY", a, param_idx=k if (a + layer) % 5 else 0))
                k += 1
        out.append(w.gate("H", layer % n))
        for a in range(n):
            out.append(w.gate("RZ", a, param_idx=k))
            k += 1
        ring = [w.gate("CNOT", (a + 1) % n, a) for a in range(n)] if n > 1 else []
        out += ring if layer % 2 == 0 else ring[::-1]
        out += [w.gate("X", a) for a in range(0, n, 3)]
        if n > 2:
            out += [w.gate("CNOT", 0, n - 1), w.gate("X", n - 1), w.gate("CNOT", n - 1, 1)]
    return w.pack(out), k


@pytest.mark.parametrize("n", [1, 2, 3, 8, 11, 12, 14, 16])
def test_gradients(q, orc, n):
    g, npar = program(n, 900 + n)
    th = w.uniform_angles(npar, n)
    H = w.tfim(n, 0.7) if n > 1 else np.array([(0.7, 1, 0), (0.4, 0, 1)], dtype=w.PAULI_DTYPE)
    e0, g0 = orc.adjoint_grad(n, g, th, H)
    scale = float(np.sum(np.abs(H["coef"])))
    h = q.qs_alloc(n)
    try:
        e, gr = q.qs_adjoint_grad(h, g, th, H)
        end = q.qs_get_state(h)
    finally:
        q.qs_free(h)
    assert abs(e - e0) < 1e-12 * scale
    assert grad_close(gr, g0, n, len(g), scale)
    assert abs(abs(end[0]) - 1.0) < 1e-12  # the state is |0> again, as complex128
    b = q.qs_batch_create([n, n], [g, g], [npar, npar], [H, H])
    try:
        es, gs = np.empty(2), np.empty(2 * npar)
        q.qs_batch_run(b, np.concatenate([th, th]), es, gs)
    finally:
        q.qs_batch_free(b)
    assert np.max(np.abs(es - e0)) < 1e-12 * scale
    assert grad_close(gs[:npar], g0, n, len(g), scale) and np.array_equal(gs[:npar], gs[npar:])
