"""Gradients of the largest blocks that are accepted."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_grad_at_the_shared_memory_limit(lib):
    """51 modes, 8 particles, 12 layers: 232,268 of the 232,448 bytes of shared memory a block's
    gradient may take. Against central differences (h = 1e-5: truncation 1e-10, rounding 1e-11,
    of terms of order one)."""
    rng = np.random.default_rng(9)
    n, recs = 51, []

    def bricks():
        for at in (0, 1):
            recs.extend((W.GIVENS, p, p + 1, *rng.uniform(0.2, 1.2, 2)) for p in range(at, n - 1, 2))
    bricks()
    for _ in range(12):
        recs.append((W.CPHASE, 24, 25, 0.4, 0.0))
        bricks()
    occ = list(range(20, 28))
    c = W.Circuit(n, W.modes_to_bits(occ), W.make_gates(recs))
    bits = np.array([W.modes_to_bits([m + d for m in occ]) for d in (0, 1, -2)], dtype=np.uint64)
    with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=lib.EF_PREC_FP64) as h:
        p = lib.ef_prob_exact(h.handle, bits)
        ang = lib.ef_circuit_get_angles(h.handle)
        _, grad = lib.ef_prob_grad(h.handle, bits, 1.0 / p)
        v = rng.normal(size=len(ang))
        v /= np.linalg.norm(v)
        hs, fd = 1e-5, 0.0
        for sign in (1, -1):
            lib.ef_circuit_set_angles(h.handle, ang + sign * hs * v)
            fd += sign * np.sum(np.log(lib.ef_prob_exact(h.handle, bits))) / (2 * hs)
    assert np.linalg.norm(grad) > 1e-3
    assert abs(np.dot(grad, v) - fd) <= 1e-7 * max(1.0, np.linalg.norm(grad))
