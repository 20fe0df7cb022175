"""Flagged results whose error budget is not a number.

A tol so small that tol max(p, floor) underflows in FP32, with a probability that
is exactly zero although its minors carry an error estimate: the budget of the
error terms left is 0 / 0. Such results are redone like any other flagged one and
take nothing from what an earlier call left in the workspace."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _circuit():
    """Two spins of 9 modes, 4 particles each. Modes 0-3: two particles, rows 2 and 3 both
    (1/2, 1/2), so that every minor with both rows is exactly zero while its pivots are not.
    Modes 4-8: two particles, all controlled phases, hence the flip patterns."""
    rng = np.random.default_rng(3)
    m, recs = 9, []
    for at in (0, m):
        recs += [(W.GIVENS, at, at + 1, math.pi / 4, 0.0), (W.GIVENS, at + 1, at + 2, math.pi / 2, 0.0),
                 (W.GIVENS, at + 2, at + 3, math.pi / 4, 0.0), (W.GIVENS, at + 3, at + 4, 0.0, 0.0)]
    def mix():
        for at in (0, m):
            for p in (5, 4, 6, 7, 5, 4, 6):
                recs.append((W.GIVENS, at + p, at + p + 1, *rng.uniform(0.3, 1.2, 2)))
    mix()
    for p in range(4, 8):
        recs += [(W.CPHASE, p, p + 1, 0.6, 0.0), (W.CPHASE, m + p, m + p + 1, 0.6, 0.0)]
    recs += [(W.CPHASE, p, m + p, 0.5, 0.0) for p in range(4, 9)]
    mix()
    occ = [0, 1, 4, 5]
    return W.Circuit(2 * m, W.modes_to_bits(occ + [m + p for p in occ]), W.make_gates(recs))


@pytest.mark.parametrize("nb", [700, 2600])  # without and with the search for equal bitstrings
def test_zero_probabilities_with_a_tiny_tol(lib, nb):
    c = _circuit()
    rng = np.random.default_rng(8)

    def spin(low):
        hi = rng.choice(np.arange(4, 9), 2, replace=False)
        return list(low) + [int(x) for x in hi]

    def strings(low):
        return np.array([W.modes_to_bits(spin(low) + [9 + x for x in spin((0, 2))]) for _ in range(nb)], dtype=np.uint64)

    some, none = strings((0, 3)), strings((2, 3))
    with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=lib.EF_PREC_FP64) as h:
        ref = lib.ef_prob_exact(h.handle, some)
    with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=lib.EF_PREC_AUTO, tol=1e-60) as h:
        p = lib.ef_prob_exact(h.handle, some)
        q, err = lib.ef_prob_exact(h.handle, none, want_err=True)
    assert np.count_nonzero(ref > 1e-6) > nb // 2 and np.all(err < 0)  # flagged: there was an estimate
    assert np.allclose(p, ref, rtol=1e-9, atol=1e-15)
    # zero to FP64 rounding of an amplitude of order one
    assert np.max(np.abs(q)) <= 1e-28
