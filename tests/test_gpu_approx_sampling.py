"""Raw Estimate: the sampled trajectories at the sizes where their storage changes.

Numbers of gates around the four gates of a Philox block, the pair of blocks
and the 32 gates of a sampling step, and above 256 (wider gate numbers);
angles from a flip in a hundred trajectories to dozens of flips in each (more
than an entry holds); trajectories around a row of 128, a segment of 4096 and
beyond. FP64 against the oracle on the same trajectories within 1e-10 (the
tolerance of the FP64 path), EF_PREC_AUTO within 1e-5, the flips counted
exactly."""
import math

import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(1, 0.3, 1), (3, 1.0, 127), (4, 0.02, 4097), (5, 1.2, 129), (8, 1.2, 700), (31, 0.3, 600), (33, 0.8, 500),
         (64, 0.1, 4100), (152, 0.05, 8300), (257, 0.02, 4200), (300, 1.0, 260)]


@pytest.mark.parametrize("k,std,t", SIZES, ids=[f"k{k}-std{s}-t{t}" for k, s, t in SIZES])
def test_sampled_trajectories_match_oracle(lib, k, std, t):
    c = W.random_fig4_circuit(10, 4, k, 2, seed=100 + k, angle_std=std)
    bits = W.sector_bitstrings_all(10, 4)
    passive = W.Circuit(c.n_modes, c.occupation, c.gates[c.gates["kind"] != W.CPHASE])
    bits = bits[np.argsort(-O.exact_probabilities(passive, bits))[:3]]  # the no-flip minors' largest
    seed = 0x5EED_0000_0001 + k
    p_ref, se_ref, _, flips_ref = O.raw_estimate(c, bits, t=t, seed=seed, return_details=True)
    floor = 1e-6 / math.comb(10, 4)
    for prec, tol in ((lib.EF_PREC_FP64, 1e-10), (lib.EF_PREC_AUTO, 1e-5)):
        with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=prec) as h:
            p, se = lib.ef_prob_approx(h.handle, bits, t, seed=seed)
            assert lib.ef_circuit_get_stats(h.handle)["sampled_flips"] == flips_ref
        assert np.max(np.abs(p - p_ref) / np.maximum(p_ref, floor)) <= tol
        assert np.max(np.abs(se - se_ref) / np.maximum(se_ref, floor)) <= (1e-8 if tol < 1e-9 else 1e-3)
