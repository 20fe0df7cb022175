"""Exact probabilities of sets in which bitstrings of a mode block repeat.

From 1024 bitstrings on, equal bitstrings of a block are factored once. The
probability of a bitstring depends neither on the set it is asked for in nor
on its place there, bit for bit: sets without the search (below 1024) are the
reference. Sets: products of few alpha and beta strings, the whole sector
repeated, uniform draws, bitstrings outside the sector among them."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CIRCUITS = {
    "lucj-12q": lambda: W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=3, angle_sampler=W.normal_var(0.1), seed=7),
    "lucj-32q": lambda: W.lucj32_exact(1)[0],
    "lucj-16q-uneven": lambda: W.lucj_circuit(8, 3, 2, 2, n_onsite=3, n_same=2, angle_sampler=W.normal_var(0.4), seed=12),
    "lucj-72q": lambda: W.lucj_circuit(36, 4, 4, 1, n_onsite=5, n_same=2, angle_sampler=W.normal_var(0.3), seed=3),
}


@pytest.mark.parametrize("name", list(CIRCUITS))
@pytest.mark.parametrize("prec", ["fp64", "fp32", "auto"])
def test_repeated_block_strings(lib, name, prec):
    c = CIRCUITS[name]()
    norb, na, nb = c.meta["norb"], c.meta["n_alpha"], c.meta["n_beta"]
    rng = np.random.default_rng(5)
    draw = W.spin_sector_bitstrings(norb, na, nb, 900, rng)
    draw[7] = W.modes_to_bits(range(na + nb))  # outside the sector
    draw[8] = 0
    # alpha words of 30 rows with beta words of 40 others (a block's modes may cross the word boundary)
    mask = W.modes_to_bits(range(norb))
    prod = np.array([(draw[i] & mask) | (draw[50 + j] & ~mask) for i in range(30) for j in range(40)], dtype=np.uint64)
    big = np.concatenate([draw, prod, draw[::-1][:333], draw[:1].repeat(70, axis=0)])
    big = big[rng.permutation(len(big))]
    precision = {"fp64": lib.EF_PREC_FP64, "fp32": lib.EF_PREC_FP32_MINOR, "auto": lib.EF_PREC_AUTO}[prec]
    with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=precision, tol=1e-6) as h:
        p, err = lib.ef_prob_exact(h.handle, big, want_err=True)
        st = lib.ef_circuit_get_stats(h.handle)
        parts = [lib.ef_prob_exact(h.handle, big[i:i + 1000], want_err=True) for i in range(0, len(big), 1000)]
        ref = [np.concatenate([x[k] for x in parts]) for k in range(2)]
        small = lib.ef_prob_exact(h.handle, big[:1000]) is not None and lib.ef_circuit_get_stats(h.handle)
    assert len(big) > 1024 and np.count_nonzero(p) > len(p) // 2
    assert np.array_equal(p, ref[0]) and np.array_equal(err, ref[1])
    if prec != "auto":  # fewer minors than bitstrings x patterns
        assert st["executed_minor_lus"] * 1000 < small["executed_minor_lus"] * len(big)
    assert st["fp64_recomputed"] == np.count_nonzero(err < 0)
