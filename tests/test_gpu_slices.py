"""Calls that run in several slices or slabs of their workspace.

Exact sets beyond 2 GiB of determinants run slice by slice, each with its own
search for equal bitstrings; a Raw Estimate whose one bitstring has more samples
than a slab splits the bitstring's chunks over slabs on two streams. Results are
those of smaller calls."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nb,slices", [("auto", 300_000, 3), ("fp32", 1_000_000, 3)])
def test_exact_slices_search_for_equal_bitstrings(lib, prec, nb, slices):
    c = W.lucj32_exact(1)[0]
    rng = np.random.default_rng(21)
    base = W.spin_sector_bitstrings(16, 8, 8, 900, rng)
    base[3] = 0  # outside the sector
    pick = rng.integers(0, len(base), nb)
    precision = lib.EF_PREC_AUTO if prec == "auto" else lib.EF_PREC_FP32_MINOR
    with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=precision, tol=1e-6) as h:
        ref, ref_err = lib.ef_prob_exact(h.handle, base, want_err=True)  # too few for the search
        p, err = lib.ef_prob_exact(h.handle, base[pick], want_err=True)
        st = lib.ef_circuit_get_stats(h.handle)
    assert np.array_equal(p, ref[pick]) and np.array_equal(err, ref_err[pick])
    if prec == "auto":
        flagged = np.count_nonzero(err < 0)
        assert 0 < flagged < nb and st["fp64_recomputed"] == flagged
    else:  # every slice factors its distinct halves once (each draws nearly all 900 of them)
        halves = sum(len(np.unique(base[:, 0] >> np.uint64(s) & np.uint64(0xffff))) for s in (0, 16))
        assert (slices - 1) * 256 * halves < st["executed_minor_lus"] <= slices * 256 * halves


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_one_bitstring_over_several_slabs(lib, prec):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # large angles: nearly every trajectory has an entry, 18 bytes each; a call with one bitstring has
    # 12 chunks per SM of just over three segments (4096 trajectories), so four segments' room: 290 KB x 12 x 152
    # pass 512 MiB, which the same trajectories cut at three segments do not
    c = W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=5, angle_sampler=lambda rng, n: rng.uniform(1.2, 2.0, n), seed=11)
    bits = W.spin_sector_bitstrings(6, 3, 3, 4, np.random.default_rng(5))
    t = 12 * sms * 12416
    with lib.Circuit(c.n_modes, c.occupation, c.gates,
                     precision=lib.EF_PREC_FP64 if prec == "fp64" else lib.EF_PREC_FP32_MINOR) as h:
        p1, s1 = lib.ef_prob_approx(h.handle, bits[:1], t, seed=3)
        launches = lib.ef_circuit_get_stats(h.handle)["kernel_launches"]
        p4, s4 = lib.ef_prob_approx(h.handle, bits, t, seed=3)
        again = lib.ef_prob_approx(h.handle, bits[:1], t, seed=3)
    assert launches > (4 if prec == "fp64" else 5)  # more than one slab
    assert again[0][0] == p1[0] and again[1][0] == s1[0]
    # the same trajectories in other groups: FP64 within 10^7 roundings of the terms, FP32 within its estimates
    assert np.allclose(p1, p4[:1], rtol=1e-8 if prec == "fp64" else 2e-5, atol=1e-12)
    assert np.allclose(s1, s4[:1], rtol=1e-6 if prec == "fp64" else 1e-3, atol=1e-12)
