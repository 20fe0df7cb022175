"""Raw Estimate calls of several slabs, and the corner cases of the sampling.

A call of 10^9 Philox blocks or more runs in several slabs on two streams. Its
results are those of smaller calls (same trajectories by the global index; FP64
within rounding of the sums), the same when repeated, and the same bit for bit
from a batch's captured graph. A circuit without particles has no minors: every
trajectory's term is its weight alone."""
import numpy as np
import pytest

import workloads as W
from oracle.philox import trajectory_uniforms

pytestmark = pytest.mark.gpu


def _big(lib, prec):
    c = W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=3, angle_sampler=W.normal_var(0.1), seed=7)
    bits = W.spin_sector_bitstrings(6, 3, 3, 1300, np.random.default_rng(4))
    return c, bits, 300_000, lib.Circuit(c.n_modes, c.occupation, c.gates, precision=prec)


@pytest.mark.parametrize("prec", ["fp64", "auto"])
def test_slabs_match_smaller_calls(lib, prec):
    c, bits, t, h = _big(lib, lib.EF_PREC_FP64 if prec == "fp64" else lib.EF_PREC_AUTO)
    with h:
        p, se = lib.ef_prob_approx(h.handle, bits, t, seed=9)
        assert np.array_equal(lib.ef_prob_approx(h.handle, bits, t, seed=9)[0], p)
        for lo, hi in ((0, 40), (600, 640), (1290, 1300)):
            q, sq = lib.ef_prob_approx(h.handle, bits[lo:hi], t, seed=9, index_base=lo)
            assert np.allclose(p[lo:hi], q, rtol=1e-11 if prec == "fp64" else 2e-5, atol=1e-18)
            assert np.allclose(se[lo:hi], sq, rtol=1e-9 if prec == "fp64" else 1e-3, atol=1e-18)


def test_slabs_in_a_batch_graph(lib):
    torch = pytest.importorskip("torch")
    c, bits, t, h = _big(lib, lib.EF_PREC_AUTO)
    with h, lib.Circuit(c.n_modes, c.occupation, c.gates) as other:
        ref = lib.ef_prob_approx(h.handle, bits, t, seed=9, want_stderr=False)
        ref2 = lib.ef_prob_exact(other.handle, bits)
        d = torch.from_numpy(bits.view(np.int64)).cuda()
        out = [torch.zeros(len(bits), dtype=torch.float64, device="cuda") for _ in range(2)]
        b = lib.ef_batch_create([h.handle, other.handle])
        try:
            for _ in range(3):  # the planning call, then two replays
                for o in out:
                    o.zero_()
                lib.ef_batch_prob_dev(b, [d.data_ptr()] * 2, [len(bits)] * 2, [o.data_ptr() for o in out], [t, 0], seed=9,
                                      stream=torch.cuda.current_stream().cuda_stream)
                torch.cuda.synchronize()
                assert np.array_equal(out[0].cpu().numpy(), ref) and np.array_equal(out[1].cpu().numpy(), ref2)
        finally:
            lib.ef_batch_destroy(b)


@pytest.mark.parametrize("prec,nb,t", [("fp64", 1900, 100_000), ("auto", 1900, 100_000), ("auto", 1825, 250_001)])
def test_long_items_are_cut(lib, prec, nb, t):
    # large angles: most trajectories flip several gates, so one bitstring's samples pass 1 MB and its item is
    # cut; the small calls split their few bitstrings finely instead. The trajectories are the same, the sums are
    # grouped differently: FP64 within 10^5 roundings of the extent (100), FP32 within twice tol
    c = W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=3, angle_sampler=W.normal_var(1.0), seed=11)
    bits = W.spin_sector_bitstrings(6, 3, 3, nb, np.random.default_rng(5))
    with lib.Circuit(c.n_modes, c.occupation, c.gates,
                     precision=lib.EF_PREC_FP64 if prec == "fp64" else lib.EF_PREC_AUTO) as h:
        p, se = lib.ef_prob_approx(h.handle, bits, t, seed=3)
        assert np.array_equal(lib.ef_prob_approx(h.handle, bits, t, seed=3)[0], p)
        for lo, hi in ((0, 30), (nb - 7, nb)):
            q, sq = lib.ef_prob_approx(h.handle, bits[lo:hi], t, seed=3, index_base=lo)
            assert np.allclose(p[lo:hi], q, rtol=1e-9 if prec == "fp64" else 2e-5, atol=1e-9 if prec == "fp64" else 1e-12)
            assert np.allclose(se[lo:hi], sq, rtol=1e-6 if prec == "fp64" else 1e-3, atol=1e-9)


def test_no_particles(lib):
    recs = [(W.GIVENS, 0, 1, 0.3, 0.1), (W.CPHASE, 0, 2, 0.9, 0.0), (W.CPHASE, 1, 3, -1.2, 0.0), (W.GIVENS, 2, 3, 0.7, 0.2)]
    c = W.Circuit(4, np.zeros(2, dtype=np.uint64), W.make_gates(recs))
    bits = np.zeros((2, 2), dtype=np.uint64)
    theta = np.array([0.9, -1.2])
    sa, ca = np.sin(np.abs(theta) / 4), np.cos(theta / 4)
    p1 = np.floor(sa / (sa + ca) * 2.0 ** 32 + 0.5) / 2.0 ** 32
    p_ref = []
    for i in range(2):
        x = trajectory_uniforms(3, i, np.arange(900), 2) < (p1 * 2.0 ** 32).astype(np.uint64)
        y = np.prod(np.where(x, 1j * np.sin(theta / 4) / p1, ca / (1 - p1)), axis=1)
        p_ref.append(abs(y.mean()) ** 2)
    for prec, tol in ((lib.EF_PREC_FP64, 1e-10), (lib.EF_PREC_AUTO, 1e-5)):
        with lib.Circuit(4, c.occupation, c.gates, precision=prec) as h:
            p = lib.ef_prob_approx(h.handle, bits, 900, seed=3, want_stderr=False)
        assert np.max(np.abs(p - p_ref)) <= tol * np.max(p_ref)
