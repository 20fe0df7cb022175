"""When equal bitstrings of a mode block are looked for: from 1024 bitstrings and 2^17 minors on.

Few flip patterns leave little to spare, so small sets of such circuits are factored as they are; large
sets search with a grid of the search's own size, whatever the number of patterns."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("onsite,same,nb,searched", [(1, 1, 2000, False), (1, 1, 16_000, False), (1, 1, 20_000, True),
                                                     (1, 1, 300_001, True), (4, 1, 4000, False), (4, 1, 4200, True),
                                                     (8, 4, 1023, False), (8, 4, 1024, True)])
def test_search_by_the_minors_it_can_spare(lib, onsite, same, nb, searched):
    c = W.lucj_circuit(16, 8, 8, 1, n_onsite=onsite, n_same=same, angle_sampler=W.normal_var(0.1), seed=7)
    rng = np.random.default_rng(3)
    base = W.spin_sector_bitstrings(16, 8, 8, 60, rng)
    alpha, beta = base[:, 0] & np.uint64(0xffff), base[:, 0] & np.uint64(0xffff0000)
    i, j = rng.integers(0, 40, nb), rng.integers(0, 60, nb)
    i[:60], j[:60] = np.arange(60) % 40, np.arange(60)  # every string occurs
    bits = np.stack([alpha[i] | beta[j], np.zeros(nb, dtype=np.uint64)], axis=1)
    with lib.Circuit(c.n_modes, c.occupation, c.gates, precision=lib.EF_PREC_FP32_MINOR) as h:
        some = lib.ef_prob_exact(h.handle, bits[-700:])
        minors = lib.ef_circuit_get_stats(h.handle)["executed_minor_lus"] // 700  # of a bitstring, both blocks
        p = lib.ef_prob_exact(h.handle, bits)
        done = lib.ef_circuit_get_stats(h.handle)["executed_minor_lus"]
    assert np.array_equal(p[-700:], some)
    distinct = [len(np.unique(x)) for x in (alpha[:40], beta)]
    assert done == (sum(distinct) * minors // 2 if searched else nb * minors)


def test_search_tables_count_in_a_slice(lib):
    """Two patterns a block: a bitstring's tables weigh as much as its determinants, and both
    stay within the 2 GiB of a slice (14 million bitstrings in one slice took 2.8 GiB)."""
    torch = pytest.importorskip("torch")
    c = W.lucj_circuit(16, 8, 8, 1, n_onsite=1, n_same=0, angle_sampler=W.normal_var(0.1), seed=7)
    base = W.spin_sector_bitstrings(16, 8, 8, 500, np.random.default_rng(3))
    nb = 14_000_000
    d = torch.from_numpy(base.view(np.int64)).cuda().repeat(nb // 500, 1).contiguous()
    out = torch.zeros(nb, dtype=torch.float64, device="cuda")
    with lib.Circuit(c.n_modes, c.occupation, c.gates) as h:
        ref = lib.ef_prob_exact(h.handle, base)  # tables and kernels are there
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lib.ef_prob_exact_dev(h.handle, d.data_ptr(), nb, out.data_ptr(), 0, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        used = free - torch.cuda.mem_get_info()[0]
    assert used <= (2 << 30) + (64 << 20)
    assert torch.equal(out.view(-1, 500), torch.from_numpy(ref).cuda().expand(nb // 500, 500))
