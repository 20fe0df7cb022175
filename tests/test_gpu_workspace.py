"""Device memory of Raw Estimate calls: with the calls in flight, not with the circuits that exist."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def _circuit(seed):
    return W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=3, angle_sampler=W.normal_var(1.0), seed=seed)


def _bits(nb):
    return W.spin_sector_bitstrings(6, 3, 3, nb, np.random.default_rng(2))


PROGRAM = """
import sys
import numpy as np, torch
import paper_2511_12416_gb300 as ef, workloads as W
nb, t, n = 2000, 25000, 12  # samples of a call: over two slabs of 512 MiB
bits = W.spin_sector_bitstrings(6, 3, 3, nb, np.random.default_rng(2))
torch.zeros(1, device="cuda")
def circuits():
    cs = [W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=3, angle_sampler=W.normal_var(1.0), seed=i) for i in range(n)]
    return [ef.Circuit(c.n_modes, c.occupation, c.gates) for c in cs]
def used():
    torch.cuda.synchronize()
    return (start - torch.cuda.mem_get_info()[0]) / 2**30
with circuits()[0] as c:  # modules and tables that stay
    ef.ef_prob_approx(c.handle, bits[:4], 1000, seed=1)
d = torch.from_numpy(bits.view(np.int64)).cuda()
outs = [torch.zeros(nb, dtype=torch.float64, device="cuda") for _ in range(n)]
torch.cuda.synchronize()
start = torch.cuda.mem_get_info()[0]
hs = circuits()
for h in hs:
    ef.ef_prob_approx(h.handle, bits, t, seed=1)
print("calls", used())
b = ef.ef_batch_create([h.handle for h in hs])
ef.ef_batch_prob_dev(b, [d.data_ptr()] * n, [nb] * n, [o.data_ptr() for o in outs], [t] * n, seed=1,
                     stream=torch.cuda.current_stream().cuda_stream)
print("batch", used())
torch.cuda.synchronize()
ef.ef_batch_destroy(b)
for h in hs:
    h.close()
print("none", used())
"""


def test_memory_of_many_circuits(lib):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, env=dict(os.environ, PYTHONPATH=root), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    gib = {k: float(v) for k, v in (line.split() for line in r.stdout.splitlines())}
    # 12 circuits of 1 GiB a call: what the pool keeps, what a batch's four streams hold besides, what stays
    assert gib["calls"] <= 2.25 and gib["batch"] <= 2.25 + 4.25 and gib["none"] <= 0.25


def test_calls_on_streams_and_threads(lib):
    torch = pytest.importorskip("torch")
    nb, t = 600, 30_000
    bits = _bits(nb)
    d = torch.from_numpy(bits.view(np.int64)).cuda()
    hs = [lib.Circuit(c.n_modes, c.occupation, c.gates) for c in (_circuit(1), _circuit(2), _circuit(3))]
    ref = [lib.ef_prob_approx(h.handle, bits, t + 1000 * i, seed=4, want_stderr=False) for i, h in enumerate(hs)]
    bad = []

    def work(i):
        torch.cuda.set_device(0)
        s = torch.cuda.Stream()
        out = torch.zeros(nb, dtype=torch.float64, device="cuda")
        s.wait_stream(torch.cuda.default_stream())
        for _ in range(15):
            lib.ef_prob_approx_dev(hs[i].handle, d.data_ptr(), nb, t + 1000 * i, 4, 0, out.data_ptr(), 0, s.cuda_stream, 0)
        s.synchronize()
        if not np.array_equal(out.cpu().numpy(), ref[i]):
            bad.append(i)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    for h in hs:
        h.close()
    assert not bad


@pytest.mark.parametrize("nb,t", [(500, 20_000), (1300, 300_000)])  # one slab; several, on two streams
def test_captured_call_owns_its_memory(lib, nb, t):
    torch = pytest.importorskip("torch")
    bits = _bits(nb)
    c, c2 = _circuit(1), _circuit(2)
    with lib.Circuit(c.n_modes, c.occupation, c.gates) as h, lib.Circuit(c2.n_modes, c2.occupation, c2.gates) as other:
        ref = lib.ef_prob_approx(h.handle, bits, t, seed=4, want_stderr=False)
        d = torch.from_numpy(bits.view(np.int64)).cuda()
        out = torch.zeros(nb, dtype=torch.float64, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())

        def call():
            lib.ef_prob_approx_dev(h.handle, d.data_ptr(), nb, t, 4, 0, out.data_ptr(), 0, s.cuda_stream, 0)
        call()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call()
        for _ in range(2):
            out.zero_()
            big = lib.ef_prob_approx(other.handle, bits, 2 * t, seed=5, want_stderr=False)  # takes the pool's memory
            g.replay()
            again = lib.ef_prob_approx(other.handle, bits, 2 * t, seed=5, want_stderr=False)
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), ref) and np.array_equal(big, again)
        del g


KEPT = """
import numpy as np, torch
import paper_2511_12416_gb300 as ef, workloads as W
bits = W.spin_sector_bitstrings(6, 3, 3, 2000, np.random.default_rng(2))
torch.zeros(1, device="cuda")
def circuit(i):
    c = W.lucj_circuit(6, 3, 3, 1, n_onsite=6, n_same=3, angle_sampler=W.normal_var(1.0), seed=i)
    return ef.Circuit(c.n_modes, c.occupation, c.gates)
hs = [circuit(i) for i in range(400)]
for h in hs:
    ef.ef_prob_approx(h.handle, bits[:14], 1800, seed=1)  # some MiB each, kept by the circuit
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
ef.ef_prob_approx(hs[0].handle, bits, 25000, seed=1)  # 1 GiB while it runs
torch.cuda.synchronize()
print((free - torch.cuda.mem_get_info()[0]) / 2**30)
"""


def test_memory_of_calls_is_kept_beside_many_circuits(lib):
    """What the circuits hold does not count against what is kept for calls, else a large call's
    memory would be mapped anew every time."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", KEPT], cwd=root, env=dict(os.environ, PYTHONPATH=root), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert 0.9 <= float(r.stdout) <= 1.25
