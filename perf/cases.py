"""The work whose speed counts: one entry per way in which a program uses the library.

Every case is a circuit family with its sizes, an entry point, a precision and a number of
bitstrings. The structure of a circuit (which modes a gate acts on) belongs to the case; its angles
and the bitstrings are drawn from the seed. Sizes are those of the configurations in ``workloads``
and of the tests, or generic ones of the same ranges.

Circuit families (as in ``workloads``):

* ``lucj``: alpha modes 0..norb-1, beta modes norb..2 norb - 1, eta particles per spin; ``layers``
  Jastrow layers (``same`` neighbour pairs per spin, ``onsite`` opposite-spin pairs) between
  Haar-random orbital rotations; with ``inverse`` the last rotation undoes the first. Angles
  N(0, angle) as a variance, or uniform in [-angle, angle] with ``uniform``.
* ``brick``: one brick layer of Givens rotations, k controlled phases between its even and odd bonds.
* ``random``: ``depth`` brick layers, k controlled phases on random pairs between them.
* ``spins``: ``depth`` stages of norb / 2 + 1 brick layers per spin (every outcome of the sector occurs),
  k controlled phases of either kind between them.
"""
from __future__ import annotations

import math
from itertools import combinations

import numpy as np
import torch

import paper_2511_12416_gb300 as ef
from paper_2511_12416_gb300.autograd import BornProbabilities

PRECISION = {"fp64": ef.EF_PREC_FP64, "fp32": ef.EF_PREC_FP32_MINOR, "auto": ef.EF_PREC_AUTO}
GATE = np.dtype([("kind", "<i4"), ("p", "<i4"), ("q", "<i4"), ("reserved", "<i4"), ("theta", "<f8"), ("phi", "<f8")])

LUCJ32 = {"family": "lucj", "norb": 16, "eta": 8, "layers": 1, "onsite": 8, "same": 4, "angle": 0.1,
          "uniform": False, "inverse": True}
LUCJ40 = {"family": "lucj", "norb": 20, "eta": 6, "layers": 2, "onsite": 4, "same": 1, "angle": 0.1,
          "uniform": False, "inverse": False}
LUCJ52 = {"family": "lucj", "norb": 26, "eta": 5, "layers": 2, "onsite": 26, "same": 25, "angle": 0.05,
          "uniform": True, "inverse": False}


def listed():
    return [
        # one circuit of the smallest kind, its whole sector, from a loop that calls many such circuits
        {"name": "exact_8_modes", "op": "exact", "api": "dev", "precision": "fp64", "family": "brick",
         "n": 8, "eta": 4, "k": 3, "circuit": 0, "nb": 70},
        # one outcome of a random circuit at half filling: the latency that an interactive user sees
        {"name": "exact_one_outcome", "op": "exact", "api": "host", "precision": "auto", "family": "random",
         "n": 24, "eta": 12, "k": 16, "depth": 4, "circuit": 7, "nb": 1},
        # the probabilities of a sampled set of bitstrings, on the device, default precision
        {"name": "exact_lucj32", "op": "exact", "api": "dev", "precision": "auto", **LUCJ32, "nb": 10000},
        # the same from and to host arrays with the error estimates, an odd and smaller set
        {"name": "exact_lucj32_host", "op": "exact", "api": "host_err", "precision": "auto", **LUCJ32, "nb": 1537},
        # reference values of a part of the set in plain FP64
        {"name": "exact_lucj32_fp64", "op": "exact", "api": "dev", "precision": "fp64", **LUCJ32, "nb": 2000},
        # inside a program that allows no allocation, FP32 minors
        {"name": "exact_noalloc_fp32", "op": "exact", "api": "noalloc", "precision": "fp32", **LUCJ32, "nb": 3000},
        # the estimator over a set of bitstrings of a circuit far beyond the Exact algorithm,
        # ceil(extent / 0.01^2) trajectories each, with standard errors and error estimates
        {"name": "raw_lucj52", "op": "raw", "api": "dev", "precision": "auto", **LUCJ52, "nb": 8192, "t": 68416},
        # a handful of bitstrings of it
        {"name": "raw_lucj52_few", "op": "raw", "api": "host", "precision": "auto", **LUCJ52, "nb": 16, "t": 68416},
        # the estimator in plain FP64 on a mid-size circuit of three layers with larger angles
        {"name": "raw_24_modes_fp64", "op": "raw", "api": "dev", "precision": "fp64", "family": "lucj", "norb": 12,
         "eta": 4, "layers": 3, "onsite": 6, "same": 3, "angle": 0.1, "uniform": False, "inverse": False,
         "nb": 500, "t": 5000},
        # estimates to a stated accuracy: rounds of the estimator that tighten their bounds
        {"name": "estimate_lucj52", "op": "estimate", **LUCJ52, "nb": 1000, "eps": 0.02, "delta": 0.01},
        # one step of fitting the angles: new angles in, log-likelihood forward and backward
        {"name": "train_lucj40", "op": "train", "precision": "auto", **LUCJ40, "nb": 4096},
        # many circuits of uneven sizes as one batch, Exact and sampled ones together
        {"name": "batch_uneven", "op": "batch", "circuits": 12, "circuit": 6, "most_bits": 10000, "t": 10000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["exact", "exact", "exact", "raw", "raw", "raw", "estimate", "train", "batch", "single"])
    if op == "single":
        n = rng.randint(4, 14) * 2
        return {"op": "exact", "api": rng.choice(["host", "dev"]), "precision": rng.choice(["auto", "auto", "fp64"]),
                "family": "random", "n": n, "eta": n // 2, "k": rng.randint(8, 14), "depth": rng.randint(3, 5),
                "circuit": rng.randint(0, 999), "nb": rng.randint(1, 8)}
    if op == "exact":
        c = _lucj(rng, 6, 40, 2, 9, (1, 1, 2), 8, 5)
        precision = rng.choice(["auto", "auto", "fp32", "fp64"])
        r = c["layers"] * max(c["onsite"], c["same"] + 1)
        # at most the minors, and the FP64 work, of the listed calls
        most = (1 << 22) // (1 << r) * 8 ** 3 // max(2, c["eta"]) ** 3
        most = most // 4 if precision == "fp64" else most
        nb = min(_log_int(rng, 30, 20000), max(1, most))
        small = nb * 2.0 ** r < 7e5 and c["norb"] <= 16
        api = rng.choice(["dev", "dev", "host", "host_err"] + (["noalloc"] if small else []))
        return {"op": "exact", "api": api, "precision": precision, **c, "nb": nb}
    if op == "raw":
        c = _lucj(rng, 6, 26, 2, 10, (1, 1, 2, 2, 3), 26, 25)
        if c["layers"] == 3 and c["norb"] > 16:
            c["layers"] = 2
        c["uniform"] = rng.random() < 0.6
        c["angle"] = 0.05 if c["uniform"] else 0.1
        if not c["uniform"]:
            c["onsite"], c["same"] = min(c["onsite"], 8), min(c["same"], 4)
        precision = rng.choice(["auto", "auto", "fp32", "fp64"])
        t = _log_int(rng, 1000, 100000)
        blocks = (c["layers"] * (c["onsite"] + 2 * c["same"]) + 3) // 4
        most = int(2e10 / (t * max(blocks, 6)) / (40 if precision == "fp64" else 8))
        return {"op": "raw", "api": rng.choice(["dev", "host"]), "precision": precision, **c,
                "nb": max(1, min(_log_int(rng, 1, 8192), most)), "t": t}
    if op == "estimate":
        c = dict(LUCJ52, norb=rng.randint(8, 26), eta=rng.randint(2, 6))
        c["onsite"], c["same"] = c["norb"], c["norb"] - 1
        return {"op": "estimate", **c, "nb": _log_int(rng, 10, 1000), "eps": rng.choice([0.02, 0.03, 0.05, 0.1]),
                "delta": rng.choice([0.01, 0.05])}
    if op == "train":
        c = _lucj(rng, 6, 24, 2, 7, (1, 2), 4, 2)
        return {"op": "train", "precision": rng.choice(["auto", "fp64"]), **c, "nb": _log_int(rng, 50, 2000)}
    return {"op": "batch", "circuits": rng.randint(3, 12), "circuit": rng.randint(0, 999),
            "most_bits": _log_int(rng, 200, 4000), "t": _log_int(rng, 1000, 8000)}


def _lucj(rng, norb_lo, norb_hi, eta_lo, eta_hi, layers, onsite_hi, same_hi):
    norb = rng.randint(norb_lo, norb_hi)
    nlay = rng.choice(layers)
    most = max(1, onsite_hi // nlay) if onsite_hi <= 12 else onsite_hi
    return {"family": "lucj", "norb": norb, "eta": rng.randint(eta_lo, max(eta_lo, min(eta_hi, norb // 2))),
            "layers": nlay, "onsite": rng.randint(1, min(most, norb)),
            "same": rng.randint(1, max(1, min(same_hi // nlay if same_hi <= 12 else same_hi, norb - 1))),
            "angle": 0.1, "uniform": False, "inverse": nlay == 1 and rng.random() < 0.5}


# ------------------------------------------------------------------ circuits and bitstrings


def _haar(n, rng):
    z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    q, r = np.linalg.qr(z)
    d = np.diag(r)
    return q * (d / np.abs(d))


def _rotation(n, rng, at):
    """A Haar-random orbital rotation as phases and nearest-neighbour Givens rotations."""
    w = _haar(n, rng)
    rots = []
    for c in range(n - 1):
        for i in range(n - 2, c - 1, -1):
            a, b = w[i, c], w[i + 1, c]
            theta, phi = math.atan2(abs(b), abs(a)), float(np.angle(-a * np.conj(b)))
            ct, st, e = math.cos(theta), math.sin(theta), np.exp(1j * phi)
            lo, hi = w[i].copy(), w[i + 1].copy()
            w[i], w[i + 1] = ct * lo - e * st * hi, np.conj(e) * st * lo + ct * hi
            rots.append((0, at + i, at + i + 1, -theta, phi))
    return [(1, at + p, at + p, 0.0, float(np.angle(w[p, p]))) for p in range(n)] + rots[::-1]


def _undo(recs):
    return [(k, p, q, -t, f) if k == 0 else (k, p, q, 0.0, -f) for k, p, q, t, f in reversed(recs)]


def _bricks(n, rng, at):
    return [(0, at + p, at + p + 1, *rng.uniform(0, 2 * math.pi, 2)) for s in (0, 1) for p in range(s, n - 1, 2)]


def _circuit(case, rng):
    """Gate records, blocks of modes that rotations join as (first mode, modes), particles per block."""
    f = case["family"]
    place = np.random.default_rng([case.get("circuit", 0), 17])  # where the gates sit: the case's, not the seed's
    if f == "lucj":
        m = case["norb"]
        rot = [_rotation(m, rng, 0) + _rotation(m, rng, m)]
        recs = list(rot[0])
        pairs = [(p, p + 1) for p in range(case["same"])]
        pairs += [(m + p, m + p + 1) for p in range(case["same"])]
        pairs += [(p, m + p) for p in range(case["onsite"])]
        for layer in range(case["layers"]):
            a = case["angle"]
            ts = rng.uniform(-a, a, len(pairs)) if case["uniform"] else rng.normal(0.0, math.sqrt(a), len(pairs))
            recs += [(2, p, q, float(t), 0.0) for (p, q), t in zip(pairs, ts)]
            recs += _undo(rot[0]) if case["inverse"] else _rotation(m, rng, 0) + _rotation(m, rng, m)
        return recs, [(0, m), (m, m)], [case["eta"]] * 2
    if f == "brick":
        n = case["n"]
        b = _bricks(n, rng, 0)
        cps = [(2, *(int(x) for x in place.choice(n, 2, replace=False)), float(rng.uniform(0, math.pi / 4)), 0.0)
               for _ in range(case["k"])]
        return b[:n // 2] + cps + b[n // 2:], [(0, n)], [case["eta"]]
    if f == "random":
        n, recs = case["n"], []
        slots = sorted(place.integers(0, case["depth"] + 1, case["k"]).tolist())
        for layer in range(case["depth"] + 1):
            recs += [(2, *(int(x) for x in place.choice(n, 2, replace=False)), float(rng.normal()), 0.0)
                     for s in slots if s == layer]
            recs += _bricks(n, rng, 0) if layer < case["depth"] else []
        return recs, [(0, n)], [case["eta"]]
    m, recs = case["norb"], []  # spins
    slots = sorted(place.integers(0, case["depth"] + 1, case["k"]).tolist())
    for layer in range(case["depth"] + 1):
        for s in slots:
            if s == layer:
                p, side = int(place.integers(0, m - 1)), int(place.integers(0, 4))
                pair = (p, m + p) if side > 1 else (side * m + p, side * m + p + 1)
                recs.append((2, *pair, float(rng.normal(0.0, math.sqrt(0.1))), 0.0))
        for _ in range(m // 2 + 1 if layer < case["depth"] else 0):
            recs += _bricks(m, rng, 0) + _bricks(m, rng, m)
    return recs, [(0, m), (m, m)], [case["eta"]] * 2


def _rows(rng, case, blocks, etas, nb):
    """Occupied modes of nb bitstrings, uniform in the sector: one (nb, eta) array per block, ascending.
    ``brick``: the sector in order; ``random``: outcomes that its few brick layers reach."""
    out = []
    for (_, n), e in zip(blocks, etas):
        if case["family"] == "brick":
            out.append(np.array(list(combinations(range(n), e)))[:nb])
            continue
        near = min(e, n - e, case["depth"]) if case["family"] == "random" else e
        width = 2 * near if case["family"] == "random" else n
        moved = np.argsort(rng.random((nb, width)), axis=1)[:, :near] + e - near
        kept = np.broadcast_to(np.arange(e - near), (nb, e - near))
        out.append(np.sort(np.concatenate([kept, moved], axis=1), axis=1))
    return out


def _words(rows, blocks, nb):
    w = np.zeros((nb, 2), dtype=np.uint64)
    for r, (at, _) in zip(rows, blocks):
        for j in range(r.shape[1]):
            m = r[:, j] + at
            np.bitwise_or.at(w, (np.arange(nb), m >> 6), np.uint64(1) << (m & 63).astype(np.uint64))
    return w


def _inputs(case, seed):
    rng = np.random.default_rng([seed, 11])
    recs, blocks, etas = _circuit(case, rng)
    gates = np.array([(k, p, q, 0, t, f) for k, p, q, t, f in recs], dtype=GATE)
    rows = _rows(rng, case, blocks, etas, case["nb"])
    bits = _words(rows, blocks, case["nb"])
    occ = _words([np.arange(e)[None, :] for e in etas], blocks, 1)[0]
    n = sum(b[1] for b in blocks)
    return {"rng": rng, "gates": gates, "blocks": blocks, "etas": etas, "rows": rows, "bits": bits, "occ": occ, "n": n}


def _members(case):
    """The circuits of a batch: uneven sizes, Exact up to 14 controlled phases, else the estimator."""
    place = np.random.default_rng([case["circuit"], 23])
    out = []
    for i in range(case["circuits"]):
        n = int(place.choice(np.arange(12, 41, 2)))
        eta = int(place.integers(2, n // 3 + 1))
        k = int(place.integers(4, 25))
        nb = int(round(math.exp(place.uniform(math.log(100.0), math.log(case["most_bits"])))))
        out.append({"family": "spins", "norb": n // 2, "eta": min(eta, n // 2), "k": k,
                    "depth": int(place.integers(1, 4)), "circuit": 1000 * case["circuit"] + i, "nb": nb,
                    "t": 0 if k <= 14 else case["t"]})
    return out


class _Batch:
    def __init__(self, circuits):
        self.circuits = circuits
        self.handle = ef.ef_batch_create([c.handle for c in circuits])

    def __del__(self):
        ef.ef_batch_destroy(self.handle)


def _device(bits):
    return torch.from_numpy(bits.view(np.int64)).cuda()


def prepare(case, seed):
    if case["op"] == "batch":
        ins = [_inputs(m, 7919 * seed + i) for i, m in enumerate(_members(case))]
        batch = _Batch([ef.Circuit(x["n"], x["occ"], x["gates"]) for x in ins])
        bits = [_device(x["bits"]) for x in ins]
        return {"case": case, "batch": batch, "bits": bits, "seed": seed, "t": [m["t"] for m in _members(case)],
                "out": [torch.zeros(len(b), dtype=torch.float64, device="cuda") for b in bits]}
    x = _inputs(case, seed)
    c = ef.Circuit(x["n"], x["occ"], x["gates"], precision=PRECISION[case.get("precision", "auto")])
    s = {"case": case, "circuit": c, "bits": x["bits"], "seed": seed}
    if case["op"] == "train":
        s["bits"] = _device(x["bits"])
        s["angles"] = torch.from_numpy(ef.ef_circuit_get_angles(c.handle))
        s["weights"] = torch.from_numpy(x["rng"].uniform(0.0, 1.0, case["nb"])).cuda()
    elif case.get("api") in ("dev", "noalloc"):
        s["bits"] = _device(x["bits"])
        s["out"] = [torch.zeros(case["nb"], dtype=torch.float64, device="cuda") for _ in range(3)]
    return s


def run(s):
    case = s["case"]
    stream = torch.cuda.current_stream().cuda_stream
    if case["op"] == "batch":
        ef.ef_batch_prob_dev(s["batch"].handle, [b.data_ptr() for b in s["bits"]], [len(b) for b in s["bits"]],
                             [o.data_ptr() for o in s["out"]], s["t"], seed=s["seed"], stream=stream)
        return {"p": s["out"]}
    h, nb = s["circuit"].handle, case["nb"]
    if case["op"] == "train":
        angles = s["angles"].detach().requires_grad_(True)
        p = BornProbabilities.apply(angles, h, s["bits"])
        loss = (s["weights"] * torch.log(p)).sum()
        loss.backward()
        return {"p": p.detach(), "grad": angles.grad}
    if case["op"] == "estimate":
        p, se, t = ef.ef_prob_estimate(h, s["bits"], case["eps"], case["delta"], seed=s["seed"])
        return {"p": p, "se": se, "t": t}
    if case["op"] == "raw":
        if case["api"] == "host":
            p, se = ef.ef_prob_approx(h, s["bits"], case["t"], seed=s["seed"])
            return {"p": p, "se": se}
        p, se, err = s["out"]
        ef.ef_prob_approx_dev(h, s["bits"].data_ptr(), nb, case["t"], s["seed"], 0, p.data_ptr(), se.data_ptr(),
                              stream, err.data_ptr())
        return {"p": p, "se": se, "err": err}
    if case["api"] == "host":
        return {"p": ef.ef_prob_exact(h, s["bits"])}
    if case["api"] == "host_err":
        p, err = ef.ef_prob_exact(h, s["bits"], want_err=True)
        return {"p": p, "err": err}
    call = ef.ef_prob_exact_noalloc_dev if case["api"] == "noalloc" else ef.ef_prob_exact_dev
    call(h, s["bits"].data_ptr(), nb, s["out"][0].data_ptr(), 0, stream)
    return {"p": s["out"][0]}


# ------------------------------------------------------------------ what a pass cannot do without


def _lu(eta):
    return 17.0 * eta + sum(8.0 * (eta - k - 1) ** 2 + 6.0 * (eta - k - 1) for k in range(eta))


def _exact_minors(case):
    """(Distinct minors per bitstring, particles): the flip patterns of every block."""
    if case["family"] == "lucj":
        return 2.0 * 2.0 ** (case["layers"] * max(case["onsite"], case["same"] + 1)), case["eta"]
    if case["family"] == "spins":
        return 2.0 * 2.0 ** (case["k"] / 2.0), case["eta"]
    return 2.0 ** case["k"], case["eta"]


def _raw_ops(case, k, t):
    # integer operations of the sampling: per four gates one Philox4x32-10 block (ten rounds of two wide
    # multiplications and four exclusive ors) and four comparisons
    return case["nb"] * float(t) * math.ceil(k / 4) * 64.0


def work(case):
    """Bytes: bitstrings in, results out. Operations: one elimination per distinct minor (complex, as
    real operations; three times for a gradient: value, inverse and accumulation), or the sampling."""
    if case["op"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for m in _members(case):
            minors, eta = _exact_minors(m)
            total["bytes"] += 24.0 * m["nb"]
            total["flops"] += _raw_ops(m, m["k"], m["t"]) if m["t"] else m["nb"] * minors * _lu(eta)
        return total
    nb = case["nb"]
    if case["op"] in ("raw", "estimate"):
        k = case["layers"] * (case["onsite"] + 2 * case["same"])
        t = case["t"] if case["op"] == "raw" else 3000.0 / case["eps"]  # rounds of growing size, about this in all
        return {"bytes": nb * 40.0, "flops": _raw_ops(case, k, t)}
    minors, eta = _exact_minors(case)
    return {"bytes": nb * 24.0, "flops": nb * minors * _lu(eta) * (3.0 if case["op"] == "train" else 1.0)}


# ------------------------------------------------------------------ the same in 64 bits, by plain dense algebra


def _f64(v):
    return torch.tensor(float(v), dtype=torch.float64)


def _segments(gates, at, n, angles=None):
    """The block's rotations between its layers of controlled phases, and the layers: (gate number
    among the controlled phases, local modes). ``angles``: per gate (theta, phi) as tensors."""
    segs, layers, j, open_ = [], [], 0, False
    rows = list(torch.eye(n, dtype=torch.complex128))
    for i, g in enumerate(gates):
        kind, p, q = int(g["kind"]), int(g["p"]) - at, int(g["q"]) - at
        theta, phi = angles[i] if angles is not None else (_f64(g["theta"]), _f64(g["phi"]))
        if kind == 2:
            modes = [m for m in (p, q) if 0 <= m < n]
            if modes:
                if not open_:
                    segs.append(torch.stack(rows))
                    layers.append([])
                    rows, open_ = list(torch.eye(n, dtype=torch.complex128)), True
                layers[-1].append((j, modes, theta))
            j += 1
            continue
        if not 0 <= p < n:
            continue
        open_ = False
        e = torch.polar(torch.ones((), dtype=torch.float64), phi)
        if kind == 1:
            rows[p] = e * rows[p]
        else:
            ct, st = torch.cos(theta), torch.sin(theta)
            rows[p], rows[q] = ct * rows[p] - e * st * rows[q], e.conj() * st * rows[p] + ct * rows[q]
    segs.append(torch.stack(rows))
    return segs, layers


def _base_phases(layer, n):
    ph = torch.zeros(n, dtype=torch.float64)
    for _, modes, theta in layer:
        for m in modes:
            ph = ph + 0.5 * theta * torch.nn.functional.one_hot(torch.tensor(m), n)
    return torch.polar(torch.ones(n, dtype=torch.float64), ph)


def _flips(layers, n, x):
    """Signs of every (layer, mode) for controlled-phase bits x (rows): list of (rows, n) tensors."""
    out = []
    for layer in layers:
        par = torch.zeros((x.shape[0], n), dtype=torch.int64, device=x.device)
        for j, modes, _ in layer:
            for m in modes:
                par[:, m] ^= x[:, j]
        out.append(1.0 - 2.0 * par.to(torch.float64))
    return out


def _columns(segs, layers, eta, signs, dev):
    """U(x)[:, first eta columns] for every row of signs."""
    n = segs[0].shape[0]
    u = segs[0].to(dev)[None, :, :eta]
    for layer, seg, sg in zip(layers, segs[1:], signs):
        t = seg.to(dev) * _base_phases(layer, n).to(dev)[None, :]
        u = torch.einsum("ij,bjk->bik", t, sg[:, :, None] * u)
    return u if signs else u.clone()


def _det(a):
    """Determinants of a batch by elimination with partial pivoting."""
    a = a.clone()
    n, at = a.shape[-1], torch.arange(a.shape[0], device=a.device)
    d = torch.ones(a.shape[0], dtype=a.dtype, device=a.device)
    for k in range(n):
        p = a[:, k:, k].abs().argmax(1) + k
        top, old = a[at, p], a[:, k].clone()
        a[at, p] = old
        a[:, k] = top
        d = d * torch.where(p != k, -1.0, 1.0) * top[:, k]
        if k + 1 < n:
            l = torch.where(top[:, k:k + 1] == 0, torch.zeros_like(a[:, k + 1:, k]),
                            a[:, k + 1:, k] / torch.where(top[:, k:k + 1] == 0, torch.ones_like(top[:, k:k + 1]), top[:, k:k + 1]))
            a[:, k + 1:] -= l[:, :, None] * top[:, None, :]
    return d


def _minors(u, rows, det):
    """det u[pattern][rows of the bitstring] as (bitstrings, patterns)."""
    e, out = rows.shape[1], []
    step = max(1, (1 << 25) // (u.shape[0] * e * e))
    for i in range(0, len(rows), step):
        r = rows[i:i + step]
        a = u[:, r.reshape(-1)].reshape(u.shape[0] * len(r), e, e)
        out.append(det(a).reshape(u.shape[0], len(r)).T)
    return torch.cat(out)


def _probabilities(x, dev, angles=None, det=_det):
    cps = [i for i, g in enumerate(x["gates"]) if int(g["kind"]) == 2]
    theta = [angles[i][0] if angles is not None else _f64(x["gates"][i]["theta"]) for i in cps]
    mode = [(int(x["gates"][i]["p"]), int(x["gates"][i]["q"])) for i in cps]
    inside = [[[at <= m < at + n for m in pq] for pq in mode] for at, n in x["blocks"]]
    shared = [j for j in range(len(cps)) if len(x["blocks"]) == 2 and any(inside[0][j]) and any(inside[1][j])]

    def weights(js):  # product weights and bits of every vector over the gates js
        bits = (torch.arange(1 << len(js))[:, None] >> torch.arange(max(1, len(js)))) & 1
        w = torch.ones(1 << len(js), dtype=torch.complex128)
        for i, j in enumerate(js):
            w = w * torch.where(bits[:, i] == 1, 1j * torch.sin(theta[j] / 4), torch.cos(theta[j] / 4) + 0j)
        return w, bits

    ws, sbits = weights(shared)
    amp = ws.to(dev)[None, :]
    for (at, n), eta, rows, ins in zip(x["blocks"], x["etas"], x["rows"], inside):
        segs, layers = _segments(x["gates"], at, n, angles)
        local = [j for j in range(len(cps)) if all(ins[j])]
        wl, lbits = weights(local)
        full = torch.zeros((len(ws) * len(wl), len(cps)), dtype=torch.int64)
        for i, j in enumerate(shared):
            full[:, j] = sbits[:, i].repeat_interleave(len(wl))
        for i, j in enumerate(local):
            full[:, j] = lbits[:, i].repeat(len(ws))
        mark = np.random.default_rng(3).integers(0, 1 << 62, (max(1, len(layers)), n))
        key = np.zeros(len(full), dtype=np.int64)
        for l, layer in enumerate(layers):
            for j, modes, _ in layer:
                for m in modes:
                    key ^= full[:, j].numpy() * mark[l, m]
        _, first, inv = np.unique(key, return_index=True, return_inverse=True)
        u = _columns(segs, layers, eta, [s.to(dev) for s in _flips(layers, n, full[torch.from_numpy(first)])], dev)
        d = _minors(u, torch.from_numpy(rows).to(dev), det)
        w = torch.zeros((len(first), len(ws)), dtype=torch.complex128)
        w = w.index_put((torch.from_numpy(inv.reshape(-1)), torch.arange(len(ws)).repeat_interleave(len(wl))),
                        wl.repeat(len(ws)), accumulate=True)
        amp = amp * (d @ w.to(dev))
    a = amp.sum(1)
    return a.real ** 2 + a.imag ** 2


def _philox(c, k0, k1):
    lo = 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & lo) ^ c[1] ^ k0, p1 & lo, ((p0 >> 32) & lo) ^ c[3] ^ k1, p0 & lo]
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    return c


def _raw(x, t, seed, dev):
    """The estimator on the trajectories that the seed and the bitstring's number give."""
    cps = [g for g in x["gates"] if int(g["kind"]) == 2]
    th = np.array([float(g["theta"]) for g in cps])
    th = th - 2 * np.pi * np.floor((th + np.pi) / (2 * np.pi))
    sa, ca = np.sin(np.abs(th) / 4), np.cos(th / 4)
    T = np.where(sa != 0, np.clip(np.floor(sa / (sa + ca) * 2.0 ** 32 + 0.5), 1, 4294967295), 0)
    p1 = T / 2.0 ** 32
    ratio = np.where(T > 0, np.sin(th / 4) / np.maximum(p1, 1e-300), 0.0) / (ca / (1 - p1))
    r0 = float(np.prod(ca / (1 - p1)))
    T = torch.from_numpy(T.astype(np.int64)).to(dev)
    lr = torch.from_numpy(np.log(np.maximum(np.abs(ratio), 1e-300))).to(dev)
    neg = torch.from_numpy((ratio < 0).astype(np.int64)).to(dev)
    blocks = [(*_segments(x["gates"], at, n), n, eta, rows) for (at, n), eta, rows in zip(x["blocks"], x["etas"], x["rows"])]
    q = torch.arange((len(cps) + 3) // 4, device=dev)[None, :]
    ps, ses = [], []
    step = 1 << 16
    for b in range(len(x["bits"])):
        ys = []
        for s0 in range(0, t, step):
            s = torch.arange(s0, min(t, s0 + step), device=dev)[:, None]
            zero = torch.zeros((len(s), q.shape[1]), dtype=torch.int64, device=dev)
            u = torch.stack(_philox([q + zero, s + zero, zero + b, zero], seed & 0xFFFFFFFF, seed >> 32), dim=2)
            bit = (u.reshape(len(s), -1)[:, :len(cps)] < T[None, :]).to(torch.int64)
            size = r0 * torch.exp(bit.to(torch.float64) @ lr)
            turns = (bit.sum(1) + 2 * (bit * neg).sum(1)) & 3  # i per flipped gate, -1 per negative ratio
            y = size * torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device=dev)[turns]
            for segs, layers, n, eta, rows in blocks:
                cols = _columns(segs, layers, eta, _flips(layers, n, bit), dev)
                y = y * _det(cols[:, torch.from_numpy(rows[b]).to(dev)].expand(len(s), eta, eta))
            ys.append(y)
        y = torch.cat(ys)
        a = y.mean()
        ps.append(float(a.abs() ** 2))
        ses.append(2 * math.sqrt(max(0.0, float((a.conj() * y).real.var())) / t) if t > 1 else 0.0)
    return np.array(ps), np.array(ses)


class _PlainDet(torch.autograd.Function):
    @staticmethod
    def forward(ctx, a):
        d = _det(a)
        ctx.save_for_backward(a, d)
        return d

    @staticmethod
    def backward(ctx, g):
        a, d = ctx.saved_tensors
        n, at = a.shape[-1], torch.arange(a.shape[0], device=a.device)
        m = torch.cat([a, torch.eye(n, dtype=a.dtype, device=a.device).expand_as(a)], 2)  # Gauss-Jordan
        for k in range(n):
            p = m[:, k:, k].abs().argmax(1) + k
            top, old = m[at, p], m[:, k].clone()
            m[at, p] = old
            top = top / top[:, k:k + 1]
            m = m - m[:, :, k:k + 1] * top[:, None, :]
            m[:, k] = top
        return (g * d.conj())[:, None, None] * m[:, :, n:].transpose(1, 2).conj()


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["op"] == "estimate":
        return None
    if case["op"] == "batch":
        out = []
        for i, m in enumerate(_members(case)):
            big = m["t"] or m["nb"] * 2.0 ** m["k"] * m["eta"] ** 3 > 3e10
            out.append(None if big else _probabilities(_inputs(m, 7919 * seed + i), dev).cpu())
        return {"p": out}
    x = _inputs(case, seed)
    if case["op"] == "raw":
        if case["nb"] * case["t"] * case["layers"] * case["norb"] ** 2 * case["eta"] > 2e10:
            return None
        p, se = _raw(x, case["t"], seed, dev)
        return {"p": p, "se": se} if case["api"] == "host" else {"p": p, "se": se, "err": None}
    if case["op"] == "train":
        flat, angles = [], []
        for g in x["gates"]:
            kind = int(g["kind"])
            vals = [torch.tensor(float(g[f]), dtype=torch.float64, requires_grad=True) for f in
                    (("theta", "phi") if kind == 0 else ("phi",) if kind == 1 else ("theta",))]
            flat += vals
            angles.append((vals[0], vals[-1]))
        p = _probabilities(x, dev, angles, _PlainDet.apply)
        w = torch.from_numpy(x["rng"].uniform(0.0, 1.0, case["nb"])).to(dev)
        grads = torch.autograd.grad((w * torch.log(p)).sum(), flat)
        return {"p": p.detach().cpu(), "grad": torch.stack([g.cpu() for g in grads])}
    p = _probabilities(x, dev).cpu()
    return {"p": p, "err": None} if case["api"] == "host_err" else {"p": p}
