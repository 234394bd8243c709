"""The calls whose speed counts: samples of random sequential adsorption run to
jamming with their first-wrap counts, through the package's public entry points.

A case is a plain dict.  ``api`` says how the samples are run:

``handle``  one shape on its own handle: ``Lattice.run``;
``small``   one CTA per sample, results to the host: ``rsa_run_small``;
``static``  the run that allocates nothing: ``rsa_run_static``;
``mix``     a batch of uneven shapes in one call: ``rsa_run_mix`` (shapes
            ``L = ratio * k`` for each k of ``ks``, n samples of each);
``wrap``    a handle's run, then for every sample the directions in which its
            first ``cover * L^2 / k`` k-mers wind, and its contact counts;
``sizes``   a handle's run, then for every sample the cluster sizes of as many
            k-mers, and its contact counts.

Sample seeds are consecutive from a random start, as a run of many samples
takes them.  Every result is a whole number.
"""
from __future__ import annotations

import math
import os

import numpy as np

from paper_1810_06800_gb300 import rsa


def listed():
    return [
        # one small request of a latency-critical loop that may not allocate
        dict(name="static_L256_k16_n4", api="static", L=256, k=16, n=4),
        # the plain small configuration: 100 samples of L = 64, k = 4, the way
        # the server runs a small job and the way a handle does
        dict(name="small_L64_k4_n100", api="small", L=64, k=4, n=100),
        dict(name="handle_L64_k4_n100", api="handle", L=64, k=4, n=100),
        # a single sample of the plain path at scale: no batch to hide behind
        dict(name="handle_L1024_k32_n1", api="handle", L=1024, k=32, n=1),
        # the plain path at scale: 1000 samples in one batch
        dict(name="handle_L1024_k32_n1000", api="handle", L=1024, k=32, n=1000),
        # wrapping probabilities at k = 1, i.e. site percolation: as many
        # k-mers as cells, so the contact graph and its search are largest
        dict(name="wrap_L512_k1_n100", api="wrap", L=512, k=1, n=100, cover=0.592746),
        # cluster sizes near the percolation threshold for long k-mers
        dict(name="sizes_L2048_k256_n32", api="sizes", L=2048, k=256, n=32, cover=0.53),
        # lattices of 100 k-mer lengths, the ratio of the published tables:
        # short k on a side that no tile divides, long k on a side that is not
        # a power of two
        dict(name="handle_L400_k4_n100", api="handle", L=400, k=4, n=100),
        dict(name="handle_L6400_k64_n4", api="handle", L=6400, k=64, n=4),
        # an odd side with a k that is no power of two
        dict(name="handle_L777_k100_n16", api="handle", L=777, k=100, n=16),
        # a batch of uneven shapes, lattices of 32 to 8192 cells a side
        dict(name="mix_k2-8-64-512_n32", api="mix", ks="2,8,64,512", ratio=16, n=32),
        # the largest lattice and the longest k-mers
        dict(name="handle_L32768_k4096_n4", api="handle", L=32768, k=4096, n=4),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _count(rng, L, most_cells, most=256):
    return _log_uniform(rng, 1, max(1, min(most, most_cells // (L * L))))


def draw(rng):
    api = rng.choice(["handle"] * 6 + ["small", "static", "mix", "wrap", "sizes"])
    if api == "small":
        L = rng.randint(8, 128)
        k = _log_uniform(rng, max(1, -(-L * L // 4096)), max(1, L // 4))
        return dict(api=api, L=L, k=k, n=rng.randint(16, 256))
    if api == "static":
        L = _log_uniform(rng, 16, 512)
        if rng.random() < 0.5:
            L = max(32, L // 32 * 32)
        k = _log_uniform(rng, 1, L // 8)
        n = _count(rng, L, 1 << 19, 16)
        return dict(api=api, L=L, k=k, n=n)
    if api == "mix":
        ratio = rng.choice([8, 16, 32])
        ks = sorted(rng.sample([1, 2, 3, 4, 8, 16, 32, 50, 64, 128, 256], rng.randint(2, 4)))
        big = ratio * ks[-1]
        return dict(api=api, ks=",".join(map(str, ks)), ratio=ratio,
                    n=_count(rng, big, 1 << 28, 64))
    if rng.random() < 0.5:
        # the served shapes: k a power of two, L / k in 8 .. 32
        k = 1 << rng.randint(0, 10)
        L = rng.choice([8, 16, 32]) * k
        L = min(L, 16384)
        cells = 1 << 30
    else:
        # any k, and up to the 100 k-mer lengths of the published tables
        k = _log_uniform(rng, 1, 400)
        L = min(_log_uniform(rng, 8, 100) * k + rng.choice([0, 0, 1, 7]), 8000)
        cells = 1 << 27
    L = max(L, 16)
    if api in ("wrap", "sizes"):
        return dict(api=api, L=L, k=k, n=_count(rng, L, cells // 16, 64),
                    cover=round(rng.uniform(0.3, 0.5), 3))
    return dict(api=api, L=L, k=k, n=_count(rng, L, cells))


def _shapes(case):
    """(L, k) of every sample of a mixed batch, shapes interleaved."""
    ks = [int(k) for k in case["ks"].split(",")]
    k = np.array(ks * case["n"], dtype=np.uint32)
    return k * np.uint32(case["ratio"]), k


def _placed(case):
    return round(case["cover"] * case["L"] ** 2 / case["k"])


def _seeds(case, seed):
    n = _shapes(case)[0].size if case["api"] == "mix" else case["n"]
    start = int(np.random.default_rng(seed).integers(0, 2**62))
    return np.arange(start, start + n, dtype=np.uint64)


def prepare(case, seed):
    state = dict(api=case["api"], seeds=_seeds(case, seed))
    if case["api"] == "mix":
        # the library's own choices for every shape, no tuning measurements
        os.environ["RSA_AUTOTUNE"] = "0"
        state["L"], state["k"] = _shapes(case)
    else:
        state["L"], state["k"] = case["L"], case["k"]
        if case["api"] in ("handle", "wrap", "sizes"):
            state["lattice"] = rsa.Lattice(case["L"], case["k"])
        if "cover" in case:
            state["m"] = _placed(case)
    return state


def run(state):
    api, seeds = state["api"], state["seeds"]
    if api == "small":
        return rsa.rsa_run_small(state["L"], state["k"], seeds)
    if api == "static":
        return rsa.rsa_run_static(state["L"], state["k"], seeds)
    if api == "mix":
        return rsa.rsa_run_mix(state["L"], state["k"], seeds)
    lat = state["lattice"]
    nj, nc = lat.run(seeds)
    if api == "handle":
        return nj, nc
    read = lat.wrap_dirs if api == "wrap" else lat.cluster_sizes
    rows = [read(i, state["m"]) for i in range(seeds.size)]
    return [nj, nc, *lat.contacts(seeds.size), np.array(rows)]


def work(case):
    """Seeds in and results out; the arithmetic is one 64-bit priority (a
    splitmix64 output, about 20 integer operations) for each of the two
    candidates of every cell."""
    if case["api"] == "mix":
        L, k = _shapes(case)
    else:
        L, k = np.full(case["n"], case["L"]), np.full(case["n"], case["k"])
    L, k = L.astype(np.float64), k.astype(np.float64)
    out = 8.0 * L.size
    if case["api"] in ("wrap", "sizes"):
        out += (14.0 if case["api"] == "wrap" else 12.0 + 4.0 * (_placed(case) + 1)) * L.size
    return {"bytes": 8.0 * L.size + out, "flops": float((2 * 20 * L * L).sum())}


# ---- the same results from the definition, one candidate after another ----

_M = (1 << 64) - 1


def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _sample(L, k, seed):
    """n_j and n_c: try every placement once in the order of its priority,
    and join each accepted k-mer to its neighbours with their displacement."""
    gamma = 0x9E3779B97F4A7C15
    base = _mix(np.array([(seed + gamma) & _M], dtype=np.uint64))
    order = np.argsort(_mix(base + np.uint64(gamma) * np.arange(1, 2 * L * L + 1, dtype=np.uint64)))
    owner, where, parent, off = {}, [], [], []
    n_c = None

    def find(a):
        dx = dy = 0
        while parent[a] != a:
            dx, dy, a = dx + off[a][0], dy + off[a][1], parent[a]
        return a, dx, dy

    for idx in order.tolist():
        o, r = divmod(idx, L * L)
        y, x = divmod(r, L)
        cells = [(y, (x + i) % L) if o == 0 else ((y + i) % L, x) for i in range(k)]
        if any(c in owner for c in cells):
            continue
        me = len(parent)
        parent.append(me)
        off.append((0, 0))
        where.append((o, y, x))
        for i, c in enumerate(cells):
            owner[c] = (me, i)
        if n_c is not None:
            continue
        for i, (cy, cx) in enumerate(cells):
            px, py = (i, 0) if o == 0 else (0, i)
            for ex, ey in ((1, 0), (-1, 0), (0, 1), (0, -1)):
                hit = owner.get(((cy + ey) % L, (cx + ex) % L))
                if hit is None:
                    continue
                b, j = hit
                jx, jy = (j, 0) if where[b][0] == 0 else (0, j)
                dx, dy = px + ex - jx, py + ey - jy   # lifted anchor of b from this one's
                if b == me and dx == 0 and dy == 0:
                    continue
                ra, ax, ay = find(me)
                rb, bx, by = find(b)
                dx, dy = ax + dx - bx, ay + dy - by   # root rb from root ra
                if ra == rb:
                    if dx or dy:
                        n_c = me + 1
                else:
                    parent[rb], off[rb] = ra, (dx, dy)   # a node from its parent
    return len(parent), n_c


def exact(case, seed):
    if case["api"] not in ("small", "static", "handle") or 2 * case["L"] ** 2 * case["n"] > 900_000:
        return None
    got = [_sample(case["L"], case["k"], int(s)) for s in _seeds(case, seed)]
    return tuple(np.array(v, dtype=np.int64) for v in zip(*got))
