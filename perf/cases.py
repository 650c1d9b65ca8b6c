"""The work that users of this library have it do, case by case, for timing.

A case is a plain dict. `kind` names the entry point that a user's program calls:

  resident  sbc_count on a graph that is already on the device (one handle, many counts)
  build     sbc_graph_create from a CSR on the device, sbc_count, close: a graph counted once
  host      sbc_count_csr: one call on a host CSR (upload, build, count)
  batch     sbc_count_batch over many resident graphs
  replay    Batch.run: the planned batch, counted again
  serve     Server.submit / wait: a burst of requests over resident graphs
  dynamic   Dynamic.insert / delete / set_sign: a count kept exact under edge updates

Graphs are seeded Chung-Lu graphs of the repository's own workloads (power-law degrees on both
sides, duplicates rejected, ids permuted, planted factions with flipped signs) or dense faction
graphs, drawn on the GPU. Counts are exact 128-bit integers, returned as four 32-bit limbs.
"""
import functools
import math

import numpy as np
import torch

import paper_2605_03603_gb300 as sbc

DEV = "cuda"

# Shapes of the repository's workloads, in edges m: sides n_u and n_v, degree exponents, signs.
SMALL = dict(graph="plain", n_u=2_000, n_v=1_500, m=20_000, gamma_u=2.1, gamma_v=2.1, flip=0.1)
QUARTER = dict(graph="plain", n_u=50_000, n_v=25_000, m=500_000, gamma_u=2.0, gamma_v=2.3, flip=0.15)
MEDIUM = dict(graph="plain", n_u=200_000, n_v=100_000, m=2_000_000, gamma_u=2.0, gamma_v=2.3, flip=0.15)
# A fifth of the 60M-edge benchmark graph (same exponents, hub cap and factions).
LARGE = dict(graph="hubs", n_u=1_000_000, n_v=200_000, m=12_000_000, gamma_u=2.4, gamma_v=1.9,
             cap_v=10_000, flip=0.2)


def listed():
    return [
        # The smallest call: a count on a small resident graph; launches and host waits are all of it.
        dict(SMALL, name="small-33", kind="resident", p=3, q=3),
        # Tuples of five on the same graph: the deep end of the (p,q) grid the paper sweeps.
        dict(SMALL, name="small-55", kind="resident", p=5, q=5),
        # A one-off call on a host CSR of ragged size, p != q, packed signs.
        dict(graph="plain", n_u=20_011, n_v=9_973, m=200_003, gamma_u=2.2, gamma_v=2.2, flip=0.1,
             name="host-200k-34", kind="host", p=3, q=4, bits=True),
        # Signed butterflies, the commonest biclique in use, over a middle-sized graph.
        dict(MEDIUM, name="medium-22", kind="resident", p=2, q=2),
        # A middle-sized graph built from a device CSR and counted once, as the benchmark's step does.
        dict(MEDIUM, name="medium-build-33", kind="build", p=3, q=3, bits=False),
        # Tuples of four on it: the longest single count that such a graph is given.
        dict(MEDIUM, name="medium-44", kind="resident", p=4, q=4),
        # p != q: four from one side and three from the other.
        dict(QUARTER, name="quarter-43", kind="resident", p=4, q=3),
        # The benchmark's graph at a fifth of its size, built and counted, packed signs.
        dict(LARGE, name="large-build-33", kind="build", p=3, q=3, bits=True),
        # A dense block with planted factions: thousands of candidates per anchor.
        dict(graph="dense", n_u=3_000, n_v=800, density=0.45, flip=0.05,
             name="dense-33", kind="resident", p=3, q=3),
        # Many independent graphs of mixed sizes in one call.
        dict(graph="recipe", n=200, m_lo=500, m_hi=500_000, name="batch-200-33", kind="batch", p=3, q=3),
        # A burst of requests of mixed (p,q) on resident graphs of mixed sizes.
        dict(graph="recipe", n=32, m_lo=1_000, m_hi=200_000, name="serve-96", kind="serve", requests=96),
        # Single-edge updates of a middle-sized graph, each with its new count.
        dict(MEDIUM, name="dynamic-33", kind="dynamic", p=3, q=3, updates=12),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _plain(rng, m_lo, m_hi):
    """A plain graph of the small to middle-sized workloads' shape: 6 to 15 edges per vertex of the
    smaller side, exponents between 2.0 and 2.4."""
    m = int(_log(rng, m_lo, m_hi))
    n_v = max(64, int(m / rng.uniform(10, 22)))
    n_u = max(64, int(n_v * rng.uniform(0.7, 2.2)))
    return dict(graph="plain", n_u=n_u, n_v=n_v, m=m, gamma_u=round(rng.uniform(2.0, 2.4), 3),
                gamma_v=round(rng.uniform(2.1, 2.4), 3), flip=round(rng.uniform(0.05, 0.2), 3))


def draw(rng):
    kind = rng.choice(["resident", "resident", "resident", "build", "build", "host", "batch", "replay",
                       "serve", "dynamic"])
    if kind == "resident":
        what = rng.randrange(5)
        if what == 0:  # dense factions
            return dict(graph="dense", n_u=int(_log(rng, 300, 3_000)), n_v=int(_log(rng, 100, 800)),
                        density=round(rng.uniform(0.2, 0.45), 3), flip=round(rng.uniform(0.02, 0.2), 3),
                        kind=kind, p=3, q=rng.randint(3, 5))
        if what == 1:  # deep tuples on small graphs
            p, q = rng.choice([(4, 4), (4, 5), (5, 4), (5, 5), (4, 7), (6, 4)])
            return dict(_plain(rng, 2_000, 20_000), kind=kind, p=p, q=q)
        if what == 2:  # tuples of four
            p, q = rng.choice([(4, 4), (4, 3), (3, 4)])
            return dict(_plain(rng, 10_000, 500_000), kind=kind, p=p, q=q)
        p, q = rng.choice([(2, 2), (2, 3), (2, 5), (3, 3), (3, 3), (3, 4), (3, 6)])
        return dict(_plain(rng, 2_000, 2_000_000), kind=kind, p=p, q=q)
    if kind == "build":
        if rng.random() < 0.3:
            m = int(_log(rng, 1_000_000, 12_000_000))
            return dict(graph="hubs", n_u=m // 12, n_v=m // 60, m=m, gamma_u=2.4, gamma_v=1.9,
                        cap_v=max(500, m // 1200), flip=0.2, kind=kind, p=3, q=3, bits=True)
        p, q = rng.choice([(2, 2), (3, 3), (3, 3), (3, 4)])
        return dict(_plain(rng, 5_000, 2_000_000), kind=kind, p=p, q=q, bits=rng.random() < 0.5)
    if kind == "host":
        p, q = rng.choice([(2, 2), (3, 3), (3, 4), (4, 3)])
        return dict(_plain(rng, 1_000, 400_000), kind=kind, p=p, q=q, bits=rng.random() < 0.5)
    if kind in ("batch", "replay"):
        p, q = rng.choice([(2, 2), (3, 3), (3, 3), (3, 4)])
        return dict(graph="recipe", n=rng.randint(20, 200), m_lo=500, m_hi=int(_log(rng, 10_000, 500_000)),
                    kind=kind, p=p, q=q)
    if kind == "serve":
        return dict(graph="recipe", n=rng.randint(8, 32), m_lo=1_000, m_hi=int(_log(rng, 5_000, 200_000)),
                    kind=kind, requests=rng.randint(16, 96))
    return dict(_plain(rng, 5_000, 2_000_000), kind=kind, p=rng.choice([3, 3, 4]), q=3,
                updates=rng.randint(4, 16))


# ------------------------------------------------------------------ graphs


@functools.lru_cache(maxsize=64)
def _weights(n, m, gamma, cap):
    """Expected degrees (i+1)^(-1/(gamma-1)) scaled to m, at most `cap`, the excess spread over the rest."""
    w = np.arange(1, n + 1, dtype=np.float64) ** (-1.0 / (gamma - 1.0))
    w *= m / w.sum()
    for _ in range(50):
        over = w > cap
        if not over.any() or over.all():
            break
        rest = m - cap * np.count_nonzero(over)
        w[over] = cap
        if rest <= 0:
            break
        w[~over] *= rest / w[~over].sum()
        if not (w > cap * (1 + 1e-9)).any():
            break
    return w


def _ends(c):
    return (_weights(c["n_u"], c["m"], c["gamma_u"], c.get("cap_u", 0.5 * c["n_v"])),
            _weights(c["n_v"], c["m"], c["gamma_v"], c.get("cap_v", 0.5 * c["n_u"])))


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _pick(w, n, gen):
    cum = torch.from_numpy(np.cumsum(w)).to(DEV)
    at = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64) * cum[-1]
    return torch.searchsorted(cum, at, right=True).clamp_(max=len(w) - 1)


def _chung_lu(c, gen):
    """m distinct (u, v) pairs, first draw wins, ids permuted."""
    n_u, n_v, m = c["n_u"], c["n_v"], c["m"]
    wu, wv = _ends(c)
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    want = m + m // 4 + 64
    while True:
        keys = torch.cat([keys, _pick(wu, want, gen) * n_v + _pick(wv, want, gen)])
        s, at = torch.sort(keys, stable=True)
        new = torch.ones_like(s, dtype=torch.bool)
        new[1:] = s[1:] != s[:-1]
        first = at[new]
        if first.numel() >= m:
            keys = keys[torch.sort(first).values[:m]]
            break
        want = 2 * (m - first.numel()) + m // 8 + 64
    u = torch.randperm(n_u, generator=gen, device=DEV)[keys // n_v]
    v = torch.randperm(n_v, generator=gen, device=DEV)[keys % n_v]
    return u, v


def _faction_signs(c, u, v, gen):
    """Planted factions, each sign flipped with probability `flip`: four with a random affinity for the
    hub graphs, two for the others."""
    n_u, n_v, k = c["n_u"], c["n_v"], 4 if c["graph"] == "hubs" else 2
    fu = torch.randint(k, (n_u,), generator=gen, device=DEV)
    fv = torch.randint(k, (n_v,), generator=gen, device=DEV)
    if k == 2:
        s = fu[u] ^ fv[v]
    else:
        s = torch.randint(2, (k * k,), generator=gen, device=DEV)[fu[u] * k + fv[v]]
    flip = torch.rand(u.numel(), generator=gen, device=DEV) < c["flip"]
    return (1 - 2 * (s ^ flip.long())).to(torch.int8)


def _csr(n_u, n_v, u, v, s):
    """CSR over U on the device, rows sorted: (offsets int64, cols int32, signs int8)."""
    key, at = torch.sort(u * n_v + v)
    off = torch.searchsorted(key, torch.arange(n_u + 1, device=DEV, dtype=torch.int64) * n_v)
    return off, (key % n_v).to(torch.int32), s[at]


def _graph(c, seed):
    gen = _generator(seed)
    if c["graph"] == "dense":
        n_u, n_v = c["n_u"], c["n_v"]
        at = torch.nonzero(torch.rand(n_u * n_v, generator=gen, device=DEV) < c["density"]).flatten()
        u, v = at // n_v, at % n_v
    else:
        u, v = _chung_lu(c, gen)
    return _csr(c["n_u"], c["n_v"], u, v, _faction_signs(c, u, v, gen))


def _packed(signs):
    """One bit per edge, set = negative, lowest bit first."""
    n = signs.numel()
    b = torch.zeros((n + 7) // 8 * 8, dtype=torch.uint8, device=DEV)
    b[:n] = (signs < 0).to(torch.uint8)
    shift = torch.arange(8, device=DEV, dtype=torch.uint8)
    return (b.view(-1, 8) << shift).sum(1, dtype=torch.int64).to(torch.uint8)


def _recipe(c, i):
    """Shape of graph i of a batch: edges log-uniform, sides between 1:4 and 4:1, about six edges per
    vertex. The shapes are the case's own; edges and signs come from the seed."""
    r = np.random.RandomState(7919 + i).rand(4)
    m = int(round(c["m_lo"] * (c["m_hi"] / c["m_lo"]) ** r[0]))
    ratio = 0.25 * 16.0 ** r[1]
    both = max(8, math.ceil(m / 6))
    n_u = max(2, round(both * ratio / (1 + ratio)))
    n_v = max(2, both - n_u)
    while n_u * n_v < 2 * m:
        n_u, n_v = n_u + 1, n_v + 1
    gamma = 1.9 + 0.6 * r[2]
    return dict(graph="recipe", n_u=n_u, n_v=n_v, m=m, gamma_u=gamma, gamma_v=gamma, flip=0.3 * r[3])


# ------------------------------------------------------------------ the cases


_MIX = [(3, 3), (3, 4), (4, 4)]  # what a server is asked for


def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    st = {"case": c}
    if c["graph"] == "recipe":
        gs = []
        for i in range(c["n"]):
            r = _recipe(c, i)
            gs.append(sbc.sbc_graph_create(r["n_u"], r["n_v"], *_graph(r, seed * 100_003 + i)))
        st["graphs"] = gs
        if kind == "replay":
            st["batch"] = sbc.Batch(gs, c["p"], c["q"])
        elif kind == "serve":
            # a resident graph has been asked for before: both of its sides are built
            for g in gs:
                for p, q in _MIX:
                    sbc.sbc_count(g, p, q)
            st["server"] = sbc.Server()
            ids = [st["server"].add_graph(g) for g in gs]
            r = np.random.RandomState(seed % (1 << 31))
            st["asked"] = [(ids[int(r.randint(len(ids)))], *_MIX[int(r.randint(3))]) for _ in range(c["requests"])]
        return st
    off, cols, signs = _graph(c, seed)
    if kind == "resident":
        st["g"] = sbc.sbc_graph_create(c["n_u"], c["n_v"], off, cols, signs)
    elif kind == "build":
        st["csr"] = (off, cols, _packed(signs) if c["bits"] else signs)
    elif kind == "host":
        st["csr"] = tuple(x.cpu().numpy() for x in (off, cols, _packed(signs) if c["bits"] else signs))
    else:
        h_off, h_cols, h_signs = (x.cpu().numpy() for x in (off, cols, signs))
        st["dyn"] = sbc.Dynamic(c["n_u"], c["n_v"], h_off, h_cols, h_signs, c["p"], c["q"])
        # new edges (each removed again), edges removed (each put back), and signs turned (and back)
        r = np.random.RandomState(seed % (1 << 31))
        ups = []
        while len(ups) < c["updates"]:
            e = int(r.randint(c["m"]))
            u = int(np.searchsorted(h_off, e, side="right")) - 1
            if len(ups) % 3 == 0:
                v = int(h_cols[r.randint(c["m"])])  # a column as often as it has edges
                row = h_cols[h_off[u]:h_off[u + 1]]
                if v not in row and (u, v) not in {(x[1], x[2]) for x in ups}:
                    ups.append(("insert", u, v, 1 if r.rand() < 0.7 else -1))
            else:
                ups.append(("delete" if len(ups) % 3 == 1 else "turn", u, int(h_cols[e]), int(h_signs[e])))
        st["updates"] = ups
    return st


def _limbs(counts):
    return np.array([[(n >> s) & 0xFFFFFFFF for s in (0, 32, 64, 96)] for n in counts], dtype=np.int64)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "resident":
        return _limbs([sbc.sbc_count(state["g"], c["p"], c["q"])])
    if kind == "build":
        off, cols, signs = state["csr"]
        with sbc.sbc_graph_create(c["n_u"], c["n_v"], off, cols, signs, sign_bits=c["bits"]) as g:
            return _limbs([sbc.sbc_count(g, c["p"], c["q"])])
    if kind == "host":
        off, cols, signs = state["csr"]
        return _limbs([sbc.sbc_count_csr(c["n_u"], c["n_v"], off, cols, signs, c["p"], c["q"], sign_bits=c["bits"])])
    if kind == "batch":
        return _limbs(sbc.sbc_count_batch(state["graphs"], c["p"], c["q"]))
    if kind == "replay":
        return _limbs(state["batch"].run())
    if kind == "serve":
        tickets = [state["server"].submit(gid, p, q) for gid, p, q in state["asked"]]
        return _limbs([state["server"].wait(t)[0] for t in tickets])
    d, counts = state["dyn"], []
    for op, u, v, s in state["updates"]:
        if op == "insert":
            counts += [d.insert(u, v, s), d.delete(u, v)]
        elif op == "delete":
            counts += [d.delete(u, v), d.insert(u, v, s)]
        else:
            counts += [d.set_sign(u, v, -s), d.set_sign(u, v, s)]
    return _limbs(counts)


# ------------------------------------------------------------------ what a pass cannot do without


def _graph_work(c):
    """(bytes of the CSR, 2-paths of the cheaper side) of a graph of this shape, from its expected
    degrees: every count reads the edges and looks at each pair of edges that share a vertex."""
    if c["graph"] == "dense":
        m = c["n_u"] * c["n_v"] * c["density"]
        paths = min(c["n_u"] * (c["n_v"] * c["density"]) ** 2, c["n_v"] * (c["n_u"] * c["density"]) ** 2) / 2
    else:
        m = c["m"]
        paths = min(float(np.sum(w * w)) / 2 for w in _ends(c))
    return 8 * (c["n_u"] + 1) + m * (4 + (0.125 if c.get("bits") else 1)), paths


def work(case):
    if case["graph"] == "recipe":
        each = [_graph_work(_recipe(case, i)) for i in range(case["n"])]
        times = case["requests"] / case["n"] if case["kind"] == "serve" else 1.0
        out = 16 * (case["requests"] if case["kind"] == "serve" else case["n"])
        return {"bytes": times * sum(b for b, _ in each) + out, "flops": times * sum(p for _, p in each)}
    b, paths = _graph_work(case)
    if case["kind"] == "dynamic":
        # an update reads the lists of its edge's two ends and of their neighbours: on average, over the
        # edges, the 2-paths per edge
        each = 2 * case["updates"] * paths / case["m"]
        return {"bytes": 5 * each + 32 * case["updates"], "flops": each}
    return {"bytes": b + 16, "flops": paths}


# ------------------------------------------------------------------ values from plain torch


def _binom(n, k):
    r = torch.ones_like(n)
    for i in range(k):
        r = r * (n - i) // (i + 1)
    return torch.where(n >= k, r, torch.zeros_like(r))


def exact(case, seed):
    """Pairs and triples of rows over a dense sign matrix, in 64 bits; None where that is too much."""
    if case["graph"] == "recipe" or case["kind"] == "dynamic" or case["p"] not in (2, 3):
        return None
    n_u, n_v, p, q = case["n_u"], case["n_v"], case["p"], case["q"]
    if n_u * n_v > 4_000_000:
        return None
    off, cols, signs = _graph(case, seed)
    A = torch.zeros(n_u, n_v, dtype=torch.float64, device=DEV)
    rows = torch.repeat_interleave(torch.arange(n_u, device=DEV), off[1:] - off[:-1])
    A[rows, cols.long()] = signs.double()
    total = 0
    for u in range(n_u):
        at = torch.nonzero(A[u]).flatten()
        if at.numel() < q:
            continue
        rel = A[u + 1:, at] * A[u, at]  # +1 same sign as u, -1 the other, 0 no edge
        same, other = (rel > 0).double(), (rel < 0).double()
        if p == 2:
            total += int(sum(_binom(x.sum(1).long(), q).sum() for x in (same, other)))
            continue
        keep = (same.sum(1) >= q) | (other.sum(1) >= q)
        same, other = same[keep], other[keep]
        for x in (same, other):
            for y in (same, other):
                total += int(torch.triu(_binom((x @ y.T).round().long(), q), 1).sum())
    return _limbs([total])
