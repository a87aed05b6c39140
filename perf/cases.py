"""Performance cases of the PLDS library: what is timed, on which inputs, and how close
two correct builds must agree.

Every case goes through the Python binding (``paper_2106_03824_gb300.plds``).  Four forms
of use, each over the graph shapes and batch sizes of the repository's own workloads:

  window  a graph kept up to date under a sliding window over an edge stream: each pass
          inserts the next batch, deletes the oldest one and reads the result
  cycle   the Ins/Del protocol: all edges inserted from empty in batches, the result read,
          all edges deleted in another order (read again half-way), back to empty
  serve   a request server on a loaded graph: uneven batches and coreness queries,
          request boundaries unchanged (results do not depend on timing)
  set     many independent graphs, one mixed round for all of them in one call
  query   reads of a loaded graph: estimates, orientation, static approximate k-core

Levels, counters and work counts are integers and the estimates are copies of one table
of doubles, so two correct builds agree bit for bit.
"""
import math
from fractions import Fraction

import numpy as np
import torch

from paper_2106_03824_gb300 import plds as P

DEV = "cuda"
LOAD_BATCH = 1_000_000  # edges per call when a state's graph is loaded


def listed():
    return [
        # a monitoring loop at its smallest: a handful of edges per call from host arrays,
        # the estimates of a small graph read back every time; only latency counts
        dict(name="cl10k_window_10", form="window", graph="chunglu", n=10_000, m=50_000, gamma=2.5, batch=10, host=True),
        # the small plain configuration: 50 insertion batches of 1,000 edges, then deletions
        dict(name="cl10k_cycle_1000", form="cycle", graph="chunglu", n=10_000, m=50_000, gamma=2.5, batch=1_000, host=True),
        # an ordinary update stream on a mid-size graph, odd batch size, device-resident edges
        dict(name="rmat17_window_9973", form="window", graph="rmat", n=1 << 17, m=16 << 17, gamma=0.0, batch=9_973, host=False),
        # the medium plain configuration's smaller batches
        dict(name="rmat18_cycle_1e5", form="cycle", graph="rmat", n=1 << 18, m=16 << 18, gamma=0.0, batch=100_000, host=False),
        # the headline protocol: R-MAT scale 20, batches of 10^6
        dict(name="rmat20_cycle_1e6", form="cycle", graph="rmat", n=1 << 20, m=16 << 20, gamma=0.0, batch=1_000_000, host=False),
        # the Mix protocol: half a million insertions and as many deletions on a 90 % load
        dict(name="rmat20_window_5e5", form="window", graph="rmat", n=1 << 20, m=16 << 20, gamma=0.0, batch=500_000, host=False),
        # the optimised variant's group size (few levels per group), a ragged batch size
        dict(name="rmat19_opt_cycle_300007", form="cycle", graph="rmat", n=1 << 19, m=16 << 19, gamma=0.0, batch=300_007, host=False, opt=True),
        # the road-like contrast: low degrees, tiny cores, long chains of moves
        dict(name="grid1201_cycle_250007", form="cycle", graph="grid", n=1201 * 1201, m=0, gamma=0.0, batch=250_007, host=False),
        # serving: requests of 10 to 300,000 edges on a social-network-shaped graph
        dict(name="cl1m_serve_48", form="serve", graph="chunglu", n=1_200_000, m=10_750_000, gamma=2.2, batch=300_000, requests=48),
        # the batched form: independent graphs, each with a mixed batch of 1-10 % of its edges
        dict(name="set128_round", form="set", graph="chunglu", graphs=128, n=100_000, m=0, gamma=0.0, batch=0),
        # reads: estimates, out-degrees, edge orientation, static approximate k-core
        dict(name="rmat19_query", form="query", graph="rmat", n=1 << 19, m=16 << 19, gamma=0.0, batch=200_000, host=False),
        # a graph well beyond the L2, batches of millions
        dict(name="cl4m8_window_4e6", form="window", graph="chunglu", n=4_800_000, m=43_000_000, gamma=2.2, batch=4_000_000, host=False),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["window", "window", "window", "cycle", "cycle", "serve", "set", "query"])
    if form == "set":
        return dict(form="set", graph="chunglu", graphs=rng.randint(8, 128), n=_logint(rng, 5_000, 100_000), m=0,
                    gamma=0.0, batch=0)
    if form == "serve":
        n = _logint(rng, 20_000, 1_200_000)
        m = int(n * rng.uniform(2.0, 9.0))
        return dict(form="serve", graph="chunglu", n=n, m=m, gamma=round(rng.uniform(2.1, 2.8), 3),
                    batch=max(100, min(300_000, m // 30)), requests=rng.randint(12, 48))
    kind = rng.choice(["chunglu", "chunglu", "rmat", "grid"])
    top = 4_800_000 if form == "window" else 1_000_000
    if kind == "rmat":
        s = rng.randint(12, 20 if form == "window" else 19)
        n, m, gamma = 1 << s, 16 << s, 0.0
    elif kind == "grid":
        side = _logint(rng, 40, 1201)
        n, m, gamma = side * side, 0, 0.0
    else:
        n = _logint(rng, 3_000, top)
        m, gamma = int(n * rng.uniform(2.0, 9.0)), round(rng.uniform(2.1, 2.8), 3)
    edges = m or 2 * n
    case = dict(form=form, graph=kind, n=n, m=m, gamma=gamma, host=rng.random() < 0.3)
    if form == "window":
        case["batch"] = _logint(rng, 1, max(2, edges // 10))
    elif form == "cycle":  # 4 to 60 batches
        case["batch"] = max(1, edges // rng.randint(4, 60))
        case["opt"] = rng.random() < 0.3
    else:
        case["batch"] = _logint(rng, 1, 200_000)
    return case


# ---------------------------------------------------------------------------
# Inputs, made on the GPU from the seed: integer arithmetic wherever the order of a
# parallel sum could show, so that a seed always gives the same edges.
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _perm(k, gen):
    return torch.argsort(torch.randint(0, 1 << 62, (k,), device=DEV, generator=gen), stable=True)


def _distinct(u, v, n, gen, m=0):
    """Distinct undirected edges of the drawn pairs, ids permuted, in random order
    (at most m of them where m is given)."""
    u, v = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.unique((u * n + v)[u != v])
    key = key[_perm(key.numel(), gen)]
    key = key[:m] if m else key
    ids = _perm(n, gen)
    e = torch.stack([ids[key // n], ids[key % n]], 1)
    return e.to(torch.int32).contiguous()


def _rmat(n, m, gen):
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros_like(u)
    for _ in range(n.bit_length() - 1):
        r = torch.rand(m, device=DEV, generator=gen)
        u = (u << 1) | (r >= 0.76)
        v = (v << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return _distinct(u, v, n, gen)


def _chunglu(n, m, gamma, gen):
    """Endpoints drawn proportional to (i+1)^(-1/(gamma-1)), cut at sqrt(2m)."""
    w = torch.arange(1, n + 1, dtype=torch.float64).pow(-1.0 / (gamma - 1.0))
    for _ in range(8):
        w = (w * (2.0 * m / w.sum())).clamp(max=math.sqrt(2.0 * m))
    cw = torch.cumsum((w * (float(1 << 40) / w.sum())).to(torch.int64), 0).to(DEV)
    k = int(1.3 * m) + 64
    total = int(cw[-1])
    u, v = (torch.searchsorted(cw, torch.randint(0, total, (k,), device=DEV, generator=gen), right=True)
            for _ in range(2))
    return _distinct(u, v, n, gen, m)


def _grid(n, gen):
    """A square lattice with a random diagonal in a tenth of its cells."""
    side = math.isqrt(n)
    i = torch.arange(side * side, device=DEV).view(side, side)
    cells = i[:-1, 1:-1].reshape(-1)
    pick = cells[torch.rand(cells.numel(), device=DEV, generator=gen) < 0.1]
    sign = torch.randint(0, 2, (pick.numel(),), device=DEV, generator=gen) * 2 - 1
    u = torch.cat([i[:, :-1].reshape(-1), i[:-1, :].reshape(-1), pick])
    v = torch.cat([i[:, 1:].reshape(-1), i[1:, :].reshape(-1), pick + side + sign])
    return _distinct(u, v, side * side, gen)


def _edges(case, gen):
    if case["graph"] == "rmat":
        return _rmat(case["n"], case["m"], gen)
    if case["graph"] == "grid":
        return _grid(case["n"], gen)
    return _chunglu(case["n"], case["m"], case["gamma"], gen)


def _group(case):
    """Levels per group of the optimised variant: the smallest L with 1.4^(50 L) >= m."""
    m, lg = case["m"] or 2 * case["n"], 1
    while Fraction(7, 5) ** (50 * lg) < m:
        lg += 1
    return lg if case.get("opt") else 0


def _handle(case):
    return P.PLDS(case["n"], levels_per_group=_group(case))


def _load(g, e):
    for s in range(0, e.shape[0], LOAD_BATCH):
        g.insert(e[s:s + LOAD_BATCH].contiguous())


def _chunks(e, b, host):
    e = e.cpu().numpy() if host else e
    return [e[s:s + b] for s in range(0, e.shape[0], b)]


def _ints(n, k):
    return [torch.zeros(n, dtype=torch.int32, device=DEV) for _ in range(k)]


class _Window:
    def __init__(self, case, seed):
        self.host = case["host"]
        e = _edges(case, _gen(seed))
        self.ring = _chunks(e, case["batch"], self.host)
        self.held = max(1, min(len(self.ring) - 1, int(0.9 * len(self.ring))))
        self.g = _handle(case)
        _load(self.g, e[:self.held * case["batch"]])
        self.k = 0
        self.levels = _ints(case["n"], 1)[0]
        self.counters = _ints(case["n"], 3)

    def run(self):
        c, k = len(self.ring), self.k
        self.k += 1
        self.g.insert(self.ring[(self.held + k) % c])
        self.g.delete(self.ring[k % c])
        if self.host:  # a host program: estimates to a host array
            return {"coreness": self.g.coreness()}
        self.g.levels(self.levels)
        self.g.counters(self.counters)
        return {"levels": self.levels, "counters": list(self.counters)}


class _Cycle:
    def __init__(self, case, seed):
        gen = _gen(seed)
        e = _edges(case, gen)
        self.ins = _chunks(e, case["batch"], case["host"])
        self.dele = _chunks(e[_perm(e.shape[0], gen)].contiguous(), case["batch"], case["host"])
        self.g = _handle(case)
        self.full, self.half = _ints(case["n"], 2)
        self.counters = _ints(case["n"], 3)
        self.coreness = torch.zeros(case["n"], dtype=torch.float64, device=DEV)

    def run(self):
        for b in self.ins:
            self.g.insert(b)
        self.g.levels(self.full)
        self.g.counters(self.counters)
        self.g.coreness(self.coreness)
        mid = len(self.dele) // 2
        for k, b in enumerate(self.dele):
            if k == mid:
                self.g.levels(self.half)
            self.g.delete(b)
        return {"levels": self.full, "counters": list(self.counters), "coreness": self.coreness, "half": self.half}


class _Serve:
    """Two halves of the request ring take turns: what one pass inserts, the next deletes."""

    def __init__(self, case, seed):
        e = _edges(case, _gen(seed))
        rs = np.random.RandomState(seed % (1 << 31))
        self.pairs = max(1, case["requests"] // 2)
        sizes = np.exp(rs.uniform(math.log(10), math.log(case["batch"]), 2 * self.pairs)).astype(int)
        sizes = np.minimum(sizes, e.shape[0] // (4 * self.pairs))
        cut = np.concatenate([[0], np.cumsum(sizes)])
        h = e[:int(cut[-1])].cpu()
        req = [h[cut[i]:cut[i + 1]].contiguous().pin_memory() for i in range(2 * self.pairs)]
        self.sides = [req[:self.pairs], req[self.pairs:]]
        self.g = _handle(case)
        _load(self.g, e[int(cut[self.pairs]):].contiguous())  # side 1 is in, side 0 is out
        self.out = [torch.zeros(case["n"], dtype=torch.float64, device=DEV) for _ in range(2)]
        torch.cuda.synchronize()
        self.server = P.Server(self.g, slots=16, max_batch=int(max(sizes)), merge_max_edges=0)
        self.k = 0

    def run(self):
        ins, dele = self.sides if self.k % 2 == 0 else self.sides[::-1]
        self.k += 1
        s = self.server
        for i in range(self.pairs):
            s.submit(s.INSERT, ins[i])
            s.submit(s.DELETE, dele[i])
            if i == self.pairs // 2:
                s.submit(s.CORENESS, out=self.out[0])
        s.submit(s.CORENESS, out=self.out[1])
        s.drain()
        done = s.poll()
        return {"coreness": list(self.out),
                "done": np.array([[r["op"], r["status"], r["valid"], r["rounds"], r["moves"]] for r in done], np.int64)}


class _Set:
    """A ring of 16 mixed rounds per graph over half of its edges; the other half stays."""
    RING = 16

    def __init__(self, case, seed):
        gen, rs = _gen(seed), np.random.RandomState(seed % (1 << 31))
        lo = min(1_000, case["n"])  # the graphs' sizes belong to the case, their edges to the seed
        ns = np.random.RandomState(7).uniform(math.log(lo), math.log(case["n"]), case["graphs"])
        ns = np.exp(ns).astype(int)
        gammas, degs, fracs = (rs.uniform(a, b, case["graphs"]) for a, b in ((2.1, 2.8), (4, 32), (0.01, 0.1)))
        r = self.RING
        base, ring = [], []
        for n, ga, d, f in zip(ns, gammas, degs, fracs):
            e = _chunglu(int(n), int(n * d / 2), float(ga), gen)
            b = max(1, min(int(f * e.shape[0]), e.shape[0] // (r + 2)))
            ring.append([e[i * b:(i + 1) * b] for i in range(r)])
            base.append(e[r * b:])
        self.s = P.PLDSSet([int(n) for n in ns])
        none = base[0][:0]
        self._update([(torch.cat([x] + c[:r // 2]), none) for x, c in zip(base, ring)])
        self.rounds = [self._pack([(c[(r // 2 + k) % r], c[k]) for c in ring]) for k in range(r)]
        self.levels = _ints(int(ns.sum()), 1)[0]
        self.views = list(torch.split(self.levels, [int(n) for n in ns]))
        self.k = 0

    @staticmethod
    def _pack(halves):
        flat = [h for pair in halves for h in pair]
        off = np.concatenate([[0], np.cumsum([h.shape[0] for h in flat])]).astype(np.int64)
        return torch.cat(flat).contiguous(), off

    def _update(self, halves):
        self.s.update(*self._pack(halves))

    def run(self):
        self.s.update(*self.rounds[self.k % self.RING])
        self.k += 1
        for g, out in zip(self.s.graphs, self.views):
            g.levels(out)
        return {"levels": self.levels}


class _Query:
    def __init__(self, case, seed):
        gen = _gen(seed)
        e = _edges(case, gen)
        self.g = _handle(case)
        _load(self.g, e)
        q = e[torch.randint(0, e.shape[0], (case["batch"],), device=DEV, generator=gen)]
        odd = torch.rand(case["batch"], device=DEV, generator=gen) < 0.3  # some absent ones
        q[:, 1] = torch.where(odd, (q[:, 1] + 1) % case["n"], q[:, 1])
        self.q = q.cpu().numpy() if case["host"] else q.contiguous()
        self.est = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
        self.static = torch.zeros_like(self.est)

    def run(self):
        self.g.coreness(self.est)
        tails = self.g.orient(self.q)
        out = self.g.out_degrees()
        _, st = self.g.static_coreness(1.0, self.static)
        return {"coreness": self.est, "tails": tails, "out_degrees": out, "static": self.static,
                "iterations": [st["outer"], st["inner"], st["visits"]]}


_FORMS = dict(window=_Window, cycle=_Cycle, serve=_Serve, set=_Set, query=_Query)


def prepare(case, seed):
    return _FORMS[case["form"]](case, seed)


def run(state):
    return state.run()


# ---------------------------------------------------------------------------
# What a pass cannot do without: 8 bytes per submitted edge; per applied update a probe
# and a slot write in each endpoint's table (4 bytes each) and three counters of each
# endpoint read and written (8 bytes each); the results.
# ---------------------------------------------------------------------------
PER_UPDATE = 8 + 64


def work(case):
    n = case["n"]
    m = case["m"] or int(2.1 * n)
    if case["form"] == "window":
        b = 2 * PER_UPDATE * min(case["batch"], m)
        return {"bytes": b + (8 if case["host"] else 16) * n, "flops": 0}
    if case["form"] == "cycle":
        return {"bytes": 2 * PER_UPDATE * m + 28 * n, "flops": 0}
    if case["form"] == "serve":  # log-uniform sizes: mean (b - 10) / ln(b / 10)
        mean = (case["batch"] - 10) / math.log(case["batch"] / 10)
        return {"bytes": case["requests"] * mean * PER_UPDATE + 16 * n, "flops": 0}
    if case["form"] == "set":  # n log-uniform from 1,000, degree 18 and 5.5 % on average
        lo = min(1_000, n)
        verts = case["graphs"] * ((n - lo) / math.log(n / lo) if n > lo else n)
        return {"bytes": 2 * 0.055 * 9 * verts * PER_UPDATE + 4 * verts, "flops": 0}
    # each adjacency read by the out-degrees and by the static k-core, a level or a bucket with it
    return {"bytes": 4 * m * 8 + case["batch"] * 12 + 20 * n, "flops": 0}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------------------
# The same results in plain torch: every round recounts every vertex's neighbours from
# the edge list, in 64-bit integers and doubles.
# ---------------------------------------------------------------------------
class _Plain:
    def __init__(self, n, lg=0):
        t, p = 1, Fraction(7, 5)
        while p < n:
            t, p = t + 1, p * Fraction(7, 5)
        self.n, self.lg, self.t = n, lg or 4 * t, t
        pw = [Fraction(7, 5) ** i for i in range(t + 1)]
        up = [min(math.floor(3 * x), n) for x in pw]
        dn = [min(math.ceil(x), n) for x in pw]
        self.up, self.dn = torch.tensor(up, device=DEV), torch.tensor(dn, device=DEV)
        self.level = torch.zeros(n, dtype=torch.int64, device=DEV)
        self.keys = torch.zeros(0, dtype=torch.int64, device=DEV)

    def _key(self, e):
        e = torch.as_tensor(e).to(DEV).long()
        return torch.unique(e.min(1).values * self.n + e.max(1).values)

    def _ends(self):
        u, v = self.keys // self.n, self.keys % self.n
        return torch.cat([u, v]), torch.cat([v, u])

    def _count(self, at, sel):
        return torch.bincount(at[sel], minlength=self.n)

    def insert(self, e):
        self.keys = torch.unique(torch.cat([self.keys, self._key(e)]))
        a, b = self._ends()
        while True:
            lv = self.level
            bad = self._count(a, lv[b] >= lv[a]) > self.up[lv // self.lg]
            if not bool(bad.any()):
                return
            low = lv[bad].min()
            self.level = lv + (bad & (lv == low)).long()

    def delete(self, e):
        self.keys = self.keys[~torch.isin(self.keys, self._key(e))]
        a, b = self._ends()
        while True:
            lv = self.level
            star = self._count(a, lv[b] >= lv[a] - 1)
            bad = (lv > 0) & (star < self.dn[(lv - 1).clamp(min=0) // self.lg])
            if not bool(bad.any()):
                return
            # the largest x <= level - 2 with enough neighbours on x or above, by halving
            sel = bad[a]
            sa, sb = a[sel], b[sel]
            lo, hi = torch.full_like(lv, -1), (lv - 1).clamp(min=0)
            while bool((bad & (hi - lo > 1)).any()):
                mid = (lo + hi) // 2
                fits = self._count(sa, lv[sb] >= mid[sa]) >= self.dn[mid.clamp(min=0) // self.lg]
                wide = hi - lo > 1
                lo, hi = torch.where(wide & fits, mid, lo), torch.where(wide & ~fits, mid, hi)
            want = lo + 1
            low = want[bad].min()
            self.level = torch.where(bad & (want == low), want, lv)

    def coreness(self):
        a, _ = self._ends()
        deg = torch.bincount(a, minlength=self.n)
        k = ((self.level + 1) // self.lg - 1).clamp(min=0)
        return torch.where(deg > 0, torch.pow(1.4, k.double()), torch.zeros((), dtype=torch.float64, device=DEV))


def _plain_static(n, e, eps_prime):
    """The static approximate k-core by bucketed peeling, the whole graph at every step."""
    eps = (math.sqrt(4 * eps_prime + 9) - 3) / 2
    rounds = max(1, math.ceil(math.log(n) / math.log(1 + 2 / eps)))
    thr = [1.0]
    while thr[-1] < n:
        thr.append(thr[-1] * (1 + eps))
    tab = torch.tensor(thr, dtype=torch.float64, device=DEV)
    a, b = torch.cat([e[:, 0], e[:, 1]]).long(), torch.cat([e[:, 1], e[:, 0]]).long()
    c = torch.bincount(a, minlength=n)
    est = torch.zeros(n, dtype=torch.float64, device=DEV)
    alive = c > 0
    bucket = torch.searchsorted(tab, c.double())
    t = cur = int(bucket[alive].min()) if bool(alive.any()) else 0
    j = 0
    while bool(alive.any()):
        peel = alive & (bucket == cur)
        est[peel] = thr[cur]
        alive &= ~peel
        lost = torch.bincount(b[peel[a]], minlength=n)
        hit = alive & (lost > 0)
        c = torch.where(hit, (c - lost).clamp(min=math.ceil(thr[t - 1]) if t else 1), c)
        bucket = torch.where(hit, torch.searchsorted(tab, c.double()).clamp(min=t), bucket)
        if not bool(alive.any()):
            break
        cur = int(bucket[alive].min())
        if j + 1 < rounds and thr[cur] <= (2 + eps) * thr[t]:
            j += 1
        else:
            t, j = cur, 0
    return est


def exact(case, seed):
    if case["form"] == "query":
        return {"static": _plain_static(case["n"], _edges(case, _gen(seed)), 1.0)}
    edges = case["m"] or 2 * case["n"]
    if case["form"] == "window" and case["host"] and edges <= 120_000:
        e = _edges(case, _gen(seed))
        x = _Plain(case["n"])
        ring = _chunks(e, case["batch"], False)
        held = max(1, min(len(ring) - 1, int(0.9 * len(ring))))
        _load(x, e[:held * case["batch"]])
        x.insert(ring[held % len(ring)])
        x.delete(ring[0])
        return {"coreness": x.coreness()}
    if case["form"] == "cycle" and edges <= 60_000:
        x = _Plain(case["n"], _group(case))
        for b in _chunks(_edges(case, _gen(seed)), case["batch"], False):
            x.insert(b)
        return {"coreness": x.coreness()}
    return None
