"""The ways a batch's level phases are spread over the GPU, against the CPU oracle.

A phase is run by one block alone (small lists), by the whole grid, or (batched form)
by a block or a cluster of blocks; a batch passes from one to another as its lists
grow and shrink.  Every quantity is an integer decided by exact arithmetic, so levels,
counters and work counts must equal the oracle's after every batch.
"""
import time

import numpy as np
import pytest

from oracle import oracle as O
from paper_2106_03824_gb300 import workloads as W
from test_gpu_parity import P, assert_same, assert_stats  # noqa: F401

pytestmark = pytest.mark.gpu


def _star_and_core(n, seed):
    """Two hubs joined to half of the vertices each (tables of many chunks) over a random graph."""
    rng = np.random.default_rng(seed)
    leaves = rng.permutation(np.arange(2, n))[: n // 2]
    hubs = np.stack([np.arange(leaves.size) % 2, leaves], 1)
    e = np.concatenate([hubs, W.erdos_renyi(n, 4 * n, seed)]).astype(np.int32)
    e = np.unique(np.sort(e, axis=1), axis=0)
    return e[rng.permutation(e.shape[0])]


GRAPHS = {
    "power": lambda: (6_000, W.shuffled(W.chung_lu(6_000, 45_000, 2.2, seed=3), 4)),
    "hubs": lambda: (5_000, _star_and_core(5_000, 5)),
    "grid": lambda: (70 * 70, W.shuffled(W.grid2d(70, 0.1, seed=2), 6)),
    "clique": lambda: (300, W.shuffled(W.erdos_renyi(300, 40_000, seed=8), 9)),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("sizes", [(1, 2, 31, 33, 257, 1000), (20_000, 1, 500, 7, 4_000), (513,)])
def test_batches_of_uneven_size(P, name, sizes):  # noqa: F811
    """Insertions from empty and deletions back, the batch sizes of `sizes` in turn
    (at most 40 batches each way, the rest in one)."""
    n, e = GRAPHS[name]()
    g, o = P.PLDS(n), O.OraclePLDS(n)
    for op in ("insert", "delete"):
        rest = e if op == "insert" else W.shuffled(e, 17)
        k = 0
        while rest.shape[0]:
            b = sizes[k % len(sizes)] if k < 40 else rest.shape[0]
            part, rest = np.ascontiguousarray(rest[:b]), rest[b:]
            getattr(g, op)(part)
            assert getattr(o, op)(part) == 0
            assert_same(g, o, f"{op} {k}")
            assert_stats(g, o, f"{op} {k}")
            k += 1
    assert int(g.levels().max()) == 0
    g.close()


@pytest.mark.parametrize("list_cap", [4, 8, 16, 32, 33])
@pytest.mark.parametrize("graph", ["rmat", "power"])
def test_short_up_lists_with_the_cutoff_by_phase(P, graph, list_cap):  # noqa: F811
    """A climbing vertex scanned by a thread in one phase and, the next phase's cutoff being
    lower, by a warp in the next gets an up-list when its table has list_cap slots: the list
    needs room for its up-degree (it had none, and lists overwrote one another)."""
    if graph == "rmat":
        n, e = 1_024, W.shuffled(W.rmat(10, 12, seed=488236076), 2)
    else:
        n, e = GRAPHS["power"]()
    g, o = P.PLDS(n, delta=0.2), O.OraclePLDS(n, delta=0.2)
    g.set_tuning(list_cap=list_cap)
    sizes = [2_887, 39, 362, 14, 3_074]
    at = 0
    for k, b in enumerate(sizes + [e.shape[0] - sum(sizes)]):
        part = np.ascontiguousarray(e[at: at + b])
        at += b
        g.insert(part)
        assert o.insert(part) == 0
        assert_same(g, o, f"batch {k}")
        assert_stats(g, o, f"batch {k}")
        if k == 1:
            back = np.ascontiguousarray(e[: at: 50])
            for x in (g, o):
                x.delete(back)
                x.insert(back)
            assert_same(g, o, "put back")
    g.close()


def test_deletions_with_a_narrowed_window(P):  # noqa: F811
    """Deletion batches of a road-like graph that leave more than 4,096 vertices pending over
    many levels: the near window is narrowed, the rest is sent to the far list and comes back
    refill by refill.  By the grid, and by a cluster (a set of one graph)."""
    side = 600
    n = side * side
    e = W.shuffled(W.grid2d(side, 0.1, seed=3), 4)
    dele = W.shuffled(e, 9)
    g, S, o = P.PLDS(n), P.PLDSSet([n]), O.OraclePLDS(n)
    g.set_tuning(trace_rounds=1)
    g.insert(e)
    S.update(*S.pack([(e, e[:0])]))
    assert o.insert(e) == 0
    assert_same(g, o, "loaded")
    m = e.shape[0]
    narrowed = refilled = 0
    for a, b in ((0, 0.3), (0.3, 0.6), (0.6, 0.8)):
        part = np.ascontiguousarray(dele[int(a * m): int(b * m)])
        g.delete(part)
        S.update(*S.pack([(part[:0], part)]))
        assert o.delete(part) == 0
        assert_same(g, o, f"deleted to {b}")
        assert_stats(g, o, f"deleted to {b}")
        assert_same(S.graphs[0], o, f"set, deleted to {b}")
        t = g.trace()[1:]
        near, movers = t[:, 1].astype(int), t[:, 2].astype(int)
        left = near[:-1] - movers[:-1]  # near entries that did not move in a round
        narrowed += int(((near[:-1] > 4096) & (left - near[1:] > near[:-1] // 2)).sum())
        refilled += int((near[1:] - left > 64).sum())
    assert narrowed >= 2 and refilled >= 4, (narrowed, refilled)
    g.close()
    S.close()


@pytest.mark.parametrize("ns", [(9_000,), (1, 2, 9_000, 40, 700), (4_000,) * 3 + (100,) * 60])
def test_set_of_uneven_graphs(P, ns):  # noqa: F811
    """A round's largest graphs go to clusters, the others to blocks: each equals the oracle."""
    rng = np.random.default_rng(1)
    edges = [W.shuffled(W.chung_lu(n, 9 * n, 2.3, seed=n), 1) if n > 2 else np.zeros((0, 2), np.int32) for n in ns]
    S, orc = P.PLDSSet(list(ns)), [O.OraclePLDS(n) for n in ns]
    for r in range(3):
        halves = []
        for e in edges:
            m = e.shape[0]
            ins = e[: int(m * (0.5, 0.8, 1.0)[r])]
            dele = e[rng.permutation(m)[: m // 6]]
            halves.append((ins, dele))
        S.update(*S.pack(halves))
        for g, o, (ins, dele) in zip(S.graphs, orc, halves):
            assert o.insert(ins) == 0 and o.delete(dele) == 0
            assert_same(g, o, f"round {r}, n={g.n}")
    S.close()


def _round_seconds(P, count):  # noqa: F811
    """Best wall time of a round of 20 insertions and 20 deletions in each of `count` graphs alike."""
    n, b = 300, 20
    es = [W.shuffled(W.chung_lu(n, 6 * n, 2.4, seed=7 + i % 8), i) for i in range(count)]
    S = P.PLDSSet([n] * count)
    S.update(*S.pack([(e[b:], e[:0]) for e in es]))
    turns = [S.pack([(e[:b], e[b:2 * b]) for e in es]), S.pack([(e[b:2 * b], e[:b]) for e in es])]
    best = float("inf")
    for _ in range(8):
        t0 = time.perf_counter()
        for t in turns:
            S.update(*t)
        best = min(best, time.perf_counter() - t0)
    o = O.OraclePLDS(n)
    for ins, dele in [(es[-1][b:], es[-1][:0])] + 8 * [(es[-1][:b], es[-1][b:2 * b]), (es[-1][b:2 * b], es[-1][:b])]:
        assert o.insert(ins) == 0 and o.delete(dele) == 0
    assert_same(S.graphs[-1], o, f"{count} graphs")
    S.close()
    return best


def test_small_graphs_alike_are_not_queued_for_clusters(P):  # noqa: F811
    """300 small graphs of one size fit one block each: a round of them takes no longer than
    one of 600 (queued for clusters, eight of them one after another, it took 2.4 times as long; now 0.6 times)."""
    assert _round_seconds(P, 300) < 1.4 * _round_seconds(P, 600)


@pytest.mark.parametrize("op", ["insert", "delete"])
@pytest.mark.parametrize("size", [100, 20_000])
def test_rejected_batch_leaves_no_trace(P, op, size):  # noqa: F811
    """A batch with an id out of range (run in one launch or as step kernels) is rejected
    whole: the per-vertex counts of its valid edges do not reach the next batch."""
    n, e = GRAPHS["power"]()
    g, o = P.PLDS(n), O.OraclePLDS(n)
    first = e[:25_000]
    g.insert(first)
    assert o.insert(first) == 0
    bad = np.concatenate([(e[25_000:] if op == "insert" else first)[:size], [[0, n]]]).astype(np.int32)
    assert getattr(g, op)(bad, check=False) == -1
    assert_same(g, o, "after the rejected batch")
    for what, part in ((op, bad[:-1]), ("insert", e[:30_000]), ("delete", e[10_000:12_000])):
        getattr(g, what)(part)
        assert getattr(o, what)(part) == 0
        assert_same(g, o, what)
        assert_stats(g, o, what)
    g.close()


@pytest.mark.parametrize("degrees", [(500, 513, 1_100), (3_000, 33_000), (40_000, 40_000, 700)])
def test_static_core_of_hubs(P, degrees):  # noqa: F811
    """Static k-core with peeled tables scanned by a warp, a block (above 1,024 slots) and
    the whole grid (above 65,536): estimates and iteration counts equal the oracle's."""
    n = 45_000
    rng = np.random.default_rng(3)
    parts = [W.erdos_renyi(2_000, 9_000, seed=1)]
    for h, d in enumerate(degrees):
        leaves = rng.permutation(np.arange(len(degrees), n))[:d]
        parts.append(np.stack([np.full(d, h), leaves], 1))
    e = np.unique(np.sort(np.concatenate(parts).astype(np.int32), axis=1), axis=0)
    g, o = P.PLDS(n), O.OraclePLDS(n)
    g.insert(e)
    assert o.insert(e) == 0
    for eps in (0.5, 1.0):
        ge, gs = g.static_coreness(eps)
        oe, os_ = o.static_coreness(eps)
        assert np.array_equal(ge, oe) and gs == os_
    g.close()


@pytest.mark.parametrize("hubs", [8, 32, 33, 170])
def test_static_core_of_many_huge_tables(P, hubs):  # noqa: F811
    """Tables above 65,536 slots (a load factor of 1/16: degrees above 4,096): up to 32 peeled
    at once are scanned by the whole grid, more by a block each."""
    n = 9_000
    leaves = np.arange(4_200)
    e = np.concatenate([np.stack([np.full(leaves.size, h), hubs + (leaves + 37 * h) % (n - hubs)], 1)
                        for h in range(hubs)]).astype(np.int32)
    g, o = P.PLDS(n), O.OraclePLDS(n)
    g.set_tuning(load_num=1, load_den=16)
    g.insert(e)
    assert o.insert(e) == 0
    ge, gs = g.static_coreness(1.0)
    oe, os_ = o.static_coreness(1.0)
    assert np.array_equal(ge, oe) and gs == os_
    g.close()


@pytest.mark.parametrize("batch", [9_000, 40_000])
def test_pool_growth_between_batches(P, batch):  # noqa: F811
    """Batches (one launch, or step kernels) that find the adjacency pool full are stopped,
    their per-vertex counts undone, and run again in a larger pool: equal to the oracle's."""
    n = 12_000
    e = W.shuffled(W.chung_lu(n, 280_000, 2.6, seed=4), 5)
    o = O.OraclePLDS(n, levels_per_group=1)
    gs = [P.PLDS(n, levels_per_group=1) for _ in range(6)]
    for k, part in enumerate(W.batches(e, batch)):
        assert o.insert(part) == 0
        for g in gs:
            g.insert(part)
            assert np.array_equal(g.levels(), o.levels()), f"batch {k}"
    assert all(g.stats()["pool_grows"] > 0 for g in gs)
    for g in gs:
        assert_same(g, o, "loaded")
        g.close()
