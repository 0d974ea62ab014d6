"""GPU parity of the launch routes a batch can take (GB300 only): which kernel
sweeps a list, what runs ahead of the host and what statistics change.
"""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from oracle import Oracle
from synth import (EdgeStream, csr_from_arcs, planted_partition, planted_stream, random_batch, rmat_directed,
                   rmat_stream)
from tests.parity import compare_states
from tests.test_gpu_edges import _bin_edge_graph, _unit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ldl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2502_18497_gb300 import ldl as mod
    mod.load()
    return mod


# short lists without hub rows (the filter and the split run ahead) and a
# stream whose sweeps have hub rows
@pytest.mark.parametrize("graph", ["planted", "rmat"])
def test_statistics_add_no_host_wait(ldl, graph):
    if graph == "planted":
        g = planted_partition(n=3000, block=50, seed=3)
        batches = planted_stream(g, batches=6, size=40, seed=3, block=50)
    else:
        g = rmat_directed(scale=14, arcs=1 << 18, seed=12)
        batches = rmat_stream(g, batches=6, size=100, seed=12)
    plain, stats = ldl.LDL.from_graph(g), ldl.LDL.from_graph(g)
    stats.set_kernel_stats(True)
    for t, b in enumerate(batches):
        p, s = plain.apply(b), stats.apply(b)
        assert s.host_syncs == p.host_syncs, f"batch {t}"
        assert np.array_equal(plain.labels(), stats.labels())
    ks = stats.kernel_stats()
    assert sum(k["launches"] for k in ks.values()) > 0
    assert (ks["sweep_hub_acc"]["launches"] > 0) == (graph == "rmat")


def _long_row(n, deg, seed):
    """A ring of 5-neighbour nodes and one node with `deg` entries."""
    rng = np.random.default_rng(seed)
    v = np.arange(1, n)
    src = np.concatenate([np.repeat(v, 4), np.zeros(deg // 2, np.int64), 1 + rng.permutation(n - 1)[: deg - deg // 2]])
    dst = np.concatenate([(1 + (v[:, None] + np.arange(4)) % (n - 1)).ravel(), 1 + rng.permutation(n - 1)[: deg // 2],
                          np.zeros(deg - deg // 2, np.int64)])
    keep = src != dst
    key = np.unique(src[keep] * n + dst[keep])
    return csr_from_arcs(n, key // n, key % n, np.ones(len(key), np.int64), True)


# the caller's last bound holds in a sweep of few nodes too: a row above it goes
# to a cluster where those are on, else to the hub path
@pytest.mark.parametrize("cluster_max_deg,path", [(32768, "sweep_cluster"), (0, "sweep_hub_acc")])
def test_last_bin_bound_holds_in_short_sweeps(ldl, cluster_max_deg, path):
    g = _long_row(1000, 1500, 3)
    o = Oracle(g)
    d = ldl.LDL.from_graph(g, cluster_max_deg=cluster_max_deg, bin_deg=(24, 96, 1024, 1024))
    for t, b in enumerate(([[0, 5, 0, 3], [7, 0, 0, 3]], [[0, 5, 1, 0], [9, 11, 0, 2]])):
        b = np.array(b, np.int32)
        d.set_kernel_stats(False)  # clears the counts, which go on without statistics
        assert o.apply(b) == 0
        d.apply(b)
        msgs = compare_states(o, d, f"batch {t}")
        assert not msgs, "\n".join(msgs[:8])
        entries = {k: x["entries"] for k, x in d.kernel_stats().items()}
        if t == 0:  # touches the long row
            assert entries[path] >= 1500


# one launch for all bins up to 262144 nodes, a launch per bin above
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("n", [262144, 262145])
def test_one_launch_or_a_launch_per_bin(ldl, directed, n):
    g = _bin_edge_graph(directed, _unit, 7, n)
    o, d = Oracle(g), ldl.LDL.from_graph(g)
    msgs = compare_states(o, d, "create")
    assert not msgs, "\n".join(msgs[:8])
    b = random_batch(EdgeStream.from_graph(g, 3), 60, 40, 20, 2, 5)
    assert o.apply(b) == 0
    d.apply(b)
    msgs = compare_states(o, d, "batch")
    assert not msgs, "\n".join(msgs[:8])


# threads that read one batch's changed labels at the same time (4096 vertices
# and fewer come through one mapped page)
def test_changed_labels_read_by_several_threads(ldl):
    g = rmat_directed(scale=14, arcs=1 << 18, seed=5)
    d = ldl.LDL.from_graph(g)
    for b in rmat_stream(g, batches=1, size=40, seed=40):
        d.apply(b)
    ids, lab = d.changed()
    assert 0 < len(ids) <= 4096
    with ThreadPoolExecutor(8) as pool:
        got = list(pool.map(lambda _: d.changed(), range(400)))
    for i, x in got:
        assert np.array_equal(i, ids) and np.array_equal(x, lab)


# every round's filter is charged to its own stage, and nothing but the order of
# launches changes while stages are timed
def test_stage_times_charge_the_filter(ldl):
    g = planted_partition(n=3000, block=50, seed=3)
    plain, timed = ldl.LDL.from_graph(g), ldl.LDL.from_graph(g)
    timed.set_timing(True)
    rounds = 0
    for b in planted_stream(g, batches=4, size=40, seed=3, block=50):
        plain.apply(b)
        rounds += timed.apply(b).decouple_rounds
        assert np.array_equal(plain.labels(), timed.labels())
    assert rounds > 0
    times = timed.stage_times()
    assert times["decouple"] > 0 and times["aggregate"] >= times["agg.emit"] > 0


# counters beyond the arena live at their home words: from the start, and from
# some way into a batch; static build and batches with hub rows and more than
# 8192 candidates in a sweep, and with rolled-back mini-batches
@pytest.mark.parametrize("words", [0, 64, 500])
@pytest.mark.parametrize("what", ["hubs", "rollbacks"])
def test_counters_beyond_the_arena(ldl, words, what):
    if what == "hubs":
        g, size = rmat_directed(scale=14, arcs=1 << 18, seed=12), 1000
        assert Oracle(g, L=0, M_static=1).counters()["candidates"] > 8192
    else:
        g, size = rmat_directed(scale=12, arcs=1 << 15, seed=0), 300
    o = Oracle(g)
    ldl.load().ldl_debug_arena_words(words)
    try:
        d = ldl.LDL.from_graph(g)
        msgs = compare_states(o, d, "create")
        assert not msgs, "\n".join(msgs[:8])
        before = o.counters()["rollbacks"]
        for t, b in enumerate(rmat_stream(g, batches=3, size=size, seed=12 if what == "hubs" else 0)):
            assert o.apply(b) == 0
            d.apply(b)
            msgs = compare_states(o, d, f"batch {t}")
            assert not msgs, "\n".join(msgs[:8])
    finally:
        ldl.load().ldl_debug_arena_words(-1)
    assert what == "hubs" or o.counters()["rollbacks"] > before > 0


# the routes a user's batches take (statistics off) with clusters and non-default
# bins: rows above the last bound in lists of a few nodes and of thousands
@pytest.mark.parametrize("cluster_max_deg,bin_deg", [(32768, None), (0, (16, 64, 256, 1024)),
                                                     (4096, (8, 8, 32, 100))])
@pytest.mark.parametrize("size", [3, 1000])
def test_bins_and_clusters_without_statistics(ldl, cluster_max_deg, bin_deg, size):
    g = rmat_directed(scale=14, arcs=1 << 18, seed=12)
    o = Oracle(g)
    d = ldl.LDL.from_graph(g, cluster_max_deg=cluster_max_deg, bin_deg=bin_deg)
    for t, b in enumerate(rmat_stream(g, batches=6, size=size, seed=12)):
        assert o.apply(b) == 0
        d.apply(b)
        msgs = compare_states(o, d, f"batch {t}")
        assert not msgs, "\n".join(msgs[:8])


def _star_and_rings(directed, leaves=2500, rings=1500):
    """Node 0 with `leaves` neighbours, each of them in a pair, and rings of ten
    nodes far from it."""
    v = np.arange(1, leaves + 1)
    w = leaves + 1 + np.arange(rings)
    ring = w - (w - leaves - 1) % 10
    src = np.concatenate([np.zeros(leaves, np.int64), v[::2], w])
    dst = np.concatenate([v, v[1::2], ring + (w - ring + 1) % 10])
    wt = np.concatenate([np.ones(leaves, np.int64), np.full(leaves // 2, 3), np.full(rings, 2)])
    if not directed:
        src, dst = np.minimum(src, dst), np.maximum(src, dst)
    order = np.argsort(src * 10_000 + dst)
    return csr_from_arcs(leaves + rings + 1, src[order], dst[order], wt[order], directed)


# a short sweep meets a hub row where the sweep before it had none: the filter
# and the split that were launched ahead give way to the hub path (or, with
# clusters on, stand), in batches that move nodes and in batches that do not
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("cluster_max_deg", [0, 32768])
def test_hub_row_appears_in_a_short_sweep(ldl, directed, cluster_max_deg):
    g = _star_and_rings(directed)
    o, d = Oracle(g), ldl.LDL.from_graph(g, cluster_max_deg=cluster_max_deg)
    path = "sweep_cluster" if cluster_max_deg else "sweep_hub_acc"
    far = 2600
    batches = [
        ([[far, far + 25, 0, 1]], False),
        ([[1, 4, 0, 1]], True),  # two leaves of different pairs
        ([[far, far + 25, 1, 0]], False),
        ([[1, 2, 1, 0], [1, 4, 2, 9], [2, 3, 0, 9]], True),
        ([[far + 40, far + 77, 0, 50], [far + 41, far + 78, 0, 50]], False),
        ([[5, 6, 1, 0], [5, far + 3, 0, 4]], True),
        ([[far + 3, far + 200, 0, 30]], None),
        ([[0, 9, 2, 20]], True),  # the hub itself
    ]
    moves = []
    for t, (b, hub) in enumerate(batches):
        b = np.array(b, np.int32)
        d.set_kernel_stats(False)  # clears the counts, which go on without statistics
        assert o.apply(b) == 0
        moves.append(d.apply(b).moves)
        msgs = compare_states(o, d, f"batch {t}")
        assert not msgs, "\n".join(msgs[:8])
        if hub is not None:
            assert (d.kernel_stats()[path]["entries"] > 0) == hub, f"batch {t}"
    assert min(moves) == 0 < max(moves)
