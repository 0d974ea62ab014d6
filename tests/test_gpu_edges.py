"""GPU parity at the sizes where single kernels change path (GB300 only).

Each test drives one kernel family over the edges of its tiles, bins or size
classes and compares the whole state with the oracle, integers exactly.
"""
import numpy as np
import pytest

from oracle import Oracle
from synth import EdgeStream, csr_from_arcs, random_batch, rmat_directed, rmat_stream
from tests.parity import compare_states

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ldl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2502_18497_gb300 import ldl as mod
    mod.load()
    return mod


# row lengths at and beside the bounds of the sweep bins and their tables
BIN_EDGES = (1, 7, 8, 9, 23, 24, 25, 31, 32, 33, 95, 96, 97, 127, 128, 129, 511, 513, 1023, 1024, 1025, 2047, 2048, 2049,
             4100)


def _bin_edge_graph(directed, weight, seed, n=6000):
    """Small cliques joined at random, and one node per degree of BIN_EDGES."""
    rng = np.random.default_rng(seed)
    k = 12
    v = np.arange(200, n)
    src = [np.repeat(v, 5)]
    dst = [(v // k * k)[:, None].repeat(5, 1).ravel() + rng.integers(0, k, 5 * len(v))]
    src.append(rng.integers(200, n, n // 2))
    dst.append(rng.integers(200, n, n // 2))
    for i, deg in enumerate(BIN_EDGES):
        to = 200 + rng.permutation(n - 200)[:deg]
        out = rng.random(deg) < 0.5 if directed else np.ones(deg, bool)
        src.append(np.where(out, i, to))
        dst.append(np.where(out, to, i))
    src, dst = np.concatenate(src), np.minimum(np.concatenate(dst), n - 1)
    keep = src != dst
    src, dst = src[keep], dst[keep]
    if not directed:
        src, dst = np.minimum(src, dst), np.maximum(src, dst)
    key = np.unique(src * n + dst)
    return csr_from_arcs(n, key // n, key % n, weight(rng, len(key)), directed)


def _ring(n, directed):
    """Every node beside its next neighbours, some rows of a few hundred."""
    rng = np.random.default_rng(n)
    v = np.arange(n)
    src = np.concatenate([np.repeat(v, 4), np.repeat(v[:8], 300)])
    dst = np.concatenate([(v[:, None] + np.arange(1, 5)).ravel() % n, rng.integers(8, n, 2400)])
    if not directed:
        src, dst = np.minimum(src, dst), np.maximum(src, dst)
    key = np.unique(src * n + dst)
    return csr_from_arcs(n, key // n, key % n, np.ones(len(key), np.int64), directed)


def _unit(rng, k):
    return np.ones(k, np.int64)


def _below(rng, k):  # 6 m^2 just below 2^62: one-word sums as large as they get
    w = rng.integers(1, 1000, k)
    return np.maximum(1, w * (870_000_000 // 2) // w.sum())


def _above(rng, k):  # 6 m^2 just above: two-word sums
    w = rng.integers(1, 1000, k)
    return np.maximum(1, w * 900_000_000 // w.sum())


def _huge(rng, k):  # sums of a row's weights carry into the upper word
    return rng.integers(1 << 27, 1 << 28, k)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("weight", [_unit, _below, _above, _huge])
def test_sweep_bins(ldl, directed, weight):
    g = _bin_edge_graph(directed, weight, 31)
    o, d = Oracle(g), ldl.LDL.from_graph(g)
    m = d.numerator()[0]
    assert (6 * m * m < 1 << 62) == (weight in (_unit, _below))
    msgs = compare_states(o, d, "create")
    assert not msgs, "\n".join(msgs[:8])
    st = EdgeStream.from_graph(g, 5)
    wmax = 1 if weight is _unit else 3
    for t in range(3):
        b = random_batch(st, 60, 40, 20, wmax, 17 * t + 1)
        assert o.apply(b) == 0
        d.apply(b)
        msgs = compare_states(o, d, f"batch {t}")
        assert not msgs, "\n".join(msgs[:8])


# sweeps of few nodes (one block each), of up to 131072 (one launch for all
# bins) and of more (a launch per bin)
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("n", [1024, 1025, 131072, 131073])
def test_sweep_sizes(ldl, directed, n):
    g = _bin_edge_graph(directed, _unit, 7, n) if n > 4400 else _ring(n, directed)
    o, d = Oracle(g), ldl.LDL.from_graph(g)
    msgs = compare_states(o, d, "create")
    assert not msgs, "\n".join(msgs[:8])
    b = random_batch(EdgeStream.from_graph(g, 3), 60, 40, 20, 2, 5)
    assert o.apply(b) == 0
    d.apply(b)
    msgs = compare_states(o, d, "batch")
    assert not msgs, "\n".join(msgs[:8])


def _dense_batch(g, size, seed):
    """`size` updates of distinct arcs (edges) of a graph on few vertices: half
    inserts anywhere, a few deletes and reweights of arcs that exist."""
    rng = np.random.default_rng(seed)
    src, col, _ = g.arcs()
    keep = (src < col) if not g.directed else (src != col)
    have = src[keep] * g.n + col[keep]
    old = rng.permutation(have)[: min(size // 4, len(have))]
    new = np.unique(rng.integers(0, g.n, 3 * size) * g.n + rng.integers(0, g.n, 3 * size))
    if not g.directed:
        new = new[new // g.n < new % g.n]
    new = rng.permutation(np.setdiff1d(new[new // g.n != new % g.n], old))[: size - len(old)]
    key = np.concatenate([new, old])
    op = np.zeros(len(key), np.int64)
    op[len(new):] = 1 + np.arange(len(old)) % 2
    w = np.where(op == 1, 0, rng.integers(1, 5, len(key)))
    return rng.permutation(np.stack([key // g.n, key % g.n, op, w], 1)).astype(np.int32)


# update counts at and beside the tiles and size classes of the batch's sorts,
# scans and adjacency updates (512, 1024, 2048, 49152 pairs, then one launch
# per sorting phase from 1.2M)
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("size", [1, 2, 256, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 24576, 24577, 49152,
                                  49153, 1_300_000])
def test_batch_sizes(ldl, directed, size):
    n = 3000 if size > 100_000 else 1500
    rng = np.random.default_rng(size)
    v = np.arange(n)
    src = np.repeat(v, 6)
    dst = np.where(rng.random(6 * n) < 0.8, src // 30 * 30 + rng.integers(0, 30, 6 * n), rng.integers(0, n, 6 * n))
    dst = np.minimum(dst, n - 1)
    keep = src != dst if directed else src < dst
    key = np.unique(src[keep] * n + dst[keep])
    g = csr_from_arcs(n, key // n, key % n, rng.integers(1, 5, len(key)), directed)
    o, d = Oracle(g), ldl.LDL.from_graph(g)
    b = _dense_batch(g, size, size + 1)
    assert len(b) == size
    undo = b.copy()[: size // 2]
    undo = undo[undo[:, 2] == 0]  # the second batch deletes some of what the first brought
    undo[:, 2:] = (1, 0)
    for t, x in enumerate((b, undo) if len(undo) else (b,)):
        assert o.apply(x) == 0
        d.apply(x)
        msgs = compare_states(o, d, f"batch {t}")
        assert not msgs, "\n".join(msgs[:8])


# changed vertices up to 4096 come through the mapped page, more by copies
@pytest.mark.parametrize("size,few", [(40, True), (60_000, False)])
def test_changed_labels(ldl, size, few):
    g = rmat_directed(scale=14, arcs=1 << 18, seed=5)
    o, d = Oracle(g), ldl.LDL.from_graph(g)
    before = np.array(o.labels())
    for b in rmat_stream(g, batches=1, size=size, seed=size):
        assert o.apply(b) == 0
        d.apply(b)
    want = np.flatnonzero(np.array(o.labels()) != before)
    assert 0 < len(want) and (len(want) <= 4096) == few
    for ids, lab in (d.changed(), d.changed_noalloc(), d.changed()):
        order = np.argsort(ids)
        assert np.array_equal(ids[order], want)
        assert np.array_equal(lab[order], np.array(o.labels())[want])
