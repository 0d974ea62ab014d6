"""GPU parity at the sizes where single kernels change path (GB300 only).

Each test drives one kernel family over the edges of its tiles, bins or size
classes and compares the whole state with the oracle, integers exactly.
"""
import numpy as np
import pytest

from oracle import Oracle
from synth import EdgeStream, csr_from_arcs, random_batch
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


def _bin_edge_graph(directed, weight, seed):
    """Small cliques joined at random, and one node per degree of BIN_EDGES."""
    rng = np.random.default_rng(seed)
    n, k = 6000, 12
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
