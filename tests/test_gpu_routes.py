"""GPU parity of the launch routes a batch can take (GB300 only): which kernel
sweeps a list, what runs ahead of the host and what statistics change.
"""
import numpy as np
import pytest

from synth import planted_partition, planted_stream, rmat_directed, rmat_stream

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
