"""Checkpoints of states with a long history (GB300 only)."""
import numpy as np
import pytest

from oracle import Oracle
from synth import EdgeStream, random_batch, random_small_graph
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


# nodes that emptied stay in the children lists: after many batches on a small
# graph those hold more ids than there are vertices
@pytest.mark.parametrize("directed", [False, True])
def test_children_lists_longer_than_the_vertex_set(ldl, tmp_path, directed):
    for seed in range(4):
        g = random_small_graph(16, 0.3, directed, wmax=4, seed=40 + seed)
        o, d = Oracle(g), ldl.LDL.from_graph(g)
        st = EdgeStream.from_graph(g, seed)
        for t in range(60):
            m = len(st.keys)
            b = random_batch(st, 6, min(5, m), min(2, max(0, m - 5)), 4, seed * 97 + t)
            assert o.apply(b) == 0
            d.apply(b)
            if t % 6 == 5:
                path = str(tmp_path / "h.ldl")
                d.save(path)
                d.close()
                d = ldl.LDL.load(path)
                msgs = compare_states(o, d, f"seed {seed} batch {t}")
                assert not msgs, "\n".join(msgs[:8])
