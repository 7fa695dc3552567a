"""GPU paths chosen by size, at the sizes where the choice or a tile ends."""
import numpy as np
import pytest

from paper_2510_23330_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_23330_gb300 import galnb
    return galnb


# tree build: one round of 256 slots per tile up to 2^20 slots, two beyond
@pytest.mark.parametrize("n", [255, 256, 257, (1 << 20) + 1])
def test_tree_topology_at_tile_edges(G, orc, n):
    p = ics.plummer(n, seed=n, n_gas=0)
    c = G.Context(n_leaf=16, n_group=64)
    c.set_particles(p)
    c.build_tree()
    key, _, _, _ = orc.morton(p)
    tree = orc.octree(key[orc.sort_order(key)], 16)
    ref = np.stack([tree["level"], tree["prefix"].astype(np.int64), tree["first"], tree["count"]], axis=1)
    assert np.array_equal(c.get("NODES"), ref)
    links = c.get("NODE_LINKS").reshape(-1, 3)
    assert np.array_equal(links[:, 0], tree["child"]) and np.array_equal(links[:, 1], tree["nchild"])
    assert np.array_equal(np.sort(c.get("GROUPS")), np.sort(orc.groups(tree, 64)))
