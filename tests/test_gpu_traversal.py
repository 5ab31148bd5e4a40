"""The octree and the dual traversal across the tiles of their one-launch
levels and depths (128 boxes, 256 pairs), bit for bit against the oracle, and
the traversal with a pair table that overflows at every kind of place (the
first depths, inside a tile, at a block's edge): grown and redone, it gives the
same pairs.  Whole numbers: no tolerance."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

PLANS = {"many_levels": lambda: W.clustered_small(1, 3000, seed=1, leaf_capacity=1, cutoff=0.5,
                                                  rho_max=0.0),
         "wide_level": lambda: W.uniform_cube(60_000, 25_000.0, seed=2, leaf_capacity=8, cutoff=1.0,
                                              rho_max=0.0),
         "translated": lambda: W.uniform_cube(5000, 10_000.0, seed=3, leaf_capacity=4, cutoff=3.0,
                                              rho_max=0.6),
         "shallow": lambda: W.uniform_cube(300, 3000.0, seed=4, leaf_capacity=2, max_depth=2)}


@pytest.mark.parametrize("name", list(PLANS))
def test_octree_and_pairs_match_the_oracle(oracle_mod, name):
    w = PLANS[name]()
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    g.attraction()
    tree, pairs = g.export_tree(), g.export_pairs()
    g.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    o.attraction()
    nodes, op = o.nodes(), o.pairs()
    for k in ("level", "prefix", "first", "count", "parent", "child_first", "nchild", "sums"):
        assert np.array_equal(tree[k], nodes[k]), k
    for k in ("X", "Y", "kind", "child_first", "depth_start"):
        assert np.array_equal(pairs[k], op[k]), k


@pytest.mark.parametrize("capacity", [1, 2, 64, 65, 66, 700, 4160, 20_011])
def test_a_table_that_overflows_is_grown_and_gives_the_same_pairs(capacity):
    w = W.uniform_cube(4096, 10_000.0, seed=5, leaf_capacity=16, cutoff=3.0, rho_max=0.3)
    dev = msp.to_device(w)
    res = []
    for cap in (None, capacity):
        g = msp.MSP(w.params)
        g.build_tree(*dev)
        if cap:
            g.set_pair_capacity(cap)
        u = g.attraction().cpu().numpy()
        sel = g.select_partners(1)
        res.append((u, sel["partner"].cpu().numpy(), g.export_pairs()))
        g.close()
    (u0, p0, a), (u1, p1, b) = res
    assert np.array_equal(u0, u1) and np.array_equal(p0, p1)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
