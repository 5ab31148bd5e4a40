"""The octree's first levels from the cells that the gather finds, against the
oracle's octree: one point, all points in one cell (the first, the last), two far
apart, empty stretches between clusters, every cell filled; limits on the depth
above and below the levels of the first block."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

SIDE = 8000.0


def _points(name, rng):
    if name == "one":
        return np.full((3, 1), 4000.5)
    if name == "first":
        return rng.random((3, 900)) * 400.0
    if name == "last":
        return SIDE - 400.0 + rng.random((3, 900)) * 399.0
    if name == "two":
        return np.array([[1.0, 7998.0]] * 3)
    if name == "clusters":
        c = rng.uniform(500, 7500, (3, 6))
        return np.clip(np.repeat(c, 300, 1) + rng.normal(0, 60, (3, 1800)), 0, 7999)
    g = (np.arange(16) + 0.5) * SIDE / 16
    return np.stack([v.ravel() for v in np.meshgrid(g, g, g)])


@pytest.mark.parametrize("max_depth", [0, 1, 3, 4, 5, 21])
@pytest.mark.parametrize("name", ["one", "first", "last", "two", "clusters", "every_cell"])
def test_octree_equals_the_oracle(oracle_mod, name, max_depth):
    pos = np.ascontiguousarray(_points(name, np.random.default_rng(3)).astype(np.float32))
    n = pos.shape[1]
    w = W.uniform_cube(n, SIDE, seed=4, leaf_capacity=2, max_depth=max_depth, cutoff=3.0)
    w.pos[:] = pos
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    t = g.export_tree()
    g.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    keys, perm = o.keys()
    nd = o.nodes()
    assert np.array_equal(t["keys"], keys) and np.array_equal(t["perm"], perm)
    for k in ("level", "prefix", "first", "count", "parent", "child_first", "nchild"):
        assert np.array_equal(t[k], nd[k]), k
