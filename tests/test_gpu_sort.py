"""The radix sort through the Morton order of a build, at the edges of its
tiles (2,048 elements) and launch (three resident blocks per SM, then tiles
by turns): keys in order, the order stable, every neuron once.  Whole numbers:
no tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp, workloads as W  # noqa: E402


def _spread(v):
    v = v.astype(np.uint64)
    for s, m in ((32, 0x1f00000000ffff), (16, 0x1f0000ff0000ff), (8, 0x100f00f00f00f00f),
                 (4, 0x10c30c30c30c30c3), (2, 0x1249249249249249)):
        v = (v | (v << np.uint64(s))) & np.uint64(m)
    return v


@pytest.mark.parametrize("kind", ["spread", "two_keys", "one_key"])
@pytest.mark.parametrize("n", [1, 2, 31, 255, 2047, 2048, 2049, 40_961, 1_300_001])
def test_morton_order_is_sorted_and_stable(n, kind):
    rng = np.random.default_rng(n)
    side = np.float32(8192.0)
    pos = (rng.random((3, n)) * float(side)).astype(np.float32)
    pos = np.minimum(pos, np.nextafter(side, np.float32(0)))
    if kind == "two_keys":
        pos[:] = np.where(rng.random(n) < 0.5, np.float32(10.0), np.float32(8000.0))
    if kind == "one_key":
        pos[:] = np.float32(77.0)
    counts = [torch.ones(n, dtype=torch.uint8, device="cuda") for _ in range(4)]
    # leaves of any size: the octree stays small
    g = msp.MSP(W.default_params(float(side), leaf_capacity=max(n, 1), max_depth=2))
    g.build_tree(torch.from_numpy(pos).cuda(), *counts)
    t = g.export_tree()
    g.close()
    q = np.floor(pos * np.float32(2 ** 21 / float(side))).astype(np.uint64)
    key = (_spread(q[0]) << np.uint64(2)) | (_spread(q[1]) << np.uint64(1)) | _spread(q[2])
    order = np.argsort(key, kind="stable")
    assert np.array_equal(t["perm"], order)
    assert np.array_equal(t["keys"], key[order])
