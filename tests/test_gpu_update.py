"""The update of synapses at the edges of its sort and of its in-place
compaction (tiles of 2,048 edges), against the oracle bit for bit: no edge, no
deletion (nothing is written), every edge deleted, a hub that holds most
edges, deletions in the last tile only, a full list."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_2301_10570_gb300 import msp  # noqa: E402


@pytest.mark.parametrize("m", [0, 1, 2047, 2048, 2049, 30_001])
@pytest.mark.parametrize("kind", ["some", "none", "all", "hub", "last"])
def test_update_matches_the_oracle(m, kind):
    rng = np.random.default_rng(m + 1)
    n = 700
    pre, post = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    typ = rng.integers(0, 2, m).astype(np.uint8)
    if kind == "hub":
        pre[rng.random(m) < 0.8] = 5
        post[rng.random(m) < 0.6] = 9
    if kind == "last" and m:
        pre[-1] = n - 1
        pre[:-1] %= n - 1
    z = [rng.uniform(0, 2.2 * m / n + 1, n).astype(np.float32) for _ in range(3)]
    if kind == "none":
        z = [np.full(n, m + 1, np.float32) for _ in range(3)]
    if kind == "all":
        z = [np.zeros(n, np.float32)] + z[1:]
    if kind == "last":
        z = [np.full(n, m + 1, np.float32) for _ in range(3)]
        z[0][n - 1] = 0.0
    (p2, q2, t2), vac = O.update_synapses(5, 9, *z, pre, post, typ)
    g = msp.MSP(W.default_params(1000.0, seed=5))
    edges = msp.edge_list(m, pre=pre, post=post, type_=typ)
    state = dict(x=torch.zeros(n, device="cuda"),
                 **{k: torch.from_numpy(v).cuda() for k, v in zip(("z_axon", "z_dend_e", "z_dend_i"), z)})
    got = [torch.full((n,), 77, dtype=torch.uint8, device="cuda") for _ in range(3)]
    g.update_synapses(9, state, edges, *got)
    torch.cuda.synchronize()
    g.close()
    k = int(edges["n"].item())
    assert k == len(p2)
    for name, ref in (("pre", p2), ("post", q2), ("type", t2)):
        assert np.array_equal(edges[name][:k].cpu().numpy(), ref), name
    for a, b in zip(got, vac):
        assert np.array_equal(a.cpu().numpy(), b)
