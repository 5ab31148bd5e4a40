"""The per-element draw at the edges of its rounds and blocks, against the
oracle: leaves of one or two points, around the staging limit of 256 and above
it, neurons with many elements among neurons with none, few leaf pairs (split
into parts) and many.  Partners are whole numbers: equal, except for draws the
oracle flags as within its band of a boundary of the distribution."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

PLAN = dict(cutoff=3.25, rho_max=0.0, p=4)


@pytest.mark.parametrize("elements", ["few", "many"])
@pytest.mark.parametrize("leaf_capacity,n", [(1, 600), (2, 900), (31, 3000), (32, 12_000), (255, 4000),
                                             (256, 4096), (257, 5000), (700, 6000)])
def test_partners_match_the_oracle(oracle_mod, leaf_capacity, n, elements):
    w = W.clustered_small(1, n, seed=leaf_capacity, leaf_capacity=leaf_capacity, **PLAN)
    rng = np.random.default_rng(n)
    if elements == "many":
        # most neurons without elements, some with up to 60
        w.vac_axon[:] = np.where(rng.random(n) < 0.9, 0, rng.integers(1, 61, n))
        w.vac_dend_e[:] = rng.integers(0, 256, n)
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    g.attraction()
    sel = g.select_partners(7)
    got = sel["partner"].cpu().numpy()
    n_syn = int(sel["n_syn"].item())
    g.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    o.attraction()
    ref = o.select_partners(7)
    ne = int(w.vac_axon.sum(dtype=np.int64))
    assert o.num_elements() == ne and len(ref["partner"]) >= ne
    same = got[:ne] == ref["partner"][:ne]
    assert np.all(same | ref["near_boundary"][:ne])
    if same.all():
        assert n_syn == ref["n_syn"]
