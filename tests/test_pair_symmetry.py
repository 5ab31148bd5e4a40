"""The near-field pairs of a traversal without translated pairs are symmetric:
with (X, Y) the list holds (Y, X).  The transposed sums of the derivatives
rest on it (they walk the list sorted by target leaf in both directions); here
over the plans that those sums accept, on the oracle's lists, which the GPU's
equal bit for bit (test_gpu_parity.py)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_10570_gb300 import workloads as W

PLANS = {"default_leaves": dict(leaf_capacity=32, cutoff=5.0, rho_max=0.0),
         "large_leaves": dict(leaf_capacity=160, cutoff=3.25, rho_max=0.0),
         "one_point_leaves": dict(leaf_capacity=1, cutoff=2.0, rho_max=0.0, max_depth=5),
         "separated_but_too_small": dict(leaf_capacity=16, cutoff=4.0, rho_max=0.5,
                                         m2l_min_pairs=1 << 40),
         "count_rule_never_expands": dict(leaf_capacity=16, cutoff=4.0, mac_mode=1, c1=1 << 30)}


@pytest.mark.parametrize("kind", ["uniform", "clustered", "one_sided"])
@pytest.mark.parametrize("name", list(PLANS))
def test_near_field_pairs_are_symmetric(name, kind):
    w = (W.uniform_cube(1537, 6000.0, seed=3, **PLANS[name]) if kind == "uniform" else
         W.clustered_small(2, 900, seed=4, **PLANS[name]))
    if kind == "one_sided":
        # all targets in one cluster, all sources in the other
        w.vac_axon[:900] = 0
        w.vac_dend_e[900:] = 0
        w.vac_dend_i[900:] = 0
    o = O.Oracle(w.params)
    o.build_tree(*w.arrays())
    o.attraction()
    p = o.pairs()
    assert not (p["kind"] == 1).any()
    near = p["kind"] == 2
    key = np.stack([p["X"][near], p["Y"][near]]).astype(np.int64)
    there, back = (np.sort(a * (1 << 32) + b) for a, b in (key, key[::-1]))
    assert len(there) > 0 and np.array_equal(there, back)
