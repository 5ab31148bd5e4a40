"""The near field of small leaves (at most eight points a leaf: lanes take
whole pairs) against the oracle, at the edges of its rules: every number of
targets from none to eight in both channels' mixes, leaves of one point, wide
leaves (difference form), and overfull leaves at the deepest level (which stay
with the general kernel).  Tolerances as for the general kernel: u 1e-5
relative, box-pair attractions 1e-5 relative and 1e-7 of the largest."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

CASES = {
    "eight": lambda: W.clustered_small(1, 3000, seed=1, leaf_capacity=8, rho_max=0.0, cutoff=3.25),
    "five": lambda: W.clustered_small(1, 2000, seed=2, leaf_capacity=5, rho_max=0.0, cutoff=3.0),
    "one": lambda: W.uniform_cube(500, 4000.0, seed=3, leaf_capacity=1, rho_max=0.0, cutoff=2.0),
    "nine_is_general": lambda: W.clustered_small(1, 2000, seed=4, leaf_capacity=9, rho_max=0.0,
                                                 cutoff=3.0),
    "wide": lambda: W.uniform_cube(300, 60_000.0, seed=5, leaf_capacity=8, rho_max=0.0, cutoff=4.0),
    "overfull": lambda: W.uniform_cube(2500, 3000.0, seed=6, leaf_capacity=8, rho_max=0.0,
                                       cutoff=1.0, max_depth=3)}


@pytest.mark.parametrize("active", [0.15, 0.75, 1.0])
@pytest.mark.parametrize("name", list(CASES))
def test_small_leaves_match_the_oracle(oracle_mod, name, active):
    w = CASES[name]()
    rng = np.random.default_rng(9)
    w.vac_axon[:] = np.where(rng.random(w.n) < active, rng.integers(1, 4, w.n), 0)
    w.type[:] = rng.random(w.n) < 0.5
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    u = g.attraction().cpu().numpy()
    again = g.attraction().cpu().numpy()
    p, st = g.export_pairs(), g.stats()
    g.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    uo = o.attraction()
    op = o.pairs()
    assert np.array_equal(u, again) and np.all(u[w.vac_axon == 0] == 0.0)
    m = uo > 1e-6 * uo.max()
    assert np.max(np.abs(u[m] - uo[m]) / uo[m]) < 1e-5
    for k in ("wE", "wI"):
        err = np.abs(p[k] - op[k])
        assert np.all(err <= 1e-5 * np.abs(op[k]) + 1e-7 * np.abs(op[k]).max()), k
    # every target with vacant axons against the sources of its partner leaves
    nd = o.nodes()
    near = op["kind"] == 2
    keys, perm = o.keys()
    act = (w.vac_axon[perm] > 0).astype(np.int64)
    cum = np.concatenate([[0], np.cumsum(act)])
    f, c = nd["first"], nd["count"]
    n_act = cum[f + c] - cum[f]
    assert st["p2p_interactions"] == int((n_act[op["X"][near]] * c[op["Y"][near]].astype(np.int64)).sum())
