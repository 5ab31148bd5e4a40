"""Coefficients and translations of every order against the oracle: few and
many far pairs per target box (odd and even numbers, for the order whose pairs
are taken two at a time), boxes of one point and of more than a chunk's 32
points.  Tolerances as for the pair tables with far pairs: attractions 1e-4
relative and 1e-7 of the largest; u 1e-5 relative to the oracle's u, where it
is above 1e-3 of the largest (below, the series' own terms cancel)."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


@pytest.mark.parametrize("p,leaf,rho,n,side", [(p, 1, 0.3, 60, 1500.0) for p in range(1, 9)] +
                         [(4, 1, 0.3, 400, 3000.0), (4, 8, 0.4, 1500, 2500.0),
                          (4, 48, 0.4, 6000, 1500.0), (6, 48, 0.4, 6000, 1500.0)])
def test_translations_match_the_oracle(oracle_mod, p, leaf, rho, n, side):
    w = W.uniform_cube(n, side, seed=p, leaf_capacity=leaf, rho_max=rho, cutoff=4.0, p=p)
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    u = g.attraction().cpu().numpy()
    again = g.attraction().cpu().numpy()
    t, st = g.export_pairs(), g.stats()
    g.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    uo = o.attraction()
    op = o.pairs()
    assert st["n_far"] > 0 and np.array_equal(u, again)
    m = uo > 1e-3 * uo.max()
    assert np.max(np.abs(u[m] - uo[m]) / uo[m]) < 1e-5
    for k in ("wE", "wI"):
        err = np.abs(t[k] - op[k])
        assert np.all(err <= 1e-4 * np.abs(op[k]) + 1e-7 * np.abs(op[k]).max()), k


@pytest.mark.parametrize("p", [1, 4, 8])
@pytest.mark.parametrize("leaf,rho,n,side", [(1, 0.3, 60, 1500.0), (4, 0.4, 200, 1000.0)])
def test_descent_through_translated_pairs_matches_the_oracle(oracle_mod, p, leaf, rho, n, side):
    w = W.uniform_cube(n, side, seed=20 + p, leaf_capacity=leaf, rho_max=rho, cutoff=4.0, p=p)
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    g.attraction()
    sel = g.select_partners(3)
    st = g.stats()
    g.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    o.attraction()
    ro = o.select_partners(3)
    differ = sel["partner"].cpu().numpy()[:st["n_elements"]] != ro["partner"]
    assert st["n_far"] > 0 and np.all(ro["near_boundary"][differ])
