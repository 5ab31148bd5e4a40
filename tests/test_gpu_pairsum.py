"""The pair sums of the derivatives and of the synapse length at the edges of
their passes, against the oracle on the same lists: leaves of one point, of
more points than a pass holds, leaves without targets, one channel only, and
leaves so wide that the transposed sums take the difference form.

Bars as in test_gpu_grad.py and test_gpu_length.py: single precision sums of
positive terms within 1e-5, the signed gradients within 2e-5 (attraction) and
1e-4 (length) of their largest magnitude.
"""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

BASE = dict(cutoff=5.0, rho_max=0.0, p=4, m2l_min_pairs=0)
CASES = {
    "one_point_leaves": (lambda: W.uniform_cube(700, 5000.0, seed=1, leaf_capacity=1, **BASE), None),
    "leaf_capacity_9": (lambda: W.clustered_small(2, 1000, seed=2, leaf_capacity=9, **BASE), None),
    "one_leaf_of_65": (lambda: W.uniform_cube(65, 900.0, seed=3, leaf_capacity=128, **BASE), None),
    "one_leaf_of_300": (lambda: W.uniform_cube(300, 900.0, seed=4, leaf_capacity=512, **BASE), None),
    "wide_leaves": (lambda: W.uniform_cube(900, 30_000.0, seed=5, leaf_capacity=200, **BASE), None),
    "excitatory_only": (lambda: W.clustered_small(1, 1500, seed=6, leaf_capacity=64, **BASE), "E"),
    "inhibitory_only": (lambda: W.clustered_small(1, 1500, seed=6, leaf_capacity=64, **BASE), "I"),
    "few_targets": (lambda: W.clustered_small(1, 1500, seed=7, leaf_capacity=40, **BASE), "few"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_pair_sums_match_the_oracle(oracle_mod, name):
    make, only = CASES[name]
    w = make()
    rng = np.random.default_rng(8)
    if only in ("E", "I"):
        w.type[:] = only == "I"
    if only == "few":
        w.vac_axon[rng.random(w.n) < 0.97] = 0
    g = rng.normal(size=w.n)
    we, wi = (rng.uniform(0.2, 3.0, w.n).astype(np.float32) for _ in range(2))
    ones = np.ones(w.n, np.uint8)
    pos, t, a, e, i = msp.to_device(w)
    one = torch.ones_like(a)
    ctx = msp.MSP(w.params)
    ctx.build_tree(pos, t, one, one, one)
    ctx.attraction()
    r = ctx.attraction_grad(t, a, e, i, g=torch.from_numpy(g).float().cuda())
    ln = ctx.length_loss(t, a, torch.from_numpy(we).cuda(), torch.from_numpy(wi).cuda(), 1000.0)
    r, gl = ({k: v.cpu().numpy().astype(np.float64) for k, v in d.items()}
             for d in (r, {k: ln[k] for k in ("gE", "gI")}))
    ctx.close()
    o = oracle_mod.Oracle(w.params)
    o.build_tree(w.pos, w.type, ones, ones, ones)
    o.attraction()
    ro = o.attraction_grad(w.type, w.vac_axon, w.vac_dend_e, w.vac_dend_i, g=g)
    for k, ko in (("u", "u"), ("du_dsigma", "dudsigma")):
        m = np.abs(ro[ko]) >= 1e-6 * np.abs(ro[ko]).max()
        assert np.max(np.abs(r[k][m] - ro[ko][m]) / np.abs(ro[ko][m])) < 1e-5, k
        assert np.all(r[k][w.vac_axon == 0] == 0.0)
    for k, ko in (("grad_w_e", "gE"), ("grad_w_i", "gI")):
        assert np.max(np.abs(r[k] - ro[ko])) <= 2e-5 * max(np.abs(ro[ko]).max(), 1e-30), k
    lo = o.length_loss(w.type, w.vac_axon, we, wi, 1000.0)
    for k in ("mean", "loss", "dmean_dsigma", "dloss_dsigma"):
        assert ln[k] == pytest.approx(lo[k], rel=1e-5), k
    for k in ("gE", "gI"):
        assert np.max(np.abs(gl[k] - lo[k])) <= 1e-4 * max(np.abs(lo[k]).max(), 1e-30), k
