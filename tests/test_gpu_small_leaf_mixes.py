"""The near field of small leaves with every mix of excitatory and inhibitory
targets that a leaf of eight points can have (45 of them, seven of one channel and
one of the other among them: four groups of targets), against the oracle.
Tolerances as for the other small leaves: u 1e-5 relative, box-pair attractions
1e-5 relative and 1e-7 of the largest."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

MIXES = [(e, i) for e in range(9) for i in range(9 - e)]


@pytest.mark.parametrize("first", [0, 19])
def test_every_mix_of_targets_in_a_leaf(oracle_mod, first):
    # 64 cells of eight points: the leaves of level 2, each with a mix of its own
    # (`first` shifts which cells the mixes beyond 45 and which neighbours meet)
    side, cell = 6000.0, 1500.0
    w = W.uniform_cube(512, side, seed=3, leaf_capacity=8, rho_max=0.0, cutoff=3.25)
    rng = np.random.default_rng(4)
    low = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(64, 3) * cell
    w.pos[:] = (np.repeat(low, 8, 0) + rng.uniform(0.05, 0.95, (512, 3)) * cell).T
    for k in range(64):
        e, i = MIXES[(first + k) % len(MIXES)]
        kind = rng.permutation(np.array([0] * e + [1] * i + [2] * (8 - e - i)))
        w.type[8 * k:8 * k + 8] = np.where(kind == 2, rng.integers(0, 2, 8), kind)
        w.vac_axon[8 * k:8 * k + 8] = np.where(kind == 2, 0, rng.integers(1, 4, 8))
    g = msp.MSP(w.params)
    g.build_tree(*msp.to_device(w))
    u = g.attraction().cpu().numpy()
    p, leaves = g.export_pairs(), g.stats()["n_leaves"]
    g.close()
    assert leaves == 64
    o = oracle_mod.Oracle(w.params)
    o.build_tree(*w.arrays())
    uo = o.attraction()
    op = o.pairs()
    assert np.all(u[w.vac_axon == 0] == 0.0)
    m = uo > 1e-6 * uo.max()
    assert np.max(np.abs(u[m] - uo[m]) / uo[m]) < 1e-5
    for k in ("wE", "wI"):
        err = np.abs(p[k] - op[k])
        assert np.all(err <= 1e-5 * np.abs(op[k]) + 1e-7 * np.abs(op[k]).max()), k
