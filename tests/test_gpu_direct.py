"""The all-pairs paths (msp_direct and msp_direct_noalloc) at the edges of
their kernels' ranges, against the oracle's FP64 brute force: one block of 32
targets, the largest size of the one-launch kernel and the next, both sides of
the change of targets per lane, odd sizes, one channel only, and clusters far
enough apart that whole tiles of sources are left out.

Tolerance: a term's exponent -k2 r^2 carries a relative rounding error of a
few 2^-24, so a term at the exponent's working range (|k2 r^2| < 20) is off by
at most 20 ln 2 * 4 * 6e-8 = 3e-6 relative, EX2 adds 2^-22; 1e-5 covers both
and the compensated sums, over targets of at least 1e-6 of the largest u.
"""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

CASES = {"one": (1, 0), "two": (2, 0), "warp": (32, 0), "warp_plus": (33, 0), "ragged": (1021, 1),
         "small_max": (8192, 1), "lists_min": (8193, 2), "two_per_lane": (39_999, 0),
         "four_per_lane": (40_000, 5), "four_per_lane_odd": (65_535, 7)}


def _network(n, k, seed):
    if k == 0:
        return W.uniform_cube(n, 625.0 * n ** (1 / 3), seed)
    side = 100_000.0 * (max(k, 2) / 8.0) ** (1 / 3)
    w = W.clustered(k, -(-n // k), side, 1500.0, min(4500.0, side / 4), seed)
    return W.subset(w, np.random.default_rng(seed).permutation(w.n)[:n])


@pytest.mark.parametrize("channel", ["both", "inhibitory"])
@pytest.mark.parametrize("name", list(CASES))
def test_all_pairs_at_the_edges_of_the_kernels(oracle_mod, name, channel):
    n, k = CASES[name]
    w = _network(n, k, seed=51)
    if channel == "inhibitory":
        w.type[:] = 1
    w.vac_axon[0] = 1
    g = msp.MSP(w.params)
    dev = msp.to_device(w)
    g.build_tree(*dev)
    got = {"direct": g.direct().cpu().numpy(),
           "noalloc": msp.direct_noalloc(*dev, w.params["sigma"]).cpu().numpy()}
    g.close()
    idx = np.sort(np.random.default_rng(1).choice(n, min(n, 500), replace=False))
    ref = oracle_mod.direct(*w.arrays(), w.params["sigma"], targets=idx)
    m = ref > 1e-6 * ref.max()
    for what, u in got.items():
        assert np.all(u[w.vac_axon == 0] == 0.0), what
        err = np.abs(u[idx][m] - ref[m]) / ref[m]
        assert err.size == 0 or err.max() < 1e-5, (what, err.max())


def test_all_pairs_in_frames_across_tiles(oracle_mod):
    # networks whose boundaries fall inside tiles and target groups, in the
    # kernels with lists (the one-launch kernel runs in test_gpu_batch.py)
    b = W.batch([4001, 700, 5003, 333, 2900], [300.0, 750.0, 1500.0, 500.0, 1100.0],
                ["uniform", "clustered", "uniform", "clustered", "uniform"], seed=9)
    pos, t, a, e, i = msp.to_device(b)
    local, side, level = msp.batch_layout(pos, b.offsets, b.sigma, 4.0, 32)
    g = msp.MSP(W.default_params(side, sigma=1.0), frames=(b.offsets, level))
    g.build_tree(local, t, a, e, i)
    u = g.direct().cpu().numpy()
    g.close()
    lp = local.cpu().numpy()
    for k in range(len(b.sigma)):
        sl = slice(int(b.offsets[k]), int(b.offsets[k + 1]))
        ref = oracle_mod.direct(np.ascontiguousarray(lp[:, sl]), b.type[sl], b.vac_axon[sl],
                                b.vac_dend_e[sl], b.vac_dend_i[sl], 1.0)
        m = ref > 1e-6 * ref.max()
        assert np.max(np.abs(u[sl][m] - ref[m]) / ref[m]) < 1e-5
