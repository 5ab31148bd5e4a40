"""The selection's synapse list written by the scan over the elements: exactly
the accepted elements in element order, whether the groups fit their dendrites
or not, with the counts of the build (also a second selection after a commit),
on dirty output buffers."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


def _expected(partner, off, t, va, ve, vi, syn):
    """Checks a synapse list: in element order, one per accepted element, at most
    the capacity per dendrite and channel and all requests where they fit."""
    req = {}
    for k in range(len(t)):
        for e in range(off[k], off[k] + va[k]):
            if partner[e] >= 0:
                req.setdefault((int(t[k]), int(partner[e])), []).append(e)
    owner = np.repeat(np.arange(len(t)), np.diff(np.append(off, len(partner))))
    pre, post, typ = syn
    assert np.array_equal(typ, (t[pre] != 0).astype(np.uint8))
    got = {}
    for p, q, c in zip(pre, post, typ):
        got.setdefault((int(c), int(q)), []).append(int(p))
    for (c, q), es in req.items():
        cap = int((vi if c else ve)[q])
        have = got.pop((c, q), [])
        assert len(have) == min(cap, len(es))
        if len(es) <= cap:
            assert have == [int(owner[e]) for e in es]
    assert not got and np.all(np.diff(pre) >= 0)


@pytest.mark.parametrize("n,cap", [(1, 3), (33, 1), (700, 5), (2049, 2), (5000, 1)])
def test_synapses_are_the_accepted_elements(n, cap):
    w = W.uniform_cube(n, 2000.0, seed=n, cutoff=4.0)
    rng = np.random.default_rng(n)
    w.vac_axon[:] = rng.integers(0, 4, n)
    w.vac_dend_e[:] = rng.integers(0, cap + 1, n)
    w.vac_dend_i[:] = rng.integers(0, cap + 1, n)
    w.type[:] = rng.random(n) < 0.4
    pos, t, a, e, i = msp.to_device(w)
    g = msp.MSP(w.params)
    g.build_tree(pos, t, a, e, i)
    g.attraction()
    off = np.concatenate([[0], np.cumsum(w.vac_axon.astype(np.int64))])[:-1]
    sel = None
    for step in range(3):
        if sel is None:
            sel = g.select_partners(step)
        else:
            for v in sel.values():
                v.fill_(1)
            g.select_partners(step, out=sel)
        m = int(sel["n_syn"])
        _expected(sel["partner"].cpu().numpy()[:int(w.vac_axon.sum())], off, w.type, w.vac_axon,
                  w.vac_dend_e, w.vac_dend_i,
                  [sel[k][:m].cpu().numpy() for k in ("syn_pre", "syn_post", "syn_type")])
        g.commit_synapses(sel, a, e, i)
    g.close()
