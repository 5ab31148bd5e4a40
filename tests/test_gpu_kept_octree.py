"""Builds that keep the octree of the build before: whatever came before a
build (the same positions once or several times, others of the same number, a
full-build replay on others), its results are those of a fresh context."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


def _nets(n):
    a = W.uniform_cube(n, 4000.0, seed=1, cutoff=4.0)
    b = W.uniform_cube(n, 4000.0, seed=2, cutoff=4.0)
    c = W.uniform_cube(n, 4000.0, seed=1, cutoff=4.0)
    c.vac_axon[:] = np.roll(c.vac_axon, 1)
    c.vac_dend_e[:] = np.roll(c.vac_dend_e, 3)
    moved = W.uniform_cube(n, 4000.0, seed=1, cutoff=4.0)
    moved.pos[1, n // 2] = 1.0                   # one coordinate of one neuron
    return dict(a=a, b=b, c=c, m=moved)


def _step(g, w, step):
    g.build_tree(*msp.to_device(w))
    u = g.attraction()
    s = g.select_partners(step)
    m = int(s["n_syn"])
    st = g.stats()
    return [u.cpu().numpy(), s["partner"].cpu().numpy(), s["syn_pre"][:m].cpu().numpy(),
            np.array([st[k] for k in ("n_nodes", "n_pairs", "n_p2p", "n_elements", "n_requests")])]


@pytest.mark.parametrize("n", [1, 300, 5000])
@pytest.mark.parametrize("order", ["aaaab", "aaacbbba", "aammaa", "abcabc", "ccaab"])
def test_any_sequence_equals_fresh_contexts(n, order):
    nets = _nets(n)
    g = msp.MSP(nets["a"].params)
    for k, name in enumerate(order):
        got = _step(g, nets[name], k)
        f = msp.MSP(nets["a"].params)
        want = _step(f, nets[name], k)
        f.close()
        for x, y in zip(got, want):
            assert np.array_equal(x, y), (k, name)
    g.close()


def test_eager_build_after_a_full_build_replay_on_other_positions():
    nets = _nets(3000)
    w = nets["a"]
    g = msp.MSP(w.params)
    pos, t, a, e, i = msp.to_device(w)
    g.build_tree(pos, t, a, e, i)
    g.attraction()
    g.step_graph_set_full_build(True)
    g.step_graph_capture(pos, t, a, e, i, 0)
    pos.copy_(torch.from_numpy(nets["b"].pos))
    g.step_graph_launch(1)
    g.step_graph_finish()
    got = _step(g, w, 5)
    f = msp.MSP(w.params)
    want = _step(f, w, 5)
    f.close()
    g.close()
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
