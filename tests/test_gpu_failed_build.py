"""A build that is refused (a position outside the domain or not finite) has
already rewritten the octree's arrays: replays captured on the octree before it
must not take them for that octree.  Their results are those of a context that
never saw the refused positions."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


def _good_and_bad(n, value):
    good = W.uniform_cube(n, 4000.0, seed=1, cutoff=4.0)
    bad = W.uniform_cube(n, 4000.0, seed=2, cutoff=4.0)
    bad.pos[2, n // 3] = value
    return good, bad


def _host_step(g, w, step):
    out = g.plasticity_step_host(step, *w.arrays())
    m = int(out["n_syn"][0])
    return [out["u"], out["partner"]] + [out[k][:m] for k in ("syn_pre", "syn_post", "syn_type")]


@pytest.mark.parametrize("value", [np.nan, -1.0])
def test_host_step_after_refused_positions(value):
    good, bad = _good_and_bad(3000, value)
    g, f = msp.MSP(good.params), msp.MSP(good.params)
    for step in range(2):                      # the second call replays
        _host_step(g, good, step)
    with pytest.raises(msp.MSPError):
        _host_step(g, bad, 2)
    for step in (3, 4):
        for a, b in zip(_host_step(g, good, step), _host_step(f, good, step)):
            assert np.array_equal(a, b), step
    g.close()
    f.close()


@pytest.mark.parametrize("refused", [False, True])
def test_step_graph_after_refused_positions(refused):
    good, bad = _good_and_bad(3000, np.nan)

    def run(with_bad):
        g = msp.MSP(good.params)
        state = msp.to_device(good)
        g.build_tree(*state)
        g.attraction()
        out = g.step_graph_capture(*state, 0, history_len=4)
        g.step_graph_launch(2)
        assert g.step_graph_finish() == (2, 0)
        if with_bad:
            with pytest.raises(msp.MSPError):
                g.build_tree(*msp.to_device(bad))
        g.step_graph_launch(1)
        nxt, _ = g.step_graph_finish()         # a halted step is finished eagerly
        assert nxt == 3
        m = int(out["n_syn"])
        res = [t.cpu().numpy() for t in state[2:]] + \
              [out[k][:m].cpu().numpy() for k in ("syn_pre", "syn_post", "syn_type")] + \
              [out["history"][:3].cpu().numpy()]
        g.close()
        return res

    for a, b in zip(run(refused), run(False)):
        assert np.array_equal(a, b)
