"""The device's bounded waits, each made to run out (a flag that nothing sets):
the kernel ends, the next synchronising call reports MSP_ERR_TIMEOUT before it
changes what its caller holds, and the context works on."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

WAITS = {"scan": 0, "sort": 1, "barrier": 2}


def _edges(n, rng):
    m = 5 * n
    pre, post = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    return msp.edge_list(m, pre=pre, post=post, type_=(rng.random(m) < 0.5).astype(np.uint8))


@pytest.mark.parametrize("call", ["build", "kept_build", "attraction", "select", "update", "append"])
@pytest.mark.parametrize("wait", list(WAITS))
def test_a_wait_that_runs_out_is_reported_by_the_next_call(wait, call):
    w = W.uniform_4k()
    n = w.n
    rng = np.random.default_rng(2)
    dev = msp.to_device(w)
    edges = _edges(n, rng)
    state = dict(x=torch.zeros(n, device="cuda"),
                 **{k: torch.from_numpy(rng.uniform(0, 6, n).astype(np.float32)).cuda()
                    for k in ("z_axon", "z_dend_e", "z_dend_i")})
    vac = [torch.full((n,), 77, dtype=torch.uint8, device="cuda") for _ in range(3)]
    g = msp.MSP(w.params)
    g.build_tree(*dev)
    if call == "kept_build":
        g.build_tree(*dev)
    g.attraction()
    sel = g.select_partners(0)
    before = [edges[k].clone() for k in ("n", "pre", "post", "type")]
    g.selftest_wait(WAITS[wait])
    run = {"build": lambda: g.build_tree(*dev), "kept_build": lambda: g.build_tree(*dev),
           "attraction": g.attraction, "select": lambda: g.select_partners(0),
           "update": lambda: g.update_synapses(3, state, edges, *vac),
           "append": lambda: g.append_synapses(sel, edges)}[call]
    with pytest.raises(msp.MSPError) as err:
        run()
    assert err.value.code == 4                           # MSP_ERR_TIMEOUT
    if call == "update":
        for k, b in zip(("n", "pre", "post", "type"), before):
            assert torch.equal(edges[k], b), k
        assert all((v == 77).all() for v in vac)
        run()                                            # reported once
        assert not any((v == 77).any() for v in vac)
    # the context works on, as one that never waited
    f = msp.MSP(w.params)
    got = []
    for c in (g, f):
        c.build_tree(*dev)
        u = c.attraction()
        s = c.select_partners(7)
        m = int(s["n_syn"])
        got.append([u, s["partner"], s["syn_pre"][:m], s["syn_post"][:m]])
        c.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


def test_no_such_wait():
    g = msp.MSP(W.uniform_4k().params)
    for which in (-1, 3):
        with pytest.raises(msp.MSPError):
            g.selftest_wait(which)
    g.close()
