"""The update of synapses where the workspace limit does not hold the scratch of
both sides' sort: one side after the other, with the same results; and an error
that changes nothing where one side does not fit either."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


@pytest.mark.parametrize("m", [300_000, 700_001])
def test_update_within_a_workspace_limit(m):
    n = 2000
    rng = np.random.default_rng(m)
    pre, post = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    typ = rng.integers(0, 2, m).astype(np.uint8)
    z = {k: torch.from_numpy(rng.uniform(0, 1.2 * m / n, n).astype(np.float32)).cuda()
         for k in ("z_axon", "z_dend_e", "z_dend_i")}
    state = dict(x=torch.zeros(n, device="cuda"), **z)

    def update(limit):
        g = msp.MSP(W.default_params(1000.0, seed=5))
        edges = msp.edge_list(m, pre=pre, post=post, type_=typ)
        vac = [torch.full((n,), 77, dtype=torch.uint8, device="cuda") for _ in range(3)]
        base = msp.workspace_bytes()
        try:
            if limit:
                msp.set_workspace_limit(base + limit)
            g.update_synapses(9, state, edges, *vac)
            used = msp.workspace_bytes() - base
        except msp.MSPError as e:
            assert e.code == 3, e                        # MSP_ERR_OOM
            assert int(edges["n"]) == m and all((v == 77).all() for v in vac)
            assert np.array_equal(edges["pre"].cpu().numpy(), pre)
            return None, 0
        finally:
            msp.set_workspace_limit(0)
            g.close()
        k = int(edges["n"])
        return [edges[f][:k] for f in ("pre", "post", "type")] + vac, used

    free, whole = update(0)
    assert 0 < free[0].numel() < m
    # 42 bytes an edge (with the buffers' quarter of headroom) were enough for a
    # sort per side: less than what both sides at once take
    limit = int(1.25 * 42 * m) + (1 << 18)
    assert limit < whole
    tight, used = update(limit)
    assert used <= limit
    for a, b in zip(free, tight):
        assert torch.equal(a, b)
    assert update(1 << 18) == (None, 0)
