"""Outputs that are one of the call's own inputs: the inputs are read before
they are written, so the results are those of separate buffers."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


@pytest.mark.parametrize("shared", ["u", "du_dsigma", "grad_w_e", "grad_w_i"])
def test_derivatives_written_over_g(shared):
    w = W.clustered_small(2, 2000, seed=4, leaf_capacity=64, rho_max=0.0, cutoff=5.0)
    pos, t, a, e, i = msp.to_device(w)
    g = torch.from_numpy(np.random.default_rng(3).normal(size=w.n)).float().cuda()
    ctx = msp.MSP(w.params)
    ctx.build_tree(pos, t, a, e, i)
    ctx.attraction()
    want = ctx.attraction_grad(t, a, e, i, g=g)
    got = {k: torch.empty_like(g) for k in want}
    got[shared] = g.clone()
    code = msp.load().msp_attraction_grad(
        ctx._h, t.data_ptr(), a.data_ptr(), e.data_ptr(), i.data_ptr(), got[shared].data_ptr(),
        *[got[k].data_ptr() for k in ("u", "du_dsigma", "grad_w_e", "grad_w_i")],
        torch.cuda.current_stream().cuda_stream)
    assert code == 0
    for k in want:
        assert torch.equal(got[k], want[k]), k
    ctx.close()
