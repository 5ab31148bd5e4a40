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


# one block, the largest size of the one-launch kernel and the next, both sides of
# the change of targets per lane
@pytest.mark.parametrize("n", [31, 1021, 8192, 8193, 40_001])
@pytest.mark.parametrize("over", ["x", "z", "between"])
def test_all_pairs_written_over_the_positions(n, over):
    w = W.uniform_cube(n, 625.0 * n ** (1 / 3), seed=n)
    w.vac_axon[::5] = 0
    pos, t, a, e, i = msp.to_device(w)
    want = msp.direct_noalloc(pos, t, a, e, i, w.params["sigma"])
    work = pos.clone()
    flat = work.view(-1)
    out = {"x": work[0], "z": work[2], "between": flat[n // 2:n // 2 + n]}[over]
    got = msp.direct_noalloc(work, t, a, e, i, w.params["sigma"], out=out)
    assert got.data_ptr() == out.data_ptr() and torch.equal(got, want)


def test_all_pairs_written_over_the_counts():
    n = 3001
    w = W.uniform_cube(n, 9000.0, seed=5)
    pos, t, a, e, i = msp.to_device(w)
    want = msp.direct_noalloc(pos, t, a, e, i, w.params["sigma"])
    room = torch.empty(n, dtype=torch.float32, device="cuda")
    counts = room.view(torch.uint8)[:4 * n].view(4, n)      # the four arrays in u's own bytes
    for k, v in enumerate((t, a, e, i)):
        counts[k] = v
    got = msp.direct_noalloc(pos, *counts, w.params["sigma"], out=room)
    assert torch.equal(got, want)
