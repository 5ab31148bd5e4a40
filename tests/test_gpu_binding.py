"""Every layout that the binding accepts gives the result of the contiguous
arrays, exactly: rows of a wider or longer tensor, a transposed one, columns
with a stride, a storage offset; given and own output buffers; a side stream."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402

LAYOUTS = {
    "contiguous": lambda p: p,
    "four_rows": lambda p: torch.cat([p, p[:1]]),
    "rows_of_wider": lambda p: torch.cat([p, p], 1)[:, :p.shape[1]],
    "transposed": lambda p: p.t().contiguous().t(),
    "strided": lambda p: p.repeat_interleave(2, 1)[:, ::2],
    "offset": lambda p: torch.cat([p.new_zeros(1), p.reshape(-1)])[1:].view(3, -1)}


@pytest.mark.parametrize("n", [1, 1023])
@pytest.mark.parametrize("layout", list(LAYOUTS))
def test_layouts_of_the_positions(layout, n):
    w = W.uniform_cube(n, 3000.0, seed=n, cutoff=4.0)
    pos, *counts = msp.to_device(w)
    given = LAYOUTS[layout](pos)
    wide = [torch.stack([c, c], 1)[:, 0] for c in counts]
    res = []
    for p, c in ((pos, counts), (given, wide)):
        g = msp.MSP(w.params)
        g.build_tree(p, *c)
        u = g.attraction()
        sel = g.select_partners(3)
        out = {k: torch.full_like(v, 7) for k, v in sel.items()}
        assert g.select_partners(3, out=out) is out
        m = int(sel["n_syn"])
        r = [u, sel["partner"], out["partner"], out["n_syn"]] + [
            s[k][:m] for s in (sel, out) for k in ("syn_pre", "syn_post", "syn_type")]
        if p.shape[0] == 3:
            r += [msp.direct_noalloc(p, *c, 750.0)]
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                r += [msp.direct_noalloc(p, *c, 750.0)]
            r += [msp.direct_noalloc(p, *c, 750.0, out=torch.empty_like(u), stream=side)]
            side.synchronize()
        res.append([v.cpu().numpy() for v in r])
        g.close()
    assert np.array_equal(res[0][1], res[0][2])
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_host_step_takes_strided_arrays():
    w = W.uniform_cube(500, 3000.0, seed=1, cutoff=4.0)
    res = []
    for arrays in (w.arrays(), [np.repeat(v, 2, -1)[..., ::2] for v in w.arrays()]):
        g = msp.MSP(w.params)
        res.append(g.plasticity_step_host(2, *arrays))
        g.close()
    assert all(np.array_equal(res[0][k], res[1][k]) for k in res[0])
