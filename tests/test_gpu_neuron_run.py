"""Many neuron steps in one launch (the state on the chip, a grid-wide barrier
per step) against the same steps one call at a time (a launch per step), bit
for bit: networks smaller than a block's share, sizes that are no multiple of
four, the largest the chip holds and one beyond, strong coupling (the steps
depend on each other's spikes).  The launch per step divides with the
division instruction, the long run with the constants' reciprocals: their
results must agree in every bit, also for the constants and the states that
make the long run fall back."""
import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


PARAMS = {"table": {}, "other_divisors": dict(tau_x=7.3, eps=0.93, eta_axon=0.11, eta_dend=-0.35,
                                              x0=-0.07, mu=0.02),
          # a significand of all ones and a middle of zero: the general division
          "general": dict(tau_x=float(np.float32(2.0) - np.float32(2.0) ** -23), eta_dend=-0.7,
                          mu=0.01)}


@pytest.mark.parametrize("name", list(PARAMS))
@pytest.mark.parametrize("n", [1, 3, 4, 7, 255, 257, 1021, 38_913, 622_594, 1_222_500, 1_400_003])
def test_steps_in_one_launch_equal_steps_one_by_one(n, name):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)

    def rand(dtype=torch.float32):
        return torch.rand(n, device="cuda", generator=gen).to(dtype)

    m = 3 * n
    pre, post = (torch.randint(0, n, (m,), dtype=torch.int32, device="cuda", generator=gen)
                 for _ in range(2))
    edges = msp.edge_list(m, pre=pre, post=post, type_=torch.zeros(m, dtype=torch.uint8))
    first = dict(x=0.2 * rand(), refractory=(4 * rand()).to(torch.uint8), calcium=rand(),
                 z_axon=3 * rand(), z_dend_e=3 * rand(), z_dend_i=3 * rand(),
                 spiked=(rand() < 0.3).to(torch.uint8))
    if n > 100:
        # values outside the range of the fast division
        for k, v in (("x", 3e20), ("calcium", float("inf")), ("calcium", float("nan")),
                     ("x", -1e30), ("calcium", 1e-42)):
            first[k][torch.randint(0, n, (3,), device="cuda", generator=gen)] = v
    params = msp.neuron_params(**dict(dict(input_per_spike=0.03), **PARAMS[name]))
    g = msp.MSP(W.default_params(1000.0, seed=11))
    once, by_one = ({k: v.clone() for k, v in first.items()} for _ in range(2))
    g.neuron_steps(90, 7, params, edges, once)
    for k in range(7):
        g.neuron_steps(90 + k, 1, params, edges, by_one)
    torch.cuda.synchronize()
    g.close()
    for k in once:
        a, b = (d[k].cpu().numpy() for d in (once, by_one))
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8)), k
    assert n < 100 or int(once["spiked"].sum()) > 0
