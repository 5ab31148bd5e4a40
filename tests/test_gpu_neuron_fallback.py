"""Neuron steps where the device refuses the cooperative launch that takes many
steps at once: the steps are launched one by one, with the same results."""
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


@pytest.mark.parametrize("n", [257, 40_003])
def test_refused_launch_goes_step_by_step(n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n)

    def rand():
        return torch.rand(n, device="cuda", generator=gen)

    pre, post = (torch.randint(0, n, (3 * n,), dtype=torch.int32, device="cuda", generator=gen)
                 for _ in range(2))
    edges = msp.edge_list(3 * n, pre=pre, post=post,
                          type_=torch.zeros(3 * n, dtype=torch.uint8))
    first = dict(x=0.2 * rand(), refractory=(4 * rand()).to(torch.uint8), calcium=rand(),
                 z_axon=3 * rand(), z_dend_e=3 * rand(), z_dend_i=3 * rand(),
                 spiked=(rand() < 0.3).to(torch.uint8))
    params = msp.neuron_params(input_per_spike=0.03)
    g = msp.MSP(W.default_params(1000.0, seed=11))
    states, launches = [], []
    for refuse in (False, True, False):
        g.selftest_refuse_cooperative(refuse)
        before = g.stats()["kernel_launches"]
        state = {k: v.clone() for k, v in first.items()}
        g.neuron_steps(90, 9, params, edges, state)
        torch.cuda.synchronize()
        launches.append(g.stats()["kernel_launches"] - before)
        states.append(state)
    g.close()
    assert launches[1] == launches[0] + 8 and launches[2] == launches[0]
    for s in states[1:]:
        for k, v in s.items():
            assert torch.equal(v, states[0][k]), k


def test_a_hub_of_many_edges_is_waited_for():
    # a neuron that spikes in every step with ten million outgoing edges: its
    # block is busy with them for half a second a step while the others wait
    n, m = 1024, 10_000_000
    post = torch.arange(m, device="cuda", dtype=torch.int32) % n
    edges = msp.edge_list(m, pre=torch.full_like(post, 5), post=post,
                          type_=torch.zeros(m, dtype=torch.uint8))
    first = {k: torch.zeros(n, device="cuda") for k in ("x", "calcium", "z_axon", "z_dend_e",
                                                        "z_dend_i")}
    first["x"][5] = 1e6
    first.update({k: torch.zeros(n, dtype=torch.uint8, device="cuda")
                  for k in ("refractory", "spiked")})
    params = msp.neuron_params(input_per_spike=1e-9, refractory=0, tau_x=1e9)
    w = W.uniform_cube(100, 1000.0, seed=1)
    g = msp.MSP(w.params)
    once, by_one = ({k: v.clone() for k, v in first.items()} for _ in range(2))
    g.neuron_steps(0, 3, params, edges, once)
    g.build_tree(*msp.to_device(w))          # synchronises: reports a wait that gave up
    for k in range(3):
        g.neuron_steps(k, 1, params, edges, by_one)
    torch.cuda.synchronize()
    g.close()
    assert int(once["spiked"][5]) == 1
    for k, v in once.items():
        assert torch.equal(v, by_one[k]), k
