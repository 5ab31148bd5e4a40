"""Several contexts on one device, in turn and from several threads: what one
context's launches ask of a kernel (shared memory that follows the expansion
order or the number of neurons) must not fail another's."""
import threading

import numpy as np
import pytest

from paper_2301_10570_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2301_10570_gb300 import msp  # noqa: E402


def _in_threads(jobs):
    """Runs the jobs at the same time; raises the first failure."""
    failed = []

    def guarded(job):
        try:
            job()
        except BaseException as e:                        # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=guarded, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if failed:
        raise failed[0]


def test_grouped_translations_of_two_orders_in_turn():
    nets = {p: W.uniform_cube(4000, 9000.0, seed=3, leaf_capacity=16, rho_max=0.5, cutoff=4.0, p=p,
                              centre_mode=1) for p in (5, 4)}
    ctx = {p: msp.MSP(w.params) for p, w in nets.items()}
    first = {}
    for p in (5, 4, 5, 4):
        ctx[p].build_tree(*msp.to_device(nets[p]))
        u = ctx[p].attraction()
        assert ctx[p].stats()["n_far"] > 0
        assert torch.equal(first.setdefault(p, u), u)
    for c in ctx.values():
        c.close()


def test_selections_of_two_orders_at_the_same_time():
    def job(p):
        w = W.uniform_cube(2000, 6000.0, seed=p, rho_max=0.25, cutoff=4.0, p=p)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            g = msp.MSP(w.params)
            g.build_tree(*msp.to_device(w))
            g.attraction()
            want = g.select_partners(5)["partner"].clone()
            for _ in range(200):
                assert torch.equal(g.select_partners(5)["partner"], want)
            g.close()

    _in_threads([lambda p=p: job(p) for p in (5, 6, 7, 8)])


def test_neuron_steps_of_two_sizes_at_the_same_time():
    params = msp.neuron_params(input_per_spike=0.03)

    def job(n):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            gen = torch.Generator(device="cuda")
            gen.manual_seed(n)
            g = msp.MSP(W.default_params(1000.0, seed=11))
            none = torch.zeros(1, dtype=torch.int32)
            edges = msp.edge_list(1, pre=none, post=none, type_=none.to(torch.uint8))
            state = {k: torch.rand(n, device="cuda", generator=gen)
                     for k in ("x", "calcium", "z_axon", "z_dend_e", "z_dend_i")}
            state.update({k: torch.zeros(n, dtype=torch.uint8, device="cuda")
                          for k in ("refractory", "spiked")})
            for k in range(200):
                g.neuron_steps(2 * k, 2, params, edges, state)
            stream.synchronize()
            g.close()

    _in_threads([lambda n=n: job(n) for n in (400_000, 700_000, 1_100_000)])
