"""The workloads that the library's speed is judged on: what a user has it do,
through its public entry points, from the smallest calls to the largest.

A case is a dict of plain values.  `listed()` holds the named ones, `draw(rng)`
gives another one of the same ranges, `prepare(case, seed)` makes its inputs on
the GPU (or, for the host-buffer call, in pinned host memory) with the context
a program keeps, `run(state)` is one pass, `work(case)` what a pass cannot do
without, and `exact(case, seed)` the computed results in double precision.

Kinds of case:
  noalloc    the all-pairs attraction without a context (direct_noalloc)
  direct     the all-pairs attraction of a built context (MSP.direct)
  step       a plasticity step as separate calls on fixed positions
  ensemble   two networks, one after the other, through one context: every
             build makes a new octree and every attraction new pair lists
  replay     plasticity steps replayed as a CUDA graph
  host       a plasticity step from and to host buffers
  batch      many independent networks in their own frames as one step
  translated the attraction with translated (far) box pairs
  gradient   the derivatives of the attraction
  length     one step of the calibration of sigma: new pair lists, the
             expected synapse length, its derivatives
  neurons    a hundred simulation steps of the neuron side and the update of
             its synapses
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2301_10570_gb300 import msp, workloads as W

SIGMA = W.SIGMA_UM
STD = 1500.0                       # width of a cluster (um)
DENSITY_SIDE = 625.0               # cube side per n^(1/3) of the uniform networks (um)
# the plans the plan chooser picks for the clustered and the uniform networks,
# and the derivatives' plan (no truncation that single precision would see)
CLUSTER_PLAN = dict(leaf_capacity=256, cutoff=3.25, rho_max=0.0, p=4)
UNIFORM_PLAN = dict(leaf_capacity=128, cutoff=3.25, rho_max=0.0, p=4)
GRAD_PLAN = dict(leaf_capacity=128, cutoff=5.0, rho_max=0.0, p=4)
DEFAULT_PLAN = dict(leaf_capacity=32, cutoff=4.0, rho_max=0.25, p=4)
PLANS = dict(cluster=CLUSTER_PLAN, uniform=UNIFORM_PLAN, grad=GRAD_PLAN, default=DEFAULT_PLAN,
             fmm4=dict(leaf_capacity=8, cutoff=4.0, rho_max=0.5, p=4),
             fmm6=dict(leaf_capacity=64, cutoff=3.5, rho_max=0.35, p=6))


def listed():
    return [
        # a program that may not allocate asks for the attraction of a small network
        dict(name="noalloc_1k", kind="noalloc", n=1021),
        # the exact attraction that plans are checked against
        dict(name="direct_131k", kind="direct", n=131_072, clusters=8),
        # the smallest network of the model: one step as separate calls, default plan
        dict(name="step_4k", kind="step", n=4096, clusters=0, plan="default"),
        # networks of an ensemble, searched one after the other with one context
        dict(name="ensemble_2x21k", kind="ensemble", n=21_013, clusters=2, plan="cluster"),
        # the headline: steps of a million clustered neurons as a graph
        dict(name="replay_1m", kind="replay", n=1_048_576, clusters=64, plan="cluster",
             full_build=False, steps=2),
        # the same with the octree rebuilt every step, uniform network
        dict(name="rebuild_262k", kind="replay", n=262_144, clusters=0, plan="uniform",
             full_build=True, steps=2),
        # a simulator whose state lives on the host
        dict(name="host_262k", kind="host", n=262_144, clusters=16, plan="cluster"),
        # a population of networks of many sizes and widths as one step
        dict(name="batch_48", kind="batch", networks=48, smallest=1024, largest=20_000),
        # the expansions: fourth order at the model's density
        dict(name="translated_65k", kind="translated", n=65_536, clusters=0, plan="fmm4"),
        # one pass of gradient descent on the dendritic weights
        dict(name="gradient_262k", kind="gradient", n=262_144, clusters=16, plan="grad"),
        # one step of the calibration of sigma against a synapse length
        dict(name="length_131k", kind="length", n=131_072, clusters=8, plan="grad"),
        # the simulation between two synapse searches
        dict(name="neurons_1m", kind="neurons", n=1_048_576, edges_per_neuron=1.5, steps=100),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def shape(lo, hi):
        n = size(lo, hi)
        return dict(n=n, clusters=rng.choice([0, max(1, n // 16_384)]))

    def planned(lo, hi, default=False):
        c = shape(lo, hi)
        c["plan"] = "cluster" if c["clusters"] else "uniform"
        if default and rng.random() < 0.3:
            c["plan"] = "default"
        return c

    kind = rng.choice(["noalloc", "direct", "step", "ensemble", "replay", "replay", "host", "batch",
                       "translated", "gradient", "length", "neurons"])
    if kind == "noalloc":
        return dict(kind=kind, n=size(64, 65_536))
    if kind == "direct":
        return dict(kind=kind, **shape(1000, 131_072))
    if kind == "step":
        return dict(kind=kind, **planned(1000, 262_144, default=True))
    if kind == "ensemble":
        return dict(kind=kind, **planned(1000, 131_072, default=True))
    if kind == "replay":
        return dict(kind=kind, **planned(4096, 700_000), full_build=rng.random() < 0.5, steps=2)
    if kind == "host":
        return dict(kind=kind, **planned(1000, 262_144))
    if kind == "batch":
        return dict(kind=kind, networks=rng.randint(5, 48), smallest=size(300, 1500),
                    largest=size(2000, 20_000))
    if kind == "translated":
        c = shape(4096, 65_536)
        c["plan"] = "fmm6" if c["clusters"] else "fmm4"
        return dict(kind=kind, **c)
    if kind == "gradient":
        return dict(kind=kind, **shape(1000, 262_144), plan="grad")
    if kind == "length":
        return dict(kind=kind, **shape(1000, 131_072), plan="grad")
    return dict(kind=kind, n=size(10_000, 1_048_576), edges_per_neuron=round(rng.uniform(0.5, 4.0), 2),
                steps=rng.choice([10, 50, 100]))


# -- inputs ---------------------------------------------------------------------

def _network(case, seed):
    """The network of a case: uniform at the model's density, or Gaussian
    clusters at the cluster spacing of the million-neuron network."""
    n, plan = case["n"], PLANS[case.get("plan", "uniform")]
    k = case.get("clusters", 0)
    if k == 0:
        edge = n ** (1.0 / 3.0)
        w = W.uniform_cube(n, DENSITY_SIDE * edge, int(seed), **plan)
        if case["kind"] == "translated":
            # a domain whose finest expanded boxes are as wide as the neurons' spacing
            w.params["side"] = DENSITY_SIDE * 2.0 ** math.ceil(math.log2(edge) - 1e-9)
    else:
        side = 100_000.0 * (k / 64.0) ** (1.0 / 3.0)
        w = W.clustered(k, -(-n // k), side, STD, min(4500.0, side / 4), int(seed), **plan)
        w = w if w.n == n else W.subset(w, np.arange(n))
    w.params["seed"] = int(seed) & 0xffffffff          # the draws' key
    return w


def _batch(case, seed):
    k = case["networks"]
    sizes = np.geomspace(case["smallest"], case["largest"], k).astype(np.int64)
    sigmas = np.linspace(300.0, 1500.0, k)[np.random.default_rng(3).permutation(k)]
    return W.batch(sizes, sigmas, ["clustered" if j % 2 else "uniform" for j in range(k)],
                   seed=int(seed))


def _selection(n):
    """Output buffers of the selection for n neurons of at most three vacant
    axonal elements, kept from step to step."""
    ne = 3 * n
    return dict(partner=torch.full((ne,), -1, dtype=torch.int32, device="cuda"),
                syn_pre=torch.zeros(ne, dtype=torch.int32, device="cuda"),
                syn_post=torch.zeros(ne, dtype=torch.int32, device="cuda"),
                syn_type=torch.zeros(ne, dtype=torch.uint8, device="cuda"),
                n_syn=torch.zeros(1, dtype=torch.int64, device="cuda"))


def _capture(s):
    """Build, attraction and capture of the step graph on the state's buffers."""
    g = s["ctx"]
    g.build_tree(s["pos"], s["type"], *s["vac"])
    g.attraction()
    g.step_graph_set_full_build(s["full_build"])
    s["out"] = g.step_graph_capture(s["pos"], s["type"], *s["vac"], first_step=s["step"])
    for k in ("partner", "syn_pre", "syn_post", "syn_type"):
        s["out"][k].zero_()


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, step=0)
    if kind == "neurons":
        return _prepare_neurons(case, seed, s)
    if kind == "batch":
        b = _batch(case, seed)
        pos, t, a, e, i = msp.to_device(b)
        local, side, level = msp.batch_layout(pos, b.offsets, b.sigma, 4.0,
                                              CLUSTER_PLAN["leaf_capacity"])
        params = W.default_params(side, sigma=1.0, seed=int(seed) & 0xffffffff, **CLUSTER_PLAN)
        s["ctx"] = msp.MSP(params, frames=(b.offsets, level))
        s["nets"] = [((local, t, a, e, i), _selection(b.n))]
        return s
    if kind == "ensemble":
        nets = [_network(case, 2 * int(seed) + j) for j in range(2)]
        s["ctx"] = msp.MSP(nets[0].params)
        s["nets"] = [(msp.to_device(w), _selection(w.n)) for w in nets]
        return s
    w = _network(case, seed)
    if kind == "host":
        def pinned(a):
            return torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()

        def zeros(n, dtype):
            return pinned(np.zeros(max(int(n), 1), dtype))
        ne = 3 * w.n
        s["ctx"] = msp.MSP(w.params)
        s["arrays"] = [pinned(v) for v in w.arrays()]
        s["out"] = dict(u=zeros(w.n, np.float32), partner=zeros(ne, np.int32),
                        syn_pre=zeros(ne, np.int32), syn_post=zeros(ne, np.int32),
                        syn_type=zeros(ne, np.uint8), n_syn=zeros(1, np.int64))
        return s
    pos, t, a, e, i = msp.to_device(w)
    if kind == "noalloc":
        s["args"] = (pos, t, a, e, i, SIGMA)
        return s
    s["ctx"] = g = msp.MSP(w.params)
    rng = np.random.default_rng(int(seed) + 1)
    if kind == "direct":
        g.build_tree(pos, t, a, e, i)
    elif kind in ("step", "translated"):
        s["nets"] = [((pos, t, a, e, i), _selection(w.n))]
    elif kind == "replay":
        s.update(pos=pos, type=t, vac=[a, e, i], full_build=bool(case["full_build"]),
                 steps=case["steps"])
        _capture(s)
    elif kind == "gradient":
        # the lists of the derivatives come from the positions alone
        ones = torch.ones_like(a)
        g.build_tree(pos, t, ones, ones, ones)
        g.attraction()
        s["args"] = (t, a, e, i)
        s["g"] = torch.from_numpy(rng.normal(size=w.n).astype(np.float32)).cuda()
    elif kind == "length":
        ones = torch.ones_like(a)
        g.build_tree(pos, t, ones, ones, ones)
        s["args"] = (t, a) + tuple(torch.from_numpy(rng.uniform(0.2, 3.0, w.n).astype(np.float32))
                                   .cuda() for _ in range(2))
    return s


def _prepare_neurons(case, seed, s):
    """Neurons at rest with calcium spread over the growth curve and random
    synapses; the elements cover them with a spread margin, so that every
    update deletes some synapses."""
    n = case["n"]
    m = int(case["edges_per_neuron"] * n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))

    def rand():
        return torch.rand(n, device="cuda", generator=gen)

    pre, post = (torch.randint(0, n, (m,), dtype=torch.int32, device="cuda", generator=gen)
                 for _ in range(2))
    typ = (rand() >= 0.8).to(torch.uint8)[pre.long()]

    def bound(idx):
        return torch.bincount(idx.long(), minlength=n).float()

    s["state"] = dict(
        x=torch.full((n,), 0.065, device="cuda"),
        refractory=torch.zeros(n, dtype=torch.uint8, device="cuda"),
        calcium=0.3 + 0.5 * rand(), z_axon=bound(pre) + 4.0 * rand(),
        z_dend_e=bound(post[typ == 0]) + 4.0 * rand(), z_dend_i=bound(post[typ == 1]) + 4.0 * rand(),
        spiked=(rand() < 0.05).to(torch.uint8))
    s["edges"] = msp.edge_list(m + m // 2 + 16, pre=pre, post=post, type_=typ)
    s["vac"] = [torch.zeros(n, dtype=torch.uint8, device="cuda") for _ in range(3)]
    s["params"], s["steps"] = msp.neuron_params(), case["steps"]
    s["ctx"] = msp.MSP(W.default_params(100_000.0, seed=int(seed) & 0xffffffff))
    return s


# -- one pass ---------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "noalloc":
        return msp.direct_noalloc(*s["args"])
    g = s["ctx"]
    if kind == "direct":
        return g.direct()
    if kind in ("step", "ensemble", "batch"):
        s["step"] += 1
        res = []
        for net, sel in s["nets"]:
            g.build_tree(*net)
            u = g.attraction()
            g.select_partners(s["step"], out=sel)
            res.append(dict(u=u, **sel))
        return res
    if kind == "translated":
        g.build_tree(*s["nets"][0][0])
        return g.attraction()
    if kind == "replay":
        first = s["step"]
        try:
            g.step_graph_launch(s["steps"])
        except msp.MSPError as e:
            if msp.STATUS.get(e.code) != "MSP_ERR_NOT_BUILT":
                raise
            # another context's workspace changed since the capture: capture again
            _capture(s)
            g.step_graph_launch(s["steps"])
        nxt, _ = g.step_graph_finish()
        s["step"] = g.run_steps(nxt, first + s["steps"] - nxt)
        return dict(vac=s["vac"], **{k: v for k, v in s["out"].items() if k != "history"})
    if kind == "host":
        s["step"] += 1
        return g.plasticity_step_host(s["step"], *s["arrays"], out=s["out"])
    if kind == "gradient":
        return g.attraction_grad(*s["args"], g=s["g"])
    if kind == "length":
        g.set_sigma(SIGMA)
        g.attraction()
        return g.length_loss(*s["args"], target=1000.0)
    g.neuron_steps(s["step"], s["steps"], s["params"], s["edges"], s["state"])
    s["step"] += s["steps"]
    g.update_synapses(s["step"], s["state"], s["edges"], *s["vac"])
    return dict(state=s["state"], vac=s["vac"],
                edges={k: s["edges"][k] for k in ("pre", "post", "type", "n")})


# -- what a pass cannot do without --------------------------------------------------

def _within(case, n, k, cutoff):
    """Neurons within the cutoff radius of a neuron, on average: Gaussian
    clusters (distances are chi with 3 degrees of freedom, scale sqrt(2) std),
    or the uniform density."""
    r = cutoff * SIGMA
    if k == 0:
        return min(n, 4.0 / 3.0 * math.pi * r ** 3 / DENSITY_SIDE ** 3)
    x = r / STD
    return n / k * (math.erf(x / 2) - x / math.sqrt(math.pi) * math.exp(-x * x / 4))


# per neuron: positions, type and three vacant counts read; u, and per element
# (1.5 a neuron) the partner and one synapse of three written
_STEP_BYTES = 16 + 4 + 1.5 * 4 + 0.5 * 9
# operations of one term w exp(-r^2 / sigma^2): three differences, r^2, the
# scale, the exponential and the sum
_TERM = 10


def work(case):
    kind = case["kind"]
    active = 0.75                                   # three of four neurons have vacant axons
    if kind == "batch":
        b = np.geomspace(case["smallest"], case["largest"], case["networks"]).astype(np.int64)
        n = float(b.sum())
        return dict(bytes=n * _STEP_BYTES, flops=active * _TERM * n * 300.0)
    n = float(case["n"])
    k = case.get("clusters", 0)
    cut = PLANS[case.get("plan", "uniform")]["cutoff"]
    near = active * n * _within(case, n, k, cut)
    if kind in ("noalloc", "direct"):
        return dict(bytes=20.0 * n, flops=active * _TERM * n * n)
    if kind == "step":
        return dict(bytes=n * _STEP_BYTES, flops=_TERM * near)
    if kind == "ensemble":
        return dict(bytes=2 * n * _STEP_BYTES, flops=2 * _TERM * near)
    if kind == "replay":
        # the vacant counts are also written; a rebuilt octree needs its sorted copy
        per = _STEP_BYTES + 6.0 + (16.0 if case["full_build"] else 0.0)
        return dict(bytes=case["steps"] * n * per, flops=case["steps"] * _TERM * near)
    if kind == "host":
        return dict(bytes=n * _STEP_BYTES, flops=_TERM * near)
    if kind == "translated":
        return dict(bytes=20.0 * n, flops=_TERM * near)
    if kind == "gradient":
        # two sums per target, one per source
        return dict(bytes=(20.0 + 4 + 16) * n, flops=2 * (_TERM + 2) * near)
    if kind == "length":
        return dict(bytes=(14.0 + 8 + 8) * n, flops=2 * (_TERM + 6) * near)
    # neuron state: five floats and two bytes read and written each step, the
    # input counts; the edges read twice and written once
    m = case["edges_per_neuron"] * n
    return dict(bytes=case["steps"] * 44.0 * n + 27.0 * m, flops=case["steps"] * 120.0 * n)


# -- the results in double precision --------------------------------------------------

def _blocks(pos, sigma, rows):
    """For blocks of targets: (slice, squared distances, kernel without the
    neuron itself) against every neuron, in double precision."""
    p = (pos.double() - pos.double().mean(dim=1, keepdim=True)).t().contiguous() / sigma
    q = (p * p).sum(1)
    for a in range(0, p.shape[0], rows):
        b = min(a + rows, p.shape[0])
        r2 = torch.addmm(q[None, :], p[a:b], p.t(), alpha=-2.0).add_(q[a:b, None]).clamp_(min=0.0)
        j = torch.arange(a, b, device=p.device)
        K = torch.exp(-r2)
        K[j - a, j] = 0.0
        r2[j - a, j] = 0.0
        yield slice(a, b), r2, K


def _rows(n):
    return max(1, min(n, (1 << 29) // max(n, 1)))


def _exact_u(pos, t, a, e, i, sigma=SIGMA):
    w = torch.stack([e, i], 1).double()
    u = torch.empty(pos.shape[1], dtype=torch.float64, device=pos.device)
    for sl, _, K in _blocks(pos, sigma, _rows(pos.shape[1])):
        u[sl] = (K @ w).gather(1, t[sl].long()[:, None])[:, 0]
    return torch.where(a > 0, u, torch.zeros_like(u))


def exact(case, seed):
    """Double precision sums over all neurons.  Drawn partners and synapses
    are whole numbers and have no such value; nor has the neuron side, whose
    spikes are decided by its single precision arithmetic."""
    kind = case["kind"]
    none = dict(partner=None, n_syn=None, syn_pre=None, syn_post=None, syn_type=None)
    if kind in ("replay", "neurons"):
        return None
    if kind == "batch":
        b = _batch(case, seed)
        d = msp.to_device(b)
        parts = []
        for k in range(case["networks"]):
            sl = slice(int(b.offsets[k]), int(b.offsets[k + 1]))
            parts.append(_exact_u(d[0][:, sl], *[v[sl] for v in d[1:]], sigma=float(b.sigma[k])))
        return [dict(u=torch.cat(parts), **none)]
    if kind == "ensemble":
        return [dict(u=_exact_u(*msp.to_device(_network(case, 2 * int(seed) + j))), **none)
                for j in range(2)]
    w = _network(case, seed)
    pos, t, a, e, i = msp.to_device(w)
    if kind in ("noalloc", "direct", "translated"):
        return _exact_u(pos, t, a, e, i)
    if kind == "step":
        return [dict(u=_exact_u(pos, t, a, e, i), **none)]
    if kind == "host":
        return dict(u=_exact_u(pos, t, a, e, i).cpu().numpy(), **none)
    n, act, ty = w.n, a > 0, t.long()[:, None]
    rng = np.random.default_rng(int(seed) + 1)
    if kind == "gradient":
        g = torch.from_numpy(rng.normal(size=n).astype(np.float32)).cuda().double() * act
        wt = torch.stack([e, i], 1).double()
        gt = torch.stack([g * (t == 0), g * (t != 0)], 1)
        u, du, gw = torch.zeros_like(g), torch.zeros_like(g), torch.zeros_like(gt)
        for sl, r2, K in _blocks(pos, SIGMA, _rows(n)):
            u[sl] = (K @ wt).gather(1, ty[sl])[:, 0]
            gw += K.t() @ gt[sl]
            du[sl] = (K.mul_(r2) @ wt).gather(1, ty[sl])[:, 0] * (2.0 / SIGMA)
        return dict(u=u * act, du_dsigma=du * act, grad_w_e=gw[:, 0], grad_w_i=gw[:, 1])
    # the expected synapse length and its derivatives
    wt = torch.stack([torch.from_numpy(rng.uniform(0.2, 3.0, n).astype(np.float32)).cuda()
                      for _ in range(2)], 1).double()
    u, v, du, dv = (torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(4))
    for sl, r2, K in _blocks(pos, SIGMA, _rows(n)):
        r = r2.sqrt() * SIGMA
        for out, f in ((u, None), (v, r), (du, r2), (dv, r2 * r)):
            out[sl] = ((K if f is None else K * f) @ wt).gather(1, ty[sl])[:, 0]
    du, dv = du * (2.0 / SIGMA), dv * (2.0 / SIGMA)
    ok = act & (u > 0)
    us, ad = torch.where(ok, u, torch.ones_like(u)), torch.where(ok, a.double(), 0.0)
    A = ad.sum()
    m = (ad * v / us).sum() / A
    dm = (ad * (dv * us - v * du) / (us * us)).sum() / A
    f = 2.0 * (m - 1000.0)
    al, be = f * ad / (A * us), f * ad * v / (A * us * us)
    G = torch.zeros(n, 2, dtype=torch.float64, device="cuda")
    ch = torch.stack([t == 0, t != 0], 1).double()
    for sl, r2, K in _blocks(pos, SIGMA, _rows(n)):
        G += (K * (r2.sqrt() * SIGMA)).t() @ (ch[sl] * al[sl, None]) - K.t() @ (ch[sl] * be[sl, None])
    return dict(loss=float((m - 1000.0) ** 2), mean=float(m), dloss_dsigma=float(f * dm),
                dmean_dsigma=float(dm), gE=G[:, 0], gI=G[:, 1])
