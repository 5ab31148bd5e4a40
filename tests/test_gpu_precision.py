"""How far single precision sums that many warps share are from 64 bits, on the
workloads of perf/cases.py: no further than with one target per lane and four warps
a leaf, the kernels before many warps shared a target.  The bars are those
kernels' errors on the same inputs (relative, over all outputs, the mean of three
seeds), a few per cent up."""
import importlib.util
import os

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_spec = importlib.util.spec_from_file_location("cases", os.path.join(ROOT, "perf", "cases.py"))
cases = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(cases)

BARS = {
    # 16 warps share an all-pairs target: 6.66e-8 before, 8.52e-8 added in order
    "all_pairs": (dict(kind="noalloc", n=15_000), dict(u=6.7e-8)),
    # 16 warps share a leaf: 1.634e-7 before, 1.706e-7 added in order
    "near_field": (dict(kind="step", n=5000, clusters=2, plan="cluster"), dict(u=1.66e-7)),
    # signed sums of lanes and warps: 3.47e-7 and 3.92e-7 before, 3.42e-7 and 4.50e-7
    # joined plainly
    "length": (dict(kind="length", n=20_000, clusters=2, plan="grad"), dict(gE=3.5e-7, gI=4.0e-7)),
}


@pytest.mark.parametrize("name", list(BARS))
def test_error_against_64_bits(name):
    case, bars = BARS[name]
    errors = {k: [] for k in bars}
    for seed in (3, 4, 5):
        state = cases.prepare(case, seed)
        got, want = cases.run(state), cases.exact(case, seed)
        if case["kind"] == "noalloc":
            got, want = dict(u=got), dict(u=want)
        elif case["kind"] == "step":
            got, want = got[0], want[0]
        for k in bars:
            a, b = got[k].double(), torch.as_tensor(want[k], dtype=torch.float64, device="cuda")
            errors[k].append(float((a - b).norm() / b.norm()))
        del state
    for k, bar in bars.items():
        assert sum(errors[k]) / 3 <= bar, (k, errors[k])
