"""Gathered levels of the adaptive tensor-core M2L: the source rows that one CTA of
a pair copies are read by MMAs that the other CTA issues.

A row read before its copy had landed would leave a stage's previous contents
in the product: wrong by far more than the tolerance, and by another amount
in the next call.  So the same call is repeated beside memory traffic on
another stream and has to give the same bits each time, and agree with FP64
within the precision's tolerance on adaptive trees (2e-5, 1e-4; bf16's pair of
8-bit significands).
"""
import numpy as np
import pytest

from paper_2305_17867_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"tf32x3": 2e-5, "bf16x3": 1e-4}


@pytest.mark.parametrize("kernel,p,precision,n", [
    ("yukawa", 8, "tf32x3", 60000),   # 81 coefficients: several chunks of K
    ("laplace", 5, "bf16x3", 20000),  # 36: one chunk, a packed tail
    ("laplace", 12, "bf16x3", 30000),
])
def test_gathered_rows_are_complete(kernel, p, precision, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.Generator(np.random.PCG64(210 + p))
    src = torch.tensor(W.plummer_points(rng, n), device="cuda")
    tgt = torch.tensor(rng.random((n // 2, 3)), device="cuda")
    w = torch.tensor(rng.normal(size=n), device="cuda")
    opt = dict(d=3, p=p, levels=-10, max_leaf=32, lam=1.0 if kernel == "yukawa" else 0.0)
    ref = FMM(kernel, precision="fp64", **opt).eval(src, w, tgt, check_status=True)
    plan = FMM(kernel, precision=precision, **opt)
    first = plan.eval(src, w, tgt, check_status=True)
    assert float((first - ref).norm() / ref.norm()) < TOL[precision]
    a = torch.zeros(32 << 20, device="cuda")
    b = torch.empty_like(a)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(8):
        with torch.cuda.stream(side):
            for _ in range(20):
                b.copy_(a)
        assert torch.equal(plan.eval(src, w, tgt), first)
    torch.cuda.synchronize()
    assert plan.last_status() == 0
