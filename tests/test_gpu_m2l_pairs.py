"""The tensor-core M2L's launch shapes: CTA pairs, stacked classes, packed K
tails, split walks and gathered rows, against the CPU oracle on the same tree.

Tolerances are the precisions' own (relative L2 against the oracle): 5e-6 for
F16X3 and TF32X3, 5e-5 for BF16X3.
"""
import numpy as np
import pytest

from paper_2305_17867_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"f16x3": 5e-6, "tf32x3": 5e-6, "bf16x3": 5e-5}


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# |j|: one tile per level alone (level 2), the riding level 2, one and several
# tile pairs; 1, 2, 4 and 8 stacked classes; tails of 1 to 4 packed K steps and
# tails that do not pack; several column blocks
@pytest.mark.parametrize("kernel,p,levels,precision", [
    ("yukawa", 6, 2, "f16x3"),       # 49: four classes, level 2 alone in its pairs
    ("laplace", 4, 2, "tf32x3"),     # 25: eight classes
    ("laplace", 5, 3, "bf16x3"),     # 36 of 48 columns, riding level 2
    ("biharmonic", 6, 4, "bf16x3"),  # 74: tail of 10 (two packed steps), N = 160
    ("biharmonic", 7, 3, "tf32x3"),  # 100: tail of 4 (tf32), one class, N = 128
    ("laplace", 8, 4, "f16x3"),      # 81: tail of 17 (four packed steps)
    ("biharmonic", 8, 4, "f16x3"),   # 130: tail of 2, N = 160 over 144 columns
    ("laplace", 7, 5, "f16x3"),      # 64: no tail; one pair per cluster
    ("biharmonic", 12, 3, "f16x3"),  # 290: two column blocks
    ("laplace", 12, 3, "tf32x3"),    # 169: tail of 9 (tf32), N = 192 over 176 columns
])
def test_uniform_shapes(torch_cuda, oracle, kernel, p, levels, precision):
    torch = torch_cuda
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(900 + 10 * p + levels)
    n = 9000 if levels < 5 else 40000
    src, w = rng.random((n, 3)), rng.uniform(-1.0, 1.0, n)
    idx = np.sort(rng.choice(n, 64, replace=False))
    lam = 1.0 if kernel == "yukawa" else 0.0
    ref = oracle.fmm_uniform(kernel, 3, p, levels, src, w, src, lam=lam, sample=idx)
    plan = FMM(kernel, d=3, p=p, levels=levels, lam=lam, precision=precision)
    s, wd = torch.tensor(src, device="cuda"), torch.tensor(w, device="cuda")
    got = plan.eval(s, wd, check_status=True)
    again = plan.eval(s, wd, check_status=True)
    assert torch.equal(got, again)  # the split walks' sums do not depend on timing
    assert rel_l2(got.cpu().numpy()[idx], ref) < TOL[precision]


@pytest.mark.parametrize("precision", ["tf32x3", "bf16x3"])
def test_gathered_wait_runs_out_and_recovers(torch_cuda, precision):
    # shortened waits on an adaptive tree with gathered levels: every role gives
    # up at its own round, the status says so and the next call is correct
    torch = torch_cuda
    from paper_2305_17867_gb300 import _lib
    from paper_2305_17867_gb300.fmm import FMM

    L = _lib.load()
    rng = np.random.Generator(np.random.PCG64(21))
    src = torch.tensor(W.plummer_points(rng, 20000), device="cuda")
    tgt = torch.tensor(rng.random((6000, 3)), device="cuda")
    w = torch.tensor(rng.normal(size=20000), device="cuda")
    plan = FMM("laplace", d=3, p=8, levels=-10, precision=precision, max_leaf=32)
    ref = plan.eval(src, w, tgt, check_status=True)
    torch.cuda.synchronize()
    assert L.fmm_set_wait_limit(plan._h, 1) == 0
    plan.eval(src, w, tgt)
    assert plan.last_status() == -5  # FMM_ERR_TIMEOUT
    assert L.fmm_set_wait_limit(plan._h, 0) == 0
    again = plan.eval(src, w, tgt, check_status=True)
    torch.cuda.synchronize()
    assert float(torch.linalg.norm(again - ref) / torch.linalg.norm(ref)) < 1e-12
