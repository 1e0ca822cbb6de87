"""NaN positions in the adaptive near field of the mixed-precision modes: they show in
the potentials they belong to, and in no others.

One leaf, so every pair is a near-field pair and x == y is the only pair left out.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["laplace", "yukawa", "biharmonic"])
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
def test_nan_positions(kernel, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(3)
    src = torch.tensor(rng.random((50, 3)), device="cuda")
    tgt = torch.tensor(rng.random((40, 3)), device="cuda")
    tgt[0] = src[0]  # a pair left out
    w = torch.tensor(rng.uniform(0.5, 1.0, 50), device="cuda")
    plan = FMM(kernel, d=3, p=6, levels=-6, max_leaf=200, precision=precision,
               lam=1.0 if kernel == "yukawa" else 0.0)
    good = plan.eval(src, w, tgt, check_status=True)
    assert bool(torch.isfinite(good).all())
    bad = tgt.clone()
    bad[7, 1] = float("nan")
    got = plan.eval(src, w, bad)
    # (the points keep their order in the one leaf, so the others' sums are the same)
    keep = torch.arange(40, device="cuda") != 7
    assert bool(torch.isnan(got[7]))
    assert float((got[keep] - good[keep]).norm() / good[keep].norm()) < 1e-6
    src[3, 2] = float("nan")
    assert bool(torch.isnan(plan.eval(src, w, tgt)).all())
