"""Roots far from the origin: the mixed-precision uniform plans on float64 points that
are no float32 values.

The box-relative coordinates have to be as exact there as near the origin: the
same points, moved by a shift, against the FP64 evaluation of the moved
points, within the FP32 mode's 2e-6 (5e-6 with the three-product tensor-core
M2L).  Shifts on both sides of the reach of the float pairs, (|x| + |lo|)/s =
2^14, at the depth used here.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-6, "f16x3": 5e-6}


@pytest.mark.parametrize("precision", ["fp32", "f16x3"])
@pytest.mark.parametrize("shift", [100.0, -300.0, 1e4, -1e6, 1e7, 3e8])
def test_shifted_root(precision, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(31)
    n = 60000
    x = shift + rng.random((n, 3))  # rounded to float64 once, here
    src = torch.tensor(x, device="cuda")
    w = torch.tensor(rng.uniform(-1.0, 1.0, n), device="cuda")
    opt = dict(d=3, p=8, levels=5, root_lo=[shift] * 3, root_size=1.0)
    ref, gref = FMM("laplace", precision="fp64", m2l="auto", **opt).eval(src, w, grad=True)
    got, ggot = FMM("laplace", precision=precision, m2l="auto", **opt).eval(src, w, grad=True)
    assert float((got - ref).norm() / ref.norm()) < TOL[precision]
    assert float((ggot - gref).norm() / gref.norm()) < TOL[precision]
