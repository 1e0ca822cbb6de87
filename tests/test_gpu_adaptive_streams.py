"""The adaptive leaf pass in its float form: near field and M2P beside the
passes over the expansions, the far field of four boxes to a warp.

Against the FP64 evaluation of the same tree, within 2e-5, the tolerance of
the three-product tf32 M2L against FP64: a leaf left out or a target given
another leaf's expansion changes the result by more than 1e-3.  Orders with an
unrolled far field and without, leaves of a few points (groups of four that
cross a level and hold boxes that are not leaves), trees without a far field,
more targets than lanes, and a caller's stream with other work around the call.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.mark.parametrize("kernel,p,n,m,max_leaf", [
    ("laplace", 5, 3000, 900, 3), ("laplace", 8, 3001, 0, 7), ("biharmonic", 7, 4000, 0, 40),
    ("yukawa", 12, 6000, 2500, 20), ("laplace", 6, 2500, 2500, 200), ("laplace", 4, 5, 3, 2),
    ("yukawa", 8, 40, 1, 64), ("laplace", 10, 1, 70, 1), ("laplace", 3, 3000, 900, 5),
    ("yukawa", 9, 3000, 0, 30), ("laplace", 11, 2000, 500, 12),
])
def test_float_leaf_pass(kernel, p, n, m, max_leaf):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(n + 31 * p)
    src = torch.tensor(rng.random((n, 3)) ** 2, device="cuda")  # denser towards the corner
    tgt = torch.tensor(rng.random((m, 3)), device="cuda") if m else None
    w = torch.tensor(rng.uniform(-1.0, 1.0, n), device="cuda")
    opt = dict(d=3, p=p, levels=-8, max_leaf=max_leaf, lam=1.3 if kernel == "yukawa" else 0.0)
    ref = FMM(kernel, precision="fp64", **opt).eval(src, w, tgt, check_status=True)
    plan = FMM(kernel, precision="tf32x3", **opt)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for k in (1.0, -3.0):  # the second call on what the first one left
            wk = torch.zeros_like(w)
            wk += k * w
            got = plan.eval(src, wk, tgt)
            wk.zero_()
            d = (got - k * ref).norm()
            scale = (k * ref).norm()
            assert float(d) <= TOL * float(scale) + 1e-300
