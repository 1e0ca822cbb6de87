"""A launch the runtime refuses is an error of the call, wherever in a stage it stands.

A PDE of order p + 1 keeps every coefficient; at these orders one kernel's block
needs more shared memory than the chip has (the FFT table's, the adaptive
P2L's) while the kernels launched after it fit.  The call has to say so
(FMM_ERR_CUDA) instead of returning potentials without that kernel's part, and
the plan's next, smaller sibling has to work.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,p,levels,fits", [
    ("fp32", 16, 3, 10), ("fp64", 12, 3, 8), ("fp32", 17, -5, 10),
])
def test_refused_launch_is_reported(precision, p, levels, fits):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300._lib import FMMError
    from paper_2305_17867_gb300.fmm import FMM

    gen = torch.Generator(device="cuda").manual_seed(9)
    n = 20000
    src = torch.rand(n, 3, generator=gen, device="cuda", dtype=torch.float64)
    w = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)

    def run(order):
        plan = FMM("laplace", d=3, p=order, levels=levels, max_leaf=100, precision=precision,
                   m2l="auto", pde=([[0, 0, order + 1]], [1.0]))
        assert plan.nj == plan.nfull
        return plan.eval(src, w, check_status=True)

    with pytest.raises(FMMError) as e:
        run(p)
    assert e.value.code == -3  # FMM_ERR_CUDA
    ref = FMM("laplace", d=3, p=fits, levels=levels, max_leaf=100, precision="fp64").eval(src, w)
    assert float((run(fits) - ref).norm() / ref.norm()) < 1e-5
