"""An evaluation that ends with an error has its streams joined to the caller's.

The mixed-precision 3D plans work on two streams of their own.  When a launch is
refused after the near field has been started there, the call returns
FMM_ERR_CUDA, and what runs must still be ordered before the caller's next
work: a copy of the output made once the caller's stream is idle has to be
final.  The refused launch is a kernel whose shared memory exceeds the chip's:
a PDE of order p + 1 keeps every coefficient, and at these orders the FFT
table's (uniform) and the M2P's (adaptive) blocks no longer fit; the runtime
returns an error and nothing of that kernel runs.
"""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,p,levels", [("laplace", 16, 3), ("yukawa", 18, -4)])
def test_failed_call_is_joined(kernel, p, levels):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300 import _lib
    from paper_2305_17867_gb300.fmm import FMM

    L = _lib.load()
    n = 400000
    gen = torch.Generator(device="cuda").manual_seed(5)
    src = torch.rand(n, 3, generator=gen, device="cuda", dtype=torch.float64)
    w = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    plan = FMM(kernel, d=3, p=p, levels=levels, max_leaf=2000, precision="fp32", m2l="auto",
               lam=1.0 if kernel == "yukawa" else 0.0, pde=([[0, 0, p + 1]], [1.0]),
               root_lo=[0.0] * 3, root_size=1.0)
    assert plan.nj == plan.nfull
    ws, wb = plan._workspace(n, n)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(2):
        phi = torch.full((n,), -7.0, device="cuda", dtype=torch.float64)
        torch.cuda.synchronize()
        rc = L.fmm_eval(plan._h, n, ptr(src), ptr(w), n, ptr(src), ptr(phi), None, ws, wb,
                        ctypes.c_void_p(stream.cuda_stream))
        stream.synchronize()
        with torch.cuda.stream(other):
            seen = phi.clone()
        other.synchronize()
        torch.cuda.synchronize()
        assert rc == -3  # FMM_ERR_CUDA
        assert bool((phi != -7.0).all())  # the near field had been started
        assert torch.equal(seen, phi)
