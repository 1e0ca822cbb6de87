"""Adaptive trees of very few boxes at every depth limit: the build's scratch is sized
by the depth there, not by the boxes (the launches compare what they use with
what the workspace holds and refuse it otherwise).

Against the direct sum: all pairs are near-field pairs (1e-12 in FP64, 2e-5 in
float); a workspace of exactly the size that fmm_workspace_size states.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("bf16x3", 2e-5)])
@pytest.mark.parametrize("depth", [1, 2, 7, 10])
@pytest.mark.parametrize("n,m", [(1, 1), (2, 0), (0, 3), (9, 40)])
def test_few_boxes(oracle, precision, tol, depth, n, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300 import _lib
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(50 + n)
    src, w, tgt = rng.random((n, 3)), rng.uniform(0.5, 1.0, n), rng.random((m, 3))
    plan = FMM("laplace", d=3, p=4, levels=-depth, max_leaf=64, precision=precision)
    s, wd = torch.tensor(src, device="cuda"), torch.tensor(w, device="cuda")
    t = torch.tensor(tgt, device="cuda") if m else s
    nt = t.shape[0]
    need = plan.workspace_bytes(n, nt)
    ws = torch.full((need + 512,), 0x5A, dtype=torch.uint8, device="cuda")
    at = (ws.data_ptr() + 255) // 256 * 256
    phi = torch.empty(nt, device="cuda", dtype=torch.float64)
    p = lambda x: ctypes.c_void_p(x.data_ptr() if x.numel() else 0)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    L = _lib.load()
    assert L.fmm_eval(plan._h, n, p(s), p(wd), nt, p(t), p(phi), None, ctypes.c_void_p(at), need,
                      stream) == 0
    assert plan.last_status() == 0 and plan.last_tree() == (1, 0)
    got = phi.cpu().numpy()
    assert bool((ws[at - ws.data_ptr() + need:] == 0x5A).all())  # nothing past the end
    if n == 0:
        assert np.all(got == 0.0)
    else:
        ref = oracle.direct("laplace", 3, src, w, tgt if m else src)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
