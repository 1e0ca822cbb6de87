"""The deepest uniform tree of the plane (L = 8): its level offsets end at
index L + 1 = 9, one past what the workspace record held, so every such call
read a pointer as a size.  FP64 against the CPU oracle on the same tree."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m2l", ["dense", "auto"])
def test_level_8_matches_oracle(oracle, m2l):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(28)
    src, w, tgt = rng.random((6000, 2)), rng.uniform(-1.0, 1.0, 6000), rng.random((40, 2))
    ref = oracle.fmm_uniform("laplace", 2, 3, 8, src, w, tgt)
    plan = FMM("laplace", d=2, p=3, levels=8, precision="fp64", m2l=m2l)
    got = plan.eval(torch.tensor(src, device="cuda"), torch.tensor(w, device="cuda"),
                    torch.tensor(tgt, device="cuda"), check_status=True).cpu().numpy()
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-12
