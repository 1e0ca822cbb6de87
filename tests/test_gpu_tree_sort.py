"""The device sort under the trees: one-block sets, sets of several look-back
tiles, their edges, odd distributions, and float32 against float64 points.

FP64 evaluations against the CPU oracle's same-tree FMM (1e-12, the FP64
parity bound): a point sorted into a wrong leaf, a lost or doubled point or a
leaf range off by one changes a potential by far more.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def points(kind, n, d, rng):
    if kind == "uniform":
        return rng.random((n, d))
    if kind == "faces":  # many points exactly on leaf faces and the root's corner
        return rng.integers(0, 16, (n, d)) / 16.0 + rng.integers(0, 2, (n, d)) * 1e-9
    x = rng.random((n, d))  # most of the points in one leaf
    x[: (4 * n) // 5] = 0.3 + 1e-3 * x[: (4 * n) // 5]
    return x


@pytest.mark.parametrize("d,levels,n,kind", [
    (3, 2, 1, "uniform"), (3, 3, 33, "uniform"), (3, 3, 1024, "faces"), (3, 4, 1025, "uniform"),
    (3, 3, 8192, "uniform"), (3, 3, 8193, "uniform"), (3, 5, 12289, "clump"),
    (3, 6, 20000, "uniform"), (2, 4, 8191, "faces"), (2, 4, 9000, "uniform"),
    (2, 8, 50000, "uniform"), (3, 4, 40961, "faces"),
])
def test_uniform_sorts(torch_cuda, oracle, d, levels, n, kind):
    torch = torch_cuda
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(7000 + n + d)
    src, w = points(kind, n, d, rng), rng.uniform(-1.0, 1.0, n)
    tgt = rng.random((60, d))
    ref = oracle.fmm_uniform("laplace", d, 3, levels, src, w, tgt)
    plan = FMM("laplace", d=d, p=3, levels=levels, precision="fp64")
    got = plan.eval(torch.tensor(src, device="cuda"), torch.tensor(w, device="cuda"),
                    torch.tensor(tgt, device="cuda"), check_status=True)
    assert rel_l2(got.cpu().numpy(), ref) < TOL


@pytest.mark.parametrize("n,kind", [(1, "uniform"), (500, "faces"), (8192, "clump"),
                                    (8193, "uniform"), (30000, "clump")])
def test_adaptive_sorts(torch_cuda, oracle, n, kind):
    torch = torch_cuda
    from paper_2305_17867_gb300.fmm import FMM

    rng = np.random.default_rng(8000 + n)
    src, w, tgt = points(kind, n, 3, rng), rng.uniform(-1.0, 1.0, n), rng.random((70, 3))
    ref, st, _ = oracle.fmm_adaptive("laplace", 3, 3, src, w, tgt, max_leaf=20, max_depth=8,
                                     want_stats=True)
    plan = FMM("laplace", d=3, p=3, levels=-8, precision="fp64", max_leaf=20)
    got = plan.eval(torch.tensor(src, device="cuda"), torch.tensor(w, device="cuda"),
                    torch.tensor(tgt, device="cuda"), check_status=True)
    assert plan.last_tree() == (st["boxes"], st["depth"])
    assert rel_l2(got.cpu().numpy(), ref) < TOL


@pytest.mark.parametrize("levels,n,lo,size", [(3, 5000, 0.0, 1.0), (4, 20000, -0.7, 2.9),
                                              (4, 20000, 900.0, 3.0), (-6, 9000, -0.7, 2.9),
                                              (3, 5000, 0.0, -1.0)])
def test_float_points(torch_cuda, levels, n, lo, size):
    # float32 points give the FP64 evaluation of their widened values, rounded
    # once; the float path's box-relative coordinates keep a root far from the
    # origin and a side that is no power of two accurate (the mixed evaluation
    # against FP64: the FP32 bound 2e-6, times the coordinates' own rounding
    # when the root lies far away)
    torch = torch_cuda
    from paper_2305_17867_gb300.fmm import FMM

    gen = torch.Generator(device="cuda").manual_seed(90 + n)
    side = abs(size)
    x = (lo + side * torch.rand(n, 3, generator=gen, device="cuda", dtype=torch.float32)
         .clamp(1e-4, 1 - 1e-4)).float()
    w = torch.rand(n, generator=gen, device="cuda", dtype=torch.float32) - 0.5
    kw = dict(d=3, p=6, levels=levels, root_lo=[lo] * 3, root_size=size, max_leaf=40)
    exact = FMM("laplace", precision="fp64", **kw)
    a = exact.eval_f32(x, w, check_status=True)
    b = exact.eval(x.double(), w.double(), check_status=True)
    assert torch.equal(a, b.float())
    mixed = FMM("laplace", precision="fp32", **kw)
    c = mixed.eval(x.double(), w.double(), check_status=True)
    e = mixed.eval_f32(x, w, check_status=True)
    assert torch.equal(e, c.float())
    assert float((c - b).norm() / b.norm()) < 2e-6
