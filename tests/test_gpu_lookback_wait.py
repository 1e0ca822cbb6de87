"""The look-back waits of the sort and of the tree build may run out: the result
must not change.

A waiter that gives up counts the tile it waited for itself.  With the limit at
one cycle nearly every wait that blocks ends that way; the evaluations must
give the bits they give with the default limit (same order of the points, same
boxes), and no status.  Sets of several tiles of 4,096 points, several tiles of 16
boxes a level, sources that are the targets and separate targets.
"""
import numpy as np
import pytest

from paper_2305_17867_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,levels,n,m", [
    (3, 5, 200003, 0),        # 49 tiles, two passes of 8 bits
    (3, 7, 8193, 30011),      # three passes, one tile more than a block's set
    (2, 8, 100000, 5),        # two passes, separate targets sorted by one block
    (-3, -9, 60000, 0), (-3, -10, 20011, 40009),  # adaptive (four passes)
])
def test_result_without_the_waits(d, levels, n, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300 import _lib
    from paper_2305_17867_gb300.fmm import FMM

    L = _lib.load()
    rng = np.random.Generator(np.random.PCG64(n + m))
    k = abs(d)
    pts = W.plummer_points(rng, n) if levels < 0 else rng.random((n, k))
    src = torch.tensor(pts, device="cuda")
    tgt = torch.tensor(rng.random((m, k)), device="cuda") if m else None
    w = torch.tensor(rng.normal(size=n), device="cuda")
    plan = FMM("laplace", d=k, p=2, levels=levels, precision="fp64", max_leaf=24)
    ref = plan.eval(src, w, tgt, check_status=True)
    tree = plan.last_tree()
    for limit in (1, 3000, 0):
        assert L.fmm_set_wait_limit(plan._h, limit) == 0
        for _ in range(3):
            assert torch.equal(plan.eval(src, w, tgt, check_status=True), ref)
            assert plan.last_tree() == tree
