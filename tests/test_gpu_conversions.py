"""Conversions of expansion coefficients between FP64 and the float and double-word
float arithmetic of the mixed-precision modes: the bits the FP64 conversions
give, h = fl(x) and l = fl(x - h).
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def unary():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300 import _lib

    L = _lib.load()

    def run(op, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        out = np.empty_like(x)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert L.fmm_selftest_unary(op, x.size, p(x), p(out)) == 0
        return out

    return run


def values(lo, hi, seed):
    """Magnitudes 2^lo .. 2^hi of both signs: random significands, and the ones at which
    rounding to 24 and 48 bits goes either way (ties, carries into the exponent)."""
    rng = np.random.default_rng(seed)
    n = 20000
    x = rng.choice([-1.0, 1.0], n) * np.exp2(rng.uniform(lo, hi, n))
    bits = x.view(np.uint64) >> np.uint64(29) << np.uint64(29)  # 24-bit significands ...
    low = rng.choice([0, 1, 1 << 28, (1 << 28) - 1, (1 << 28) + 1, (1 << 29) - 1, 1 << 4, 3 << 3],
                     n).astype(np.uint64)
    edge = (bits | low).view(np.float64)  # ... and the rest at the edges
    edge[: n // 4] = (bits[: n // 4] | np.uint64(0xFFFFFE0000000) | low[: n // 4]).view(np.float64)
    return np.concatenate([x, edge, [0.0, 1.0, -1.0]])


@pytest.mark.parametrize("lo,hi", [(-60, 115), (-3, 3), (-63.5, -62.5), (116, 118.5),
                                   (-128, -80), (-151, -124)])  # subnormal low and high parts
def test_as_the_fp64_conversions(unary, lo, hi):
    x = values(lo, hi, abs(int(hi * 10)))
    h = x.astype(np.float32)
    with np.errstate(over="ignore", invalid="ignore"):
        low = (x - h.astype(np.float64)).astype(np.float32)
        want = h.astype(np.float64) + low.astype(np.float64)
    assert np.array_equal(unary(0, x), want)
    assert np.array_equal(unary(1, x), h.astype(np.float64))
