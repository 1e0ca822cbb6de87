"""The table-driven FP64 logarithm of the planar near field, held to the accuracy of
the CUDA math library's log, which it stands in for: at most 1 ulp (the bound
CUDA documents) and an rms error no more than 1% larger, against 80 bits or more.

Ranges: around 1, the reduced interval with its seams at 3/4 and 3/2 and at
the table's midpoints, the squared distances a near field meets, and the whole
exponent range with powers of two and subnormals.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble


def reference(x):
    """log(x) in long double; on machines where that is double, a two-term correction."""
    if np.finfo(LD).nmant > 60:
        return np.log(x.astype(LD))
    import mpmath

    mpmath.mp.prec = 120
    return np.array([mpmath.log(float(v)) for v in x])


def sets(rng):
    n = 200000
    k = np.arange(96, 193) / 128.0
    mid = (k[:-1] + k[1:]) / 2
    seams = np.concatenate([k, mid, [0.75, 1.5, 1.0]])
    near = np.concatenate([np.nextafter(seams, 0), seams, np.nextafter(seams, 4)])
    near = near[near != 1.0]
    yield "near 1", 1.0 + rng.uniform(-1, 1, n) / 256
    yield "reduced", np.concatenate([rng.uniform(0.75, 1.5, n), near])
    yield "distances", np.exp(rng.uniform(np.log(1e-9), np.log(8.0), n))
    yield "all", np.concatenate([np.exp2(rng.uniform(-1022, 1023.9, n)),
                                 np.exp2(np.arange(-1074.0, 1024.0))])


def test_within_cudas_bound():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_17867_gb300 import _lib

    L = _lib.load()

    def run(op, x):
        out = np.empty_like(x)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert L.fmm_selftest_unary(op, x.size, p(x), p(out)) == 0
        return out

    for name, x in sets(np.random.default_rng(17)):
        x = np.ascontiguousarray(x[x > 0])
        x = x[x != 1.0]
        exact = reference(x)
        ulp = np.spacing(np.abs(exact.astype(np.float64)))
        ours = np.abs(((run(2, x) - exact) / ulp).astype(np.float64))
        cuda = np.abs(((run(3, x) - exact) / ulp).astype(np.float64))
        rms = lambda e: float(np.sqrt(np.mean(e * e)))
        print(f"{name}: max {ours.max():.4f} rms {rms(ours):.4f}; "
              f"CUDA max {cuda.max():.4f} rms {rms(cuda):.4f}")
        assert ours.max() <= 1.0
        assert rms(ours) <= 1.01 * rms(cuda)
    assert run(2, np.array([1.0]))[0] == 0.0
