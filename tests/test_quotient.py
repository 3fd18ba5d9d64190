"""Error bound of the quotients that the FP32 path's output rows are formed with: q = n (1 / d), corrected once by its remainder,
q + (n - q d) (1 / d), each step rounded to fp32 and the two in the correction fused (Markstein 1990)."""
import numpy as np


def _fma(a, b, c):
    return (a.astype(np.longdouble) * b.astype(np.longdouble) + c.astype(np.longdouble)).astype(np.float32)


def test_the_corrected_quotient_is_within_an_ulp():
    rng = np.random.default_rng(7)
    n = (rng.standard_normal(400000) * 10.0 ** rng.uniform(-12, 12, 400000)).astype(np.float32)
    d = (10.0 ** rng.uniform(-12, 12, 400000)).astype(np.float32)
    inv = (np.float32(1) / d).astype(np.float32)
    q = n * inv
    q = _fma(_fma(-q, d, n), inv, q)
    exact = n.astype(np.longdouble) / d.astype(np.longdouble)
    ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(np.longdouble)
    assert (np.abs(q.astype(np.longdouble) - exact) <= ulp).all()
    assert (q == exact.astype(np.float32)).mean() > 0.999
