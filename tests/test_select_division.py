"""The selection's division by a range (two norms share it, so the kernel keeps
a correctly rounded reciprocal and corrects n inv twice by its residual) gives
the correctly rounded quotient for every n that the rule lets through: fp32
steps restated with the C library's fmaf, against IEEE division."""
import ctypes

import numpy as np

_m = ctypes.CDLL("libm.so.6")
_m.fmaf.argtypes = [ctypes.c_float] * 3
_m.fmaf.restype = ctypes.c_float


def _quotient(n, d):
    n, d = np.float32(n), np.float32(d)
    inv = np.float32(1.0) / d
    q = np.float32(n * inv)
    for _ in range(2):
        q = np.float32(_m.fmaf(_m.fmaf(float(q), float(-d), float(n)), float(inv), float(q)))
    return q


def test_quotient_is_correctly_rounded():
    g = np.random.default_rng(0)
    cases = []
    # ranges over the whole admitted interval, quotients over (0, 1]
    d = np.exp2(g.uniform(-98, 20, 20000)).astype(np.float32)
    cases.append((np.maximum(d * g.random(20000), 2.0 ** -98).astype(np.float32), d))
    # mantissas next to a power of two and all ones, where one correction is not enough
    for m in (1, 2, 3, 2 ** 23 - 1, 2 ** 23 - 2, 2 ** 23 - 3, 2 ** 22, 2 ** 22 - 1):
        d = np.uint32((127 << 23) | m).view(np.float32)
        n = ((127 << 23) | g.integers(0, 2 ** 23, 1500)).astype(np.uint32).view(np.float32)
        cases.append((n, np.full(1500, d)))
        cases.append((np.full(1500, d), n))
    # the ends: the smallest norm's difference over the largest range, n = d, n = 0
    cases.append((np.float32([2.0 ** -98, 2.0 ** -98, 2.0 ** 20, 0.0]), np.float32([2.0 ** 20, 2.0 ** -98, 2.0 ** 20, 3.0])))
    for n, d in cases:
        want = n / d
        got = np.array([_quotient(a, b) for a, b in zip(n, d)], np.float32)
        bad = np.flatnonzero(got.view(np.uint32) != want.view(np.uint32))
        assert bad.size == 0, (n[bad[:3]], d[bad[:3]], got[bad[:3]], want[bad[:3]])
    # +0 stays +0 (the ordered key takes the bits as they are)
    assert _quotient(0.0, 3.0).view(np.uint32) == 0
