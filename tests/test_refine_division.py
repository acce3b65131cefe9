"""The refinement's quotients and reciprocals (FMA corrections of a guess) are the rounded ones of `/`, over the operands'
range: masses, mass ratios, phases to 1e9 rad and their derivatives, frequencies to the power of a third."""
import ctypes as C

import numpy as np

from paper_2110_13115_gb300 import _native as N


def _run(a, b):
    q, inv = np.empty_like(a), np.empty_like(a)
    p = [C.c_void_p(x.ctypes.data) for x in (a, b, q, inv)]
    N.load().rbx_refine_division(len(a), *p)
    return q, inv


def test_against_division():
    rng = np.random.default_rng(1)
    n = 1 << 20
    for lo, hi in ((-1, 1), (-12, 12), (-60, 60)):
        a, b = (np.exp2(rng.uniform(lo, hi, n)) * (1 + rng.random(n)) for _ in range(2))
        a = np.where(rng.random(n) < 0.5, -a, a)
        q, inv = _run(a, b)
        assert np.array_equal(q, a / b) and np.array_equal(inv, 1.0 / (a * b))
    # mantissas at their ends, among them the divisors just below a power of two
    ends = np.array([1.0, np.nextafter(1, 2), np.nextafter(2, 1), 2 - 2.0 ** -51, 1.5, 1 + 2.0 ** -26, 4 / 3, 5 / 3])
    ends = (ends[:, None] * np.exp2(np.arange(-40.0, 41.0))).ravel()
    a, b = (x.ravel().copy() for x in np.meshgrid(ends, ends))
    q, inv = _run(a, b)
    assert np.array_equal(q, a / b)
    assert (inv != 1.0 / (a * b)).sum() == 0
    z = np.zeros(4)
    q, _ = _run(z, np.array([0.1, 3.0, 1e-9, 1e9]))
    assert np.array_equal(q, z)
