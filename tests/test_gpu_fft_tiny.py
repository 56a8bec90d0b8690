"""The FP64 low-order velocity for vorticities near the lower end of FP64 (zm_fft.cu): block floating point
takes its unit from the largest value, down to the denormal numbers.

u is linear in w, so a power of two on w is one on u: exactly, as long as no bit of w or u falls below
2^-1074 (w consists of multiples of 2^-18, and u has 53 bits, the leading one above 2^-60).  Below that, u differs
from the scaled one by the roundings to multiples of 2^-1074 of s, of s N and of the scaled u, half a
unit each, and by the integers' own noise, less than another half: 2 units.
"""
import numpy as np
import pytest

from paper_2406_05490_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(64, 128), (24, 40), (8, 8)])
def test_tiny_vorticity(n1, n2):
    from paper_2406_05490_gb300 import zm
    a, b = inputs.mesh_coords(n1, n2)
    z = np.stack([a, b, 0 * a])
    w = np.rint(np.random.default_rng(n1).normal(size=(2, n1 * n2)) * 2.0 ** 18) * 2.0 ** -18
    m = zm.ZModel(n1, n2, order=zm.ZM_ORDER_LOW)
    u = m.velocity(z, w, want_wdot=False)
    for j in (-936, -944, -960):
        assert np.array_equal(m.velocity(z, np.ldexp(w, j), want_wdot=False), np.ldexp(u, j)), j
    for j in (-1005, -1050):  # the second: denormal numbers only
        d = m.velocity(z, np.ldexp(w, j), want_wdot=False) - np.ldexp(u, j)
        assert np.max(np.abs(d)) <= 2 * 2.0 ** -1074, j
    m.close()
