"""How close the FP64 low-order velocity (integer FFT, zm_fft.cu) is to the exact Riesz transform of a
field of 16 modes, on a flat interface.

Reference: R_l cos(theta) = (k_l / |k|) sin(theta), summed over the modes in extended precision (numpy
longdouble).  Tolerance, relative L2: a value in a row is held to about one unit after each of at most ten
chunks of stages, a row's largest value is 2^55 units or more, and a sum of 16 modes with its spectra has
rms values within 2^3 of its largest ones: 2^-52 sqrt(10) = 7.0e-16; the rounding of w to FP64 and of u adds
2^-53 each (1.6e-16 together): 7.2e-16 in all, 1e-15.
"""
import numpy as np
import pytest

from paper_2406_05490_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-15


@pytest.mark.parametrize("n1,n2", [(128, 128), (256, 256), (152, 304), (608, 152), (320, 192)])
def test_modes(n1, n2):
    from paper_2406_05490_gb300 import zm
    L = np.longdouble
    rng = np.random.default_rng(n1 + n2)
    i, j = np.meshgrid(np.arange(n1), np.arange(n2), indexing="ij")
    pi2 = L("6.28318530717958647692528676655900576839433879875")
    w, s = np.zeros((2, n1, n2), dtype=L), np.zeros((n1, n2), dtype=L)
    for _ in range(16):
        m = rng.integers(2, 9, size=2)
        # the phase in turns, reduced exactly before the multiplication by 2 pi
        turns = ((m[0] * i * n2 + m[1] * j * n1) % (n1 * n2)).astype(L) / L(n1 * n2)
        theta = pi2 * turns + L(rng.uniform(0, 6.25))
        for c in range(2):
            a = L(rng.normal())
            w[c] += a * np.cos(theta)
            s += a * (L(m[c]) / np.sqrt(L(m[0] * m[0] + m[1] * m[1]))) * np.sin(theta)
    x, y = inputs.mesh_coords(n1, n2)
    model = zm.ZModel(n1, n2, order=zm.ZM_ORDER_LOW)
    u = model.velocity(np.stack([x, y, 0 * x]), w.astype(np.float64).reshape(2, -1), want_wdot=False)
    model.close()
    ref = -s.reshape(-1) / 2
    e = float(np.sqrt(((u[2] - ref) ** 2).sum() / (ref * ref).sum()))
    print(f"{n1}x{n2}: rel L2 u {e:.2e}")
    assert e <= TOL
