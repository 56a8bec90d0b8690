"""The FP64 low-order velocity's integer FFT (zm_fft.cu, zm_fix.cuh) where its plan and its block
floating point can go wrong: the shortest and the longest rows, one to four chunks per row, every kind of
side in either direction, fields of one value, of noise and of one mode, exponents from one end of FP64
to the other, values that are not finite.

Tolerance on u against numpy's FP64 transform: block floating point rounds by a few units per chunk and
pass (at most 10 chunks), relative to a row's largest value and at least 54 bits below it; over four
transforms and a crest factor of up to 2^5 that is below 2^-54 2^5 10 = 1.8e-14; numpy's own transform
and the normal (FP64 stencils) are below 1e-15: 2e-14.
"""
import numpy as np
import pytest

from paper_2406_05490_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 2e-14


def velocity(n1, n2, z, w, L1=1.0, L2=1.0):
    from paper_2406_05490_gb300 import zm
    m = zm.ZModel(n1, n2, L1=L1, L2=L2, order=zm.ZM_ORDER_LOW)
    u = m.velocity(z, w, want_wdot=False)
    m.close()
    return u


def flat(n1, n2, L1=1.0, L2=1.0):
    a, b = inputs.mesh_coords(n1, n2, L1, L2)
    return np.stack([a, b, 0 * a])


def reference(n1, n2, w, L1=1.0, L2=1.0):
    """u3 = -s/2 on a flat interface (N = (0, 0, 1))."""
    t1 = (np.fft.fftfreq(n1) * n1 / L1)[:, None]
    t2 = (np.fft.fftfreq(n2) * n2 / L2)[None, :]
    k = np.sqrt(t1 * t1 + t2 * t2)
    k[0, 0] = 1.0
    s = np.fft.fft2(w[0].reshape(n1, n2)) * (-1j * t1 / k) + np.fft.fft2(w[1].reshape(n1, n2)) * (-1j * t2 / k)
    s[0, 0] = 0
    s[n1 // 2, :] = 0
    s[:, n2 // 2] = 0
    return -0.5 * np.fft.ifft2(s).real.reshape(-1)


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


SIDES = [(8, 8), (8, 16), (32, 64), (512, 8), (8, 8192), (8192, 8), (24, 40), (3 << 6, 5 << 5), (7 << 4, 9 << 3),
         (11 << 3, 13 << 4), (15 << 5, 17 << 3), (19 << 3, 19 << 4), (8, 15 << 9), (17 << 8, 8), (256, 19 << 5)]


@pytest.mark.parametrize("n1,n2", SIDES)
@pytest.mark.parametrize("kind", ["noise", "mode"])
def test_against_numpy(n1, n2, kind):
    if kind == "noise":
        w = np.random.default_rng(n1 + n2).normal(size=(2, n1 * n2))
    else:
        a, b = inputs.mesh_coords(n1, n2)
        w = np.stack([np.sin(2 * np.pi * (a + b)), 1e-6 * np.cos(2 * np.pi * (2 * a - b) + 0.3)])
    u = velocity(n1, n2, flat(n1, n2), w)
    e = rel(u[2], reference(n1, n2, w))
    print(f"{n1}x{n2} {kind}: {e:.2e}")
    assert e <= TOL
    assert np.all(u[:2] == 0.0)


def test_lengths_differ():
    n1, n2, L1, L2 = 48, 128, 0.7, 3.0
    w = np.random.default_rng(2).normal(size=(2, n1 * n2))
    z = flat(n1, n2, L1, L2)
    z[0] += 0.0
    assert rel(velocity(n1, n2, z, w, L1, L2)[2], reference(n1, n2, w, L1, L2)) <= TOL


@pytest.mark.parametrize("n1,n2", [(64, 128), (24, 40)])
def test_exponents(n1, n2):
    """Powers of two scale u exactly; a constant field and a zero field give zero; one value far above
    all others keeps its own velocity."""
    w = np.random.default_rng(3).normal(size=(2, n1 * n2))
    z = flat(n1, n2)
    u = velocity(n1, n2, z, w)
    for j in (1, -7, 400, -400, 900, -800):
        assert np.array_equal(velocity(n1, n2, z, np.ldexp(w, j)), np.ldexp(u, j)), j
    assert np.all(velocity(n1, n2, z, np.zeros_like(w)) == 0.0)
    c = velocity(n1, n2, z, np.full_like(w, 0.7))
    assert np.max(np.abs(c)) <= 0.7 * TOL
    w[0, 77] = 1e30
    assert rel(velocity(n1, n2, z, w)[2], reference(n1, n2, w)) <= TOL


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_not_finite(value):
    """One value that is not finite makes all of u NaN or infinite, and the next call is clean."""
    from paper_2406_05490_gb300 import zm
    n1, n2 = 40, 64
    z, w = inputs.random_state(n1, n2, seed=4)
    m = zm.ZModel(n1, n2, order=zm.ZM_ORDER_LOW)
    u = m.velocity(z, w, want_wdot=False)
    bad = w.copy()
    bad[1, 1234] = value
    assert not np.any(np.isfinite(m.velocity(z, bad, want_wdot=False)))
    assert np.array_equal(m.velocity(z, w, want_wdot=False), u)
    m.close()
