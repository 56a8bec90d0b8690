"""The FP64 high-order sum on meshes of 56^2 nodes and more (zm_brdw.cu): far tile pairs in FP32
pairs and integers, near ones in FP64.

The same state with every length times 2^-130 lies outside the range of the far form, so that all
pairs take the plain FP64 form, and u is unchanged by such a scaling: the two calls differ by the
far form alone.  Tolerance on their difference: the plain sums have at most 2^14 terms, whose random
walk of FP64 roundings is below 2^-53 2^7 = 1.4e-14, and a far pair's independent error of about
2^-46 is below that after the sum; 2e-14.  Against the oracle the repository's FP64 bound, 1e-12.
"""
import numpy as np
import pytest

import oracle
from paper_2406_05490_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL64 = 1e-12
TOL_PLAIN = 2e-14


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def velocity(n1, n2, z, w, periodic=True, delta=None, k=0, j=0):
    """u for lengths times 2^k and strengths times 2^j."""
    from paper_2406_05490_gb300 import zm
    L = 2.0 ** k
    m = zm.ZModel(n1, n2, L1=L, L2=L, periodic=periodic, delta=np.ldexp(delta, k))
    u = m.velocity(np.ldexp(z, k), np.ldexp(w, j), want_wdot=False)
    m.close()
    return u


@pytest.mark.parametrize("n1,n2,periodic", [(56, 56, True), (57, 65, False), (63, 121, True), (640, 5, False),
                                            (5, 641, False), (9, 400, True), (96, 97, True), (128, 128, True)])
def test_far_form_against_the_plain_form_and_the_oracle(n1, n2, periodic):
    """The smallest mesh of the range, edge tiles one node wide, meshes narrower than a tile, both
    boundary rules, both classification factors."""
    z, w = inputs.random_state(n1, n2, seed=n1 + 3 * n2)
    delta = 0.1 / max(n1, n2)
    u = velocity(n1, n2, z, w, periodic, delta)
    plain = velocity(n1, n2, z, w, periodic, delta, k=-130)
    u_ref, _ = oracle.derivative(oracle.Mesh(n1, n2, periodic=periodic), z, w, 0.5, 1.0, 0.0, delta)
    print(f"{n1}x{n2} periodic={periodic}: rel L2 u plain {rel(u, plain):.2e} oracle {rel(u, u_ref):.2e}")
    assert not np.array_equal(u, plain)  # the far form ran
    assert rel(u, plain) <= TOL_PLAIN and rel(u, u_ref) <= TOL64


@pytest.mark.parametrize("delta", [0.5, 40.0])
def test_core_size_beyond_the_tiles(delta):
    """A core larger than the tiles (far pairs with delta^2 in front), and one beyond the range of the
    far form (every pair near)."""
    n = 64
    z, w = inputs.random_state(n, seed=5)
    u_ref, _ = oracle.derivative(oracle.Mesh(n, periodic=True), z, w, 0.5, 1.0, 0.0, delta)
    assert rel(velocity(n, n, z, w, delta=delta), u_ref) <= TOL64


def test_scaling_by_powers_of_two_is_exact_in_range():
    """u scales exactly while lengths and strengths fit the far form, and agrees beyond it."""
    n = 64
    z, w = inputs.random_state(n, seed=9)
    d = 0.1 / n
    u = velocity(n, n, z, w, delta=d)
    for k, j in ((-40, 0), (60, 0), (0, 250), (-30, -300)):
        assert np.array_equal(velocity(n, n, z, w, delta=d, k=k, j=j), np.ldexp(u, j)), (k, j)
    for k, j in ((120, 0), (0, 500), (0, -600)):
        assert rel(np.ldexp(velocity(n, n, z, w, delta=d, k=k, j=j), -j), u) <= TOL_PLAIN, (k, j)


def test_points_far_from_the_mesh_and_not_finite():
    """One node far outside the coordinate range makes its tiles near to all; a NaN or an infinite
    strength reaches every velocity, as in a plain sum."""
    n = 64
    z, w = inputs.random_state(n, seed=11)
    z[0, 100] = 1e6
    u_ref, _ = oracle.derivative(oracle.Mesh(n, periodic=True), z, w, 0.5, 1.0, 0.0, 0.1 / n)
    assert rel(velocity(n, n, z, w, delta=0.1 / n), u_ref) <= TOL64
    z, w = inputs.random_state(n, seed=11)
    for field, value in ((z, np.nan), (w, np.inf)):
        keep = field[0, 1000]
        field[0, 1000] = value
        assert not np.any(np.isfinite(velocity(n, n, z, w, delta=0.1 / n)))
        field[0, 1000] = keep
