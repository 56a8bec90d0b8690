"""A far pair of the FP64 high-order sum (zm_brdw.cu) is held to FP64 precision by itself, whatever the
near pairs contribute: where the strength is confined to a patch, every velocity away from it consists
of far pairs alone.

Reference: the sum in extended precision (numpy longdouble, more than 64 bits) over the same FP64 source
strengths.  Positions are multiples of 2^-36, mesh spacings powers of two and w2 = 0, so that the kernel's
strengths are reproduced here bit for bit: the stencil sums are exact, and one rounding each follows.

Errors are taken relative to sqrt(R_i^2 + |u_i|^2), R_i = sqrt(sum_j (K_ij |r_ij| |gamma'_j|)^2): the
size of the terms and that of their sum.
Tolerances, u = 2^-53: a pair of the plain form rounds its differences (u each), |r|^2 (3 u, 4.5 u in
K), K (1 u), the cross product (2 u) and the sum (1 u), below 10 u in all.  The far form has
t (1 u), q and K in fixed point (2 u), s x g (2 u), the three terms of M - t x G (4 u) and the sum
(1 u), 10 u as well: 16 u at the worst target leaves room for second-order terms, and independent
roundings give an rms below half of the sum of the bounds, 5 u.  (Pairs held to 2^-46 err by 100 u.)
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
DELTA = 2.0 ** -10


def interface(n1, n2, seed):
    """Positions, multiples of 2^-36, of a rough interface over the unit square."""
    rng = np.random.default_rng(seed)
    a, b = np.meshgrid(np.arange(n1) / n1, np.arange(n2) / n2, indexing="ij")

    def rough(amp):
        return np.rint(rng.uniform(-amp, amp, size=(n1, n2)) * 2.0 ** 36) * 2.0 ** -36

    smooth = np.rint(0.05 * np.cos(2 * np.pi * (a + 2 * b)) * 2.0 ** 36) * 2.0 ** -36
    return np.stack([a + rough(0.2 / n1), b + rough(0.2 / n2), smooth + rough(0.1 / n1)])


def strengths(z, w1):
    """pref (w1 D2 z), as the library forms it (w2 = 0), periodic."""
    n1, n2 = w1.shape
    dx1, dx2 = 1.0 / n1, 1.0 / n2
    pref = dx1 * dx2 / (4.0 * 3.14159265358979323846)
    g = []
    for c in range(3):
        f = z[c]

        def at(k):
            v = np.roll(f, -k, axis=1)
            if c == 1:  # the seam of z2
                v = v.copy()
                if k > 0:
                    v[:, n2 - k:] += 1.0
                else:
                    v[:, :-k] -= 1.0
            return v

        d = ((at(-2) - at(2)) + 8.0 * (at(1) - at(-1))) * (1.0 / (12.0 * dx2))
        g.append(pref * (w1 * d))
    return np.stack(g).reshape(3, -1)


def exact(z, g, targets):
    """u in extended precision at `targets` (flat indices), and the size errors are relative to."""
    L = np.longdouble
    zf, gf = z.reshape(3, -1).astype(L), g
    src = np.flatnonzero(np.any(gf != 0.0, axis=0))
    zs, gs = zf[:, src], gf[:, src].astype(L)
    gn = np.sqrt((gs * gs).sum(axis=0))
    u, size = np.empty((3, len(targets)), dtype=L), np.empty(len(targets))
    for k, i in enumerate(targets):
        r = zs - zf[:, [i]]
        q = (r * r).sum(axis=0) + L(DELTA) * L(DELTA)
        K = 1 / (q * np.sqrt(q))
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            u[c, k] = (K * (r[a] * gs[b] - r[b] * gs[a])).sum()
        size[k] = float(np.sqrt(((K * gn) ** 2 * (r * r).sum(axis=0)).sum() + (u[:, k] ** 2).sum()))
    return u, size


def velocity(z, w1, shift=0.0):
    from paper_2406_05490_gb300 import zm
    n1, n2 = w1.shape
    zz = z.reshape(3, -1).copy()
    zz[0] += shift
    w = np.stack([w1.ravel(), np.zeros(n1 * n2)])
    m = zm.ZModel(n1, n2, periodic=True, delta=DELTA)
    u = m.velocity(zz, w, want_wdot=False)
    m.close()
    return u


@pytest.mark.parametrize("n1,n2", [(64, 64), (128, 64)])
@pytest.mark.parametrize("kind", ["one node", "random patch", "alike patch"])
def test_strength_confined_to_a_patch(n1, n2, kind):
    z = interface(n1, n2, seed=n1 + n2)
    rng = np.random.default_rng(3)
    w1 = np.zeros((n1, n2))
    i0, j0 = 21, 37
    if kind == "one node":
        w1[i0, j0] = 0.7310585786300049
    else:
        p = rng.normal(size=(7, 6)) if kind == "random patch" else 1.0 + 0.1 * rng.uniform(size=(7, 6))
        w1[i0:i0 + 7, j0:j0 + 6] = p
    g = strengths(z, w1)
    centre = z[:, i0 + 3, j0 + 3]
    dist = np.sqrt(((z.reshape(3, -1) - centre[:, None]) ** 2).sum(axis=0))
    away = np.flatnonzero(dist > 0.4)
    targets = away[:: max(1, len(away) // 400)]
    u = velocity(z, w1)[:, targets]
    ref, size = exact(z, g, targets)
    err = np.sqrt((((u - ref).astype(np.float64)) ** 2).sum(axis=0)) / size
    rms, worst = float(np.sqrt(np.mean(err * err))), float(err.max())
    print(f"{n1}x{n2} {kind}: relative error rms {rms / U:.2f} u, worst {worst / U:.2f} u")
    assert rms <= 5 * U and worst <= 16 * U


def test_strength_everywhere():
    """Relative L2 error of u over sampled targets; 2^13 terms of like size whose near ones are sums of
    FP64 pairs: 2e-15, about three times the error of plain sums of this length."""
    n1, n2 = 128, 64
    z = interface(n1, n2, seed=1)
    a, b = np.meshgrid(np.arange(n1) / n1, np.arange(n2) / n2, indexing="ij")
    w1 = np.sin(2 * np.pi * (a + b)) + 0.3
    targets = np.random.default_rng(2).choice(n1 * n2, 64, replace=False)
    u = velocity(z, w1)[:, targets]
    ref, _ = exact(z, strengths(z, w1), targets)
    err = float(np.linalg.norm((u - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64)))
    print(f"128x64, strength everywhere: rel L2 u {err:.2e}")
    assert err <= 2e-15


def test_the_origin_of_the_coordinates_does_not_matter():
    """Shifting an interface by an amount that keeps its coordinates exact changes no bit of u: the far
    form serves it wherever it lies."""
    z = interface(64, 64, seed=4)
    w1 = np.random.default_rng(5).normal(size=(64, 64))
    u = velocity(z, w1)
    for shift in (8.0, 1024.0, -65536.0):
        assert np.array_equal((z[0] + shift) - shift, z[0])
        assert np.array_equal(velocity(z, w1, shift), u), shift
