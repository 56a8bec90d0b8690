"""The FP64 high-order sum with far pairs in integers (zm_brdw.cu, meshes of 56^2 nodes and more) where
single evaluations on plain interfaces do not go: medium order, whose evaluation builds the low-order
geometry first and this sum's records after it; several steps; an interface folded over itself, where
tiles far apart on the mesh meet in space; and the index-checked build on ragged tiles.

Against the oracle the repository's FP64 bound, 1e-12 relative L2.  The checked build counts no index
violation and gives the default build's bits.  Run as a program with a file name, this file writes the
outputs of the checked cases there.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2406_05490_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

TOL64 = 1e-12


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("order,n1,n2,periodic", [("medium", 80, 56, True), ("medium", 64, 72, True),
                                                  ("high", 57, 65, False), ("high", 90, 61, True)])
def test_evaluation_and_steps(order, n1, n2, periodic):
    import oracle
    from paper_2406_05490_gb300 import zm
    z, w = inputs.random_state(n1, n2, seed=n1 * 3 + n2, periodic=periodic)
    delta = 0.1 / max(n1, n2)
    m = oracle.Mesh(n1, n2, periodic=periodic)
    od = {"medium": oracle.ORDER_MEDIUM, "high": oracle.ORDER_HIGH}[order]
    u_ref, wd_ref = oracle.derivative(m, z, w, 0.6, 1.2, 0.01, delta, order=od)
    zr, wr = oracle.run(m, z, w, 0.6, 1.2, 0.01, delta, 2e-3, 3, order=od)
    model = zm.ZModel(n1, n2, periodic=periodic, atwood=0.6, g=1.2, mu=0.01, delta=delta,
                      order={"medium": zm.ZM_ORDER_MEDIUM, "high": zm.ZM_ORDER_HIGH}[order])
    u, wd = model.velocity(z, w)
    model.set_state(z, w)
    model.step(2e-3, 3)
    z1, w1 = model.get_state()
    model.close()
    e = [rel(u, u_ref), rel(wd, wd_ref), rel(z1, zr), rel(w1, wr)]
    print(f"{order} {n1}x{n2}: rel L2 u {e[0]:.2e} wdot {e[1]:.2e}, 3 steps z {e[2]:.2e} w {e[3]:.2e}")
    assert max(e) <= TOL64


def test_folded_interface():
    """z1 = a + 0.25 sin 2 pi a overhangs: nodes 20 and more mesh points apart come within 2 dx."""
    import oracle
    from paper_2406_05490_gb300 import zm
    n = 128
    a, b = inputs.mesh_coords(n)
    z = np.stack([a + 0.25 * np.sin(2 * np.pi * a), b + 0.05 * np.sin(2 * np.pi * a),
                  0.03 * np.sin(2 * np.pi * a) + 0.02 * np.cos(2 * np.pi * b)])
    _, w = inputs.random_state(n, seed=17)
    u_ref, wd_ref = oracle.derivative(oracle.Mesh(n, periodic=True), z, w, 0.5, 1.0, 0.0, 0.1 / n)
    model = zm.ZModel(n, periodic=True, atwood=0.5, g=1.0, delta=0.1 / n)
    u, wd = model.velocity(z, w)
    model.close()
    print(f"folded 128^2: rel L2 u {rel(u, u_ref):.2e} wdot {rel(wd, wd_ref):.2e}")
    assert rel(u, u_ref) <= TOL64 and rel(wd, wd_ref) <= TOL64


def checked_cases(path):
    from paper_2406_05490_gb300 import zm
    zm.load()
    zm.zm_bounds_status(clear=True)
    res = {}
    for name, n1, n2, periodic in (("high", 57, 65, False), ("high", 9, 400, True), ("high", 5, 641, False),
                                   ("high", 640, 5, False), ("high", 200, 90, True), ("medium", 80, 56, True)):
        z, w = inputs.random_state(n1, n2, seed=n1 + 7 * n2, periodic=periodic)
        m = zm.ZModel(n1, n2, periodic=periodic, atwood=0.6, g=1.2, mu=0.01, delta=0.1 / max(n1, n2),
                      order={"medium": zm.ZM_ORDER_MEDIUM, "high": zm.ZM_ORDER_HIGH}[name])
        u, wd = m.velocity(z, w)
        m.set_state(z, w)
        m.step(1e-3, 1)
        zs, ws = m.get_state()
        m.close()
        for k, v in (("u", u), ("wd", wd), ("z", zs), ("w", ws)):
            res[f"{name}{n1}x{n2}{k}"] = v
    hits, first, line = zm.zm_bounds_status(clear=True)
    res["build"] = np.array([int(zm.zm_checked_build()), hits, first, line], dtype=np.int64)
    np.savez(path, **res)


def test_checked_build(tmp_path):
    out = {}
    for variant in ("default", "checked"):
        env = dict(os.environ)
        env.pop("ZM_LIB", None)
        if variant == "checked":
            env["ZM_LIB"] = "checked"
        path = str(tmp_path / f"{variant}.npz")
        subprocess.run([sys.executable, os.path.abspath(__file__), path], env=env, check=True, timeout=600)
        out[variant] = dict(np.load(path))
    plain, chk = out["default"], out["checked"]
    assert plain.pop("build")[0] == 0
    checked, hits, first, line = (int(v) for v in chk.pop("build"))
    assert checked == 1 and hits == 0, f"{hits} index violations, first index {first} at line {line}"
    assert sorted(plain) == sorted(chk)
    for k in plain:
        assert np.all(np.isfinite(plain[k])) and np.array_equal(plain[k], chk[k]), k


if __name__ == "__main__":
    checked_cases(sys.argv[1])
