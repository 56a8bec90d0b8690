"""The FP64 high-order sum (zm_brdw.cu) where a source split holds more than the 64 tiles that are
classified at once, so that both staging buffers are handed from one batch of tiles to the next.

192 x 184 nodes make 552 tiles in 8 splits of 69.  Against the oracle with the repository's FP64
bound, and bitwise equal between calls: a buffer overwritten while it is read would show as neither.
"""
import numpy as np
import pytest

import oracle
from paper_2406_05490_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL64 = 1e-12


def test_splits_of_more_than_64_tiles():
    from paper_2406_05490_gb300 import zm
    n1, n2 = 192, 184
    z, w = inputs.random_state(n1, n2, seed=7)
    delta = 0.1 / n1
    m = zm.ZModel(n1, n2, periodic=True, atwood=0.5, g=1.0, delta=delta)
    u, wd = m.velocity(z, w)
    again = [m.velocity(z, w) for _ in range(3)]
    m.close()
    u_ref, wd_ref = oracle.derivative(oracle.Mesh(n1, n2, periodic=True), z, w, 0.5, 1.0, 0.0, delta)
    eu, ew = (float(np.linalg.norm(a - b) / np.linalg.norm(b)) for a, b in ((u, u_ref), (wd, wd_ref)))
    print(f"192x184: rel L2 u {eu:.2e} wdot {ew:.2e}")
    assert eu <= TOL64 and ew <= TOL64
    assert all(np.array_equal(u, a) and np.array_equal(wd, b) for a, b in again)
