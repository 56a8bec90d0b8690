"""Cutoff sum with a core size delta beyond the cutoff c.

The decision |r|^2 <= c^2 does not involve delta, and holds to a relative band of 2^-20 of c around the
boundary whatever delta is.  The compared quantity of a far tile pair is |r|^2 + delta^2 in FP32, whose
rounding grows with delta^2, so these pairs need a wider window for the exact decision.  Reference and
tolerance are those of the cutoff tests: the oracle with the band pairs of each target assigned as the
result suggests, u to 1e-6 relative L2.  A single pair decided wrongly outside the band moves u of its
target by a percent or so, that is, u by 1e-4 in this norm.
"""
import pytest

import oracle
from paper_2406_05490_gb300 import inputs
from test_gpu_cutoff import TOL32, band_corrected_reference, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delta", [0.15, 0.8, 4.0, 15.0])
@pytest.mark.parametrize("n1,n2,periodic,cutoff", [(96, 80, True, 0.2), (128, 96, False, 0.2)])
def test_core_larger_than_the_cutoff(n1, n2, periodic, cutoff, delta):
    from paper_2406_05490_gb300 import zm
    z, w = inputs.random_state(n1, n2, seed=n1 + n2, periodic=periodic)
    model = zm.ZModel(n1, n2, periodic=periodic, atwood=0.5, g=1.0, delta=delta, fp32c=True)
    zm.zm_set_cutoff(model.h, cutoff)
    u, _ = model.velocity(z, w)
    model.close()
    m = oracle.Mesh(n1, n2, periodic=periodic)
    u_ref, _, nband, nflip = band_corrected_reference(m, z, w, u, 0.5, 1.0, 0.0, delta, cutoff)
    err = rel(u, u_ref)
    print(f"delta {delta} cutoff {cutoff} {n1}x{n2}: rel L2 u {err:.3e}; band pairs {nband}, flipped {nflip}")
    assert err <= TOL32
