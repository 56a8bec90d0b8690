"""The double-word state's conversions on device arrays (integer splitting and joining) against the
plain conversions that host arrays take: the same FP64 state put in either way has to step and come back
the same, at magnitudes inside and outside the integer form's range, on both kinds of side.

A double word holds at least 48 bits of each displacement, in either conversion: the states read back
differ from what was put in by at most 2^-48 of the displacement and one FP64 rounding of the sum with the
mesh coordinate (2^-53)."""
import numpy as np
import pytest

from paper_2406_05490_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(8, 8), (24, 40), (64, 512)])
def test_device_arrays_equal_host_arrays(n1, n2):
    import torch
    from paper_2406_05490_gb300 import zm
    z, w = inputs.random_state(n1, n2, seed=n1)
    N = n1 * n2
    rng = np.random.default_rng(n2)
    # strengths over the whole FP32 range and beyond the integer form's, with zeros, both signs and ties
    w *= np.exp2(rng.integers(-110, 90, size=w.shape))
    w[0, : N // 8] = 0.0
    w[1, : N // 8] = np.ldexp(1.0 + 2.0 ** -24, 3) * rng.choice([-1.0, 1.0], N // 8)
    z[2] *= np.exp2(rng.integers(-70, 3, size=N))
    m = zm.ZModel(n1, n2, order=zm.ZM_ORDER_LOW, df64=True)
    m.set_state(z, w)
    zh, wh = m.get_state()
    zd, wd = torch.from_numpy(z).cuda(), torch.from_numpy(w).cuda()
    zo, wo = torch.empty_like(zd), torch.empty_like(wd)
    zm.zm_set_state(m.h, zd, wd)
    zm.zm_get_state(m.h, zo, wo)
    m.sync()
    assert np.array_equal(zo.cpu().numpy(), zh) and np.array_equal(wo.cpu().numpy(), wh)
    a, b = inputs.mesh_coords(n1, n2)
    disp = z - np.stack([a, b, 0 * a])
    assert np.all(np.abs(zh - z) <= 2.0 ** -48 * np.abs(disp) + 2.0 ** -52 * np.abs(z) + 1e-44)
    assert np.all(np.abs(wh - w) <= 2.0 ** -48 * np.abs(w) + 1e-44)
    # either array alone, and a step from either kind of input
    only = torch.empty_like(wd)
    zm.zm_get_state(m.h, None, only)
    m.sync()
    assert torch.equal(only, wo)
    w2 = inputs.random_state(n1, n2, seed=1)[1]
    m.set_state(z, w2)
    m.step(1e-4, 1)
    zs, ws = m.get_state()
    zm.zm_set_state(m.h, zd, torch.from_numpy(w2).cuda())
    m.step(1e-4, 1)
    z2, w3 = m.get_state()
    m.close()
    assert np.array_equal(zs, z2) and np.array_equal(ws, w3)
