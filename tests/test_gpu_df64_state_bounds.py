"""Double-word contexts convert device arrays in place, by kernels that read or write them.  An array that
runs past the end of its allocation is refused on the host, as the copy that such a call once began with
was refused, and nothing is launched; arrays that end with their allocation are used in place."""
import pytest

pytestmark = pytest.mark.gpu


def test_arrays_that_run_past_their_allocation_are_refused():
    import torch
    from paper_2406_05490_gb300 import zm
    n = 2048
    N = n * n
    m = zm.ZModel(n, order=zm.ZM_ORDER_LOW, df64=True)
    whole = torch.zeros(1 << 25, dtype=torch.float64, device="cuda")  # 256 MB: an allocation of its own
    ok_z, ok_w = whole[: 3 * N], whole[3 * N: 5 * N]
    last = whole[-3 * N:]  # ends with the allocation
    short = whole[-(1 << 16):].data_ptr()  # 512 KB before its end
    zm.zm_set_state(m.h, ok_z, ok_w)
    for z, w in ((short, ok_w), (ok_z, short)):
        for call in (lambda: zm.zm_set_state(m.h, z, w), lambda: zm.zm_velocity(m.h, z, w, ok_z)):
            with pytest.raises(zm.ZMError):
                call()
    zm.zm_get_state(m.h, last, None)
    zm.zm_set_state(m.h, last, ok_w)
    m.sync()  # nothing failed on the device
    m.close()
