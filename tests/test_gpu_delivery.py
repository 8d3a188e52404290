"""One dataset with device pointers: the counts reach the caller's buffer at
any address, as a copy takes them there, and nothing around it is touched."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1, 2, 3, 4, 6])
@pytest.mark.parametrize("m", [1, 5, 300])
def test_counts_at_any_address(offset, m):
    import torch
    from paper_1409_3901_gb300 import tukey
    g = np.random.default_rng(m)
    x = g.integers(-20, 21, (30, 3)).astype(np.int32)
    z = g.integers(-20, 21, (m, 3)).astype(np.int32)
    want = tukey.Context(0).depth(x, z)
    xd, zd = torch.from_numpy(x).cuda(), torch.from_numpy(z).cuda()
    buf = torch.full((4 * m + 16,), 0x5A, dtype=torch.uint8, device="cuda")
    ctx = tukey.Context(0, device_pointers=True)
    rc = tukey.lib.td_depth(ctx.ptr, ctypes.c_void_p(xd.data_ptr()), 30, 3, ctypes.c_void_p(zd.data_ptr()), m,
                            ctypes.c_void_p(buf.data_ptr() + offset), None)
    assert rc == tukey.TD_OK
    got = buf.cpu().numpy()
    assert np.array_equal(np.frombuffer(got[offset:offset + 4 * m].tobytes(), np.int32), want)
    assert (got[:offset] == 0x5A).all() and (got[offset + 4 * m:] == 0x5A).all()
