"""Fields set from and read into memory that the caller names as a device's:
the handle's own device by a kernel, anything else by a copy call, which
reaches it or answers with an error (page-locked host memory is reached)."""
import ctypes

import numpy as np
import pytest

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("shift", [0, 1, 2])   # bytes past the element's alignment
@pytest.mark.parametrize("where", ["cuda", "pinned"])
def test_on_device_pointers(where, shift, prec):
    import torch
    from paper_2011_14043_gb300 import Simulation
    from paper_2011_14043_gb300._lib import COMPS, lib
    n = (33, 7, 5)
    u0 = random_fields(*n, 2)
    dt = np.float64 if prec == "f64" else np.float32
    s = Simulation(*n, 1e-3, scheme="flod", precision=prec, cfl=3.0)
    for c, v in u0.items():
        raw = np.ascontiguousarray(v.astype(dt)).view(np.uint8).reshape(-1)
        buf = torch.zeros(raw.size + 16, dtype=torch.uint8)
        buf = buf.cuda() if where == "cuda" else buf.pin_memory()
        buf[shift:shift + raw.size].copy_(torch.from_numpy(raw))
        torch.cuda.synchronize()
        p = ctypes.c_void_p(buf.data_ptr() + shift)
        assert lib().fdtd_set_field(s._h, COMPS[c], p, 1) == 0
        s.synchronize()
        assert np.array_equal(s.get_field(c), v.astype(dt)), c
        buf.zero_()
        torch.cuda.synchronize()
        assert lib().fdtd_get_field(s._h, COMPS[c], p, 1) == 0
        s.synchronize()
        got = buf[shift:shift + raw.size].cpu().numpy().copy().view(dt)
        assert np.array_equal(got, raw.view(dt)), c     # (values: the walls' -0 comes back as 0)
        assert not buf[:shift].any() and not buf[shift + raw.size:].any()
    s.close()
