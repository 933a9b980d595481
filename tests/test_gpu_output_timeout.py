"""A bounded wait that gives up in the output solve of a read (the FADI and
FLOD2 output transforms of large grids take the TMA-fed y/z kernel): the read itself answers
FDTD_ERR_TIMEOUT, and not the call after it.  The flag is set by the library's
test hook; the kernels run to their end."""
import numpy as np
import pytest

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu

TIMEOUT = -4
N = (256, 200, 216)     # (beyond the line of the fused procedures)
SMALL = (64, 40, 48)


@pytest.fixture(scope="module")
def u0():
    import torch
    return {c: torch.from_numpy(v.astype(np.float32)).cuda() for c, v in random_fields(*N, 2).items()}


def stepped(scheme, u0, n=N, tune=(0, 0)):
    from paper_2011_14043_gb300 import Simulation
    s = Simulation(*n, 1e-3, scheme=scheme, precision="f32", cfl=4.0, tune=tune)
    s.set_fields(u0)
    s.step(3)
    s.synchronize()
    return s


READS = {
    "host": lambda s: s.get_field("ez"),
    "device": lambda s: s.get_field("ez", device=True),
    "energy": lambda s: s.energy(),
    "set_field": lambda s: s.set_field("ez", np.zeros(s.shape("ez"), np.float32)),
}


@pytest.mark.parametrize("read", sorted(READS))
@pytest.mark.parametrize("scheme", ["fadi", "flod2"])
@pytest.mark.parametrize("nth", [0, 1])
def test_timeout_of_the_output_solve_is_reported_by_the_read(scheme, read, nth, u0):
    from paper_2011_14043_gb300 import FdtdError
    from paper_2011_14043_gb300._lib import lib
    s = stepped(scheme, u0)
    try:
        assert lib().fdtd_debug_fail_wait(nth) == 0   # the y or the z lines of the output solve
        with pytest.raises(FdtdError) as err:
            READS[read](s)
        assert err.value.code == TIMEOUT
    finally:
        lib().fdtd_debug_fail_wait(-1)
    with pytest.raises(FdtdError) as err:             # the samples stay unusable
        s.get_field("hx", device=True)
    assert err.value.code == TIMEOUT
    s.close()


@pytest.mark.parametrize("scheme", ["fadi", "flod2"])
def test_timeout_of_a_step_is_reported_by_the_read(scheme, u0):
    from paper_2011_14043_gb300 import FdtdError
    from paper_2011_14043_gb300._lib import lib
    s = stepped(scheme, u0)
    try:
        lib().fdtd_debug_fail_wait(0)
        s.set_timing(True)    # launches one by one (a captured step counted at its capture)
        s.step(1)
    finally:
        lib().fdtd_debug_fail_wait(-1)
    with pytest.raises(FdtdError) as err:
        s.get_field("ez", device=True)
    assert err.value.code == TIMEOUT
    s.close()


@pytest.mark.parametrize("scheme", ["fadi", "flod2"])
def test_reads_without_a_timeout(scheme, u0):
    """Host and device reads of every component agree, before and after."""
    s = stepped(scheme, u0)
    for _ in range(2):
        for c in u0:
            a = s.get_field(c, device=True).cpu().numpy()
            assert np.array_equal(a, s.get_field(c)), c
        s.step(2)
    s.close()


@pytest.mark.parametrize("scheme", ["fadi", "flod2"])
def test_small_grids_solve_their_output_without_waits(scheme):
    """Below that line the output solve has no wait to check, whatever kernels
    the steps take (tune[1] bit 7: a launch per pair, TMA-fed y/z lines)."""
    from paper_2011_14043_gb300._lib import lib
    fields = random_fields(*SMALL, 3)
    s = stepped(scheme, fields, SMALL, (0, 128))
    try:
        lib().fdtd_debug_fail_wait(0)
        a = s.get_field("ez", device=True).cpu().numpy()
    finally:
        lib().fdtd_debug_fail_wait(-1)
    assert np.array_equal(a, s.get_field("ez"))
    s.close()
