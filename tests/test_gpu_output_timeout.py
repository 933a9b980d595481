"""A bounded wait that gives up in the output solve of a read (the FADI and
FLOD2 output transforms take the TMA-fed y/z kernel): the read itself answers
FDTD_ERR_TIMEOUT, and not the call after it.  The flag is set by the library's
test hook; the kernels run to their end."""
import numpy as np
import pytest

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu

TIMEOUT = -4
N = (64, 40, 48)
U0 = random_fields(*N, 2)


def stepped(scheme):
    from paper_2011_14043_gb300 import Simulation
    # tune[1] bit 7: a launch per pair on a grid of this size, y and z lines by the TMA-fed kernel
    s = Simulation(*N, 1e-3, scheme=scheme, precision="f32", cfl=4.0, tune=(0, 128))
    s.set_fields(U0)
    s.step(3)
    s.synchronize()
    return s


READS = {
    "host": lambda s: s.get_field("ez"),
    "device": lambda s: s.get_field("ez", device=True),
    "energy": lambda s: s.energy(),
    "set_field": lambda s: s.set_field("ez", U0["ez"]),
}


@pytest.mark.parametrize("read", sorted(READS))
@pytest.mark.parametrize("scheme", ["fadi", "flod2"])
@pytest.mark.parametrize("nth", [0, 1])
def test_timeout_of_the_output_solve_is_reported_by_the_read(scheme, read, nth):
    from paper_2011_14043_gb300 import FdtdError
    from paper_2011_14043_gb300._lib import lib
    s = stepped(scheme)
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
def test_timeout_of_a_step_is_reported_by_the_read(scheme):
    from paper_2011_14043_gb300 import FdtdError
    from paper_2011_14043_gb300._lib import lib
    s = stepped(scheme)
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
def test_reads_without_a_timeout(scheme):
    """Host and device reads of every component agree, before and after."""
    s = stepped(scheme)
    for _ in range(2):
        for c in U0:
            a = s.get_field(c, device=True).cpu().numpy()
            assert np.array_equal(a, s.get_field(c)), c
        s.step(2)
    s.close()
