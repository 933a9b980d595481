"""A batch or a reverse-mode context keeps its handles on the kernels it runs
them by while it lives, and no longer: afterwards (and after a creation that
failed) they step as a handle that never was in one.  Seen by the launches of
a step (one per procedure where the fused kernel runs, one per pair where it
does not) and by the bits."""
import ctypes

import numpy as np
import pytest

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu

N = (40, 33, 28)
U0 = random_fields(*N, 1)
EPS = np.random.default_rng(5).uniform(1.0, 4.0, N[::-1])


def make(media):
    from paper_2011_14043_gb300 import Simulation
    s = Simulation(*N, 1e-3, scheme="fadi", precision="f32", cfl=4.0)
    if media == "blocks":
        s.set_material(EPS)
    s.set_fields(U0)
    return s


def launches(s, n):
    s.step(1)       # (captures)
    s.reset_stats()
    s.step(n)
    return s.stats()["launches"] / n


def same(a, b):
    for c in U0:
        assert np.array_equal(a.get_state(c), b.get_state(c)), c


@pytest.mark.parametrize("media", ["uniform", "blocks"])
def test_after_a_batch(media):
    from paper_2011_14043_gb300 import Batch
    a, b, fresh = make(media), make(media), make(media)
    assert launches(a, 4) == 2 and launches(fresh, 4) == 2
    one, two = Batch([a, b]), Batch([a])
    if media == "uniform":
        assert launches(a, 4) == 6      # while a batch lives
        one.close()
        assert launches(a, 4) == 6      # two of them
    one.close()
    two.close()
    assert launches(a, 32) == 2
    # a handle that was only put into a batch has the bits of one that never was
    three = Batch([b])
    three.close()
    b.step(24)
    fresh.step(19)
    same(b, fresh)
    for s in (a, b, fresh):
        s.close()


def test_batch_destroyed_after_its_handles():
    from paper_2011_14043_gb300 import Batch
    sims = [make("uniform"), make("blocks")]
    b = Batch(sims)
    b.step(2)
    b.synchronize()
    for s in sims:
        s.close()
    b.close()


def adj_create(s, ok=True):
    from paper_2011_14043_gb300._lib import lib
    h = ctypes.c_void_p()
    blk = (ctypes.c_int32 * 6)(2, 4, 2, 4, 2, 4)
    rc = lib().fdtd_adj_create(s._h, blk, 6, 3, ctypes.byref(h))
    assert (rc == 0) == ok, rc
    return h


def test_after_a_context():
    from paper_2011_14043_gb300._lib import lib
    s, fresh = make("blocks"), make("blocks")
    # a creation that runs out of memory leaves the handle as it was
    lib().fdtd_debug_fail_alloc(0)
    try:
        adj_create(s, ok=False)
    finally:
        lib().fdtd_debug_fail_alloc(-1)
    h, h2 = adj_create(s), adj_create(s)
    lib().fdtd_adj_destroy(h)
    lib().fdtd_adj_destroy(h2)
    s.step(20)
    fresh.step(20)
    same(s, fresh)
    assert launches(s, 16) == 2
    s.close()
    fresh.close()


def test_after_a_failed_context():
    from paper_2011_14043_gb300._lib import lib
    s = make("blocks")
    lib().fdtd_debug_fail_alloc(0)
    try:
        adj_create(s, ok=False)
    finally:
        lib().fdtd_debug_fail_alloc(-1)
    assert launches(s, 16) == 2
    s.close()


def test_while_a_context_lives():
    from paper_2011_14043_gb300._lib import lib
    s = make("blocks")
    h, J = adj_create(s), ctypes.c_double()
    assert lib().fdtd_adj_forward(h, ctypes.byref(J)) == 0
    assert launches(s, 4) == 6
    lib().fdtd_adj_destroy(h)
    assert launches(s, 4) == 2
    s.close()
