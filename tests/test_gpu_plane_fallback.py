"""Small 2-D grids on a device that cannot hold the plane kernel's cluster (the
library's test hook answers the question with no): the steps run by the other
kernels, as they do with a launch-shape override."""
import numpy as np
import pytest

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("scheme", ["fadi", "flod2"])
def test_steps_without_the_cluster(scheme, prec):
    from paper_2011_14043_gb300 import Simulation
    from paper_2011_14043_gb300._lib import lib
    n = (65, 50, 1)
    u0 = random_fields(*n, 3)
    cur = np.random.default_rng(1).standard_normal(12) * 1e-3

    def run(tune, refuse):
        s = Simulation(*n, 1e-3, scheme=scheme, precision=prec, cfl=4.0, tune=tune)
        s.set_fields(u0)
        s.set_source("ez", 30, 20, 0, cur)
        pids = [s.add_probe("ez", 12, 13, 0)] if prec == "f64" and scheme == "fadi" else []
        lib().fdtd_debug_fail_cluster(0 if refuse else -1)
        try:
            s.step(5)       # (asked at the first step alone)
            s.reset_stats()
            s.step(7)
        finally:
            lib().fdtd_debug_fail_cluster(-1)
        launches = s.stats()["launches"]
        out = {c: s.get_state(c) for c in u0}, [s.get_probe(p, 12) for p in pids]
        s.close()
        return launches, out

    one, plane = run((0, 0), False)
    many, other = run((0, 0), True)
    _, forced = run((0, 16), False)     # (tune[1] bit 4 takes another path than the plane kernel)
    assert one == 1 and many > 7
    for c in u0:
        assert np.array_equal(other[0][c], forced[0][c]), c
        tol = 1e-12 if prec == "f64" else 1e-4
        assert np.linalg.norm(other[0][c] - plane[0][c]) <= tol * np.linalg.norm(plane[0][c]), c
    assert all(np.array_equal(a, b) for a, b in zip(other[1], forced[1]))
