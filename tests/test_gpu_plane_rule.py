"""Which 2-D FP32 grids run every step of a call in one launch: up to 128 x 128
cells, with a source up to 256 cells a side; both sides of the line against
the FP64 oracle."""
import numpy as np
import pytest

from gpu_helpers import energy_norm_rel, oracle_problem, random_fields
from oracle import schemes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("source", [False, True])
@pytest.mark.parametrize("dims,plain", [((128, 128), True), ((256, 64), True), ((127, 129), True), ((129, 128), False),
                                        ((65, 256), False), ((200, 200), False), ((257, 20), None)])
def test_plane_line(dims, plain, source):
    from paper_2011_14043_gb300 import Simulation
    nx, ny = dims
    d, steps = 1e-3, 6
    u0 = random_fields(nx, ny, 1, 3)
    cur = np.random.default_rng(2).standard_normal(steps) * 1e-3
    s = Simulation(nx, ny, 1, d, scheme="fadi", precision="f32", cfl=5.0)
    s.set_fields(u0)
    src = ("ez", nx // 2, ny // 3, 0, cur) if source else None
    if source:
        s.set_source(*src)
    s.step(1)
    s.reset_stats()
    s.step(steps - 1)
    one = plain is not None and (plain or source)
    assert (s.stats()["launches"] == 1) == one
    w0 = {c: v.astype(np.float32).astype(np.float64) for c, v in u0.items()}
    ref, _, _ = S.run_fundamental(oracle_problem(nx, ny, 1, d, d, d, s.dt, source=src), "fadi", w0, steps)
    assert energy_norm_rel(s.get_fields(), ref) <= 1e-4     # the library's stated bound for a few steps
    s.close()
