"""Captured runs of 16 fused steps, chained by programmatic edges, against the
same launches one by one: bit for bit, over runs, single steps and both, with
a source inside the launches (per-node media) and without."""
import numpy as np
import pytest

from gpu_helpers import random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(40, 33, 28), (96, 64, 80), (256, 20, 17), (9, 250, 5)])
@pytest.mark.parametrize("media", ["uniform", "blocks", "source"])
@pytest.mark.parametrize("scheme", ["fadi", "flod", "fss", "flod2"])
def test_fused_graphs_bit_identical_to_single_launches(scheme, media, dims):
    from paper_2011_14043_gb300 import Simulation
    nx, ny, nz = dims
    u0 = random_fields(*dims, 4)
    eps = np.random.default_rng(6).uniform(1.0, 6.0, dims[::-1])
    cur = np.random.default_rng(7).standard_normal(60) * 1e-3
    sims = []
    for path in (0, 8):    # tune[1] bit 3: launches one by one
        s = Simulation(*dims, 1e-3, scheme=scheme, precision="f32", cfl=5.0, tune=(0, path))
        if media != "uniform":
            s.set_material(eps)
        s.set_fields(u0)
        if media == "source":
            s.set_source("ex", nx // 2, ny // 2, nz // 2, cur)
        sims.append(s)
    procedures = 3 if scheme == "fss" else 2
    for n in (1, 16, 37, 3):
        sims[0].reset_stats()
        for s in sims:
            s.step(n)
        # (one launch per procedure: the fused kernels ran; FLOD2 and FADI start with a few of their own)
        if n == 37:
            counters = 2 + 5 if media == "source" else 0
            assert procedures * n <= sims[0].stats()["launches"] <= procedures * n + counters
        for c in u0:
            assert np.array_equal(sims[0].get_state(c), sims[1].get_state(c)), (n, c)
    for s in sims:
        s.close()


@pytest.mark.parametrize("dims,lines", [((190, 180, 182), True), ((190, 100, 182), True), ((60, 50, 40), False)])
def test_fp64_probed_graphs_bit_identical_to_single_launches(dims, lines):
    """Per-node media with a probe and a source, with pairs of at least 32768 lines
    along y and z, along y alone, and of fewer (the former captured one
    after the other, the latter on parallel branches)."""
    from paper_2011_14043_gb300 import Simulation
    nx, ny, nz = dims
    assert (nx * nz >= 32768) == lines
    eps = np.random.default_rng(6).uniform(1.0, 6.0, dims[::-1])
    u0 = random_fields(*dims, 4)
    cur = np.random.default_rng(7).standard_normal(9) * 1e-3
    got = []
    for path in (0, 8):
        s = Simulation(*dims, 1e-3, scheme="fadi", precision="f64", cfl=5.0, tune=(0, path))
        s.set_material(eps)
        s.set_fields(u0)
        s.set_source("ez", nx // 2, ny // 2, nz // 2, cur)
        pids = [s.add_probe("ez", nx // 2, ny // 2, nz // 2), s.add_probe("hx", 3, 4, 5)]
        s.step(3)
        s.step(4)
        got.append([s.get_state(c) for c in u0] + [s.get_probe(p, 7) for p in pids])
        s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*got))
