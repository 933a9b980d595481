"""Reverse mode and what its handle is given around it: the reverse pass belongs to the run
that fdtd_adj_forward made, whatever source the handle is given before,
between and after the passes; probe sets larger than one block takes."""
import numpy as np
import pytest

from oracle import adjoint as AD
from oracle import grid as G

from gpu_helpers import oracle_problem, random_fields

pytestmark = pytest.mark.gpu

N = (14, 12, 10)
STEPS, EVERY = 9, 4
BLOCK = (8, 12, 3, 8, 2, 7)
EPS = np.random.default_rng(3).uniform(1.0, 6.0, N[::-1])
CUR = np.random.default_rng(4).standard_normal(STEPS + 1) * 1e-5
SOURCE = ("ez", 5, 6, 4, CUR)
DT = 4.0 * G.Grid(*N, 1e-3, 1e-3, 1e-3).dt_cfl()
U0 = random_fields(*N, 6)


def start(prec, source, block=BLOCK):
    from paper_2011_14043_gb300.adjoint import AdjointRun, ProbeEnergyProblem
    return AdjointRun(ProbeEnergyProblem(*N, 1e-3, steps=STEPS, probe_block=block, dt=DT, precision=prec,
                                         checkpoint_every=EVERY, source=source, fields=U0), EPS)


def gradient(run, jbar=1.0):
    return run.backward(jbar, out=np.empty_like(EPS))


def oracle(source, block=BLOCK):
    P = oracle_problem(*N, 1e-3, 1e-3, 1e-3, DT, eps=EPS, source=source)
    J, g, _ = AD.gradient(P, U0, STEPS, AD.probe_masks(G.Grid(*N, 1e-3, 1e-3, 1e-3), block))
    return J, g


# other sources: a longer table, a shorter one, another sample, another component, none
OTHERS = [SOURCE[:4] + (np.ones(4096),), SOURCE[:4] + (np.ones(2),), ("ez", 3, 4, 5, 2 * CUR),
          ("ex", 7, 5, 3, np.ones(77)), ("ez", 0, 0, 0, np.empty(0))]


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_repeated_reverse_passes_keep_the_source_of_the_forward_run(prec):
    J_ref, g_ref = oracle(SOURCE)
    run = start(prec, SOURCE)
    J = run.forward()
    g = gradient(run)
    assert abs(J / J_ref - 1.0) <= (1e-12 if prec == "f64" else 1e-4)
    assert np.linalg.norm(g - g_ref) <= (1e-6 if prec == "f64" else 1e-3) * np.linalg.norm(g_ref)
    for other in OTHERS:
        run.sim.set_source(*other)
        assert np.array_equal(gradient(run), g), other[:4]
    # another scale, and back
    assert np.array_equal(gradient(run, -2.0), -2.0 * g)   # (a power of two: exact)
    assert np.array_equal(gradient(run), g)
    run.close()


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("first", [None, ("ex", 7, 5, 3, np.ones(3))])
def test_the_source_set_before_the_forward_run_counts(first, prec):
    """The context is created on a handle without a source, or with another
    one of another component, sample and length."""
    run = start(prec, first)
    run.sim.set_source(*SOURCE)
    J = run.forward()
    g = gradient(run)
    run.close()
    same = start(prec, SOURCE)
    assert same.forward() == J
    assert np.array_equal(gradient(same), g)
    same.close()
    J_ref, g_ref = oracle(SOURCE)
    assert abs(J / J_ref - 1.0) <= (1e-12 if prec == "f64" else 1e-4)
    assert np.linalg.norm(g - g_ref) <= (1e-6 if prec == "f64" else 1e-3) * np.linalg.norm(g_ref)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_probe_sets_of_more_than_4096_samples(prec):
    """Every interior E sample of a 16 x 16 x 12 part of the grid as a probe."""
    from paper_2011_14043_gb300.adjoint import AdjointRun, ProbeEnergyProblem
    n, block = (18, 17, 14), (1, 17, 0, 16, 1, 13)
    eps = np.random.default_rng(8).uniform(1.0, 6.0, n[::-1])
    u0 = random_fields(*n, 9)
    g = G.Grid(*n, 1e-3, 1e-3, 1e-3)
    dt = 4.0 * g.dt_cfl()
    src = ("ey", 9, 8, 7, CUR)
    masks = AD.probe_masks(g, block)
    assert sum(int(np.sum(m)) for m in masks.values()) > 4096
    J_ref, g_ref, _ = AD.gradient(oracle_problem(*n, 1e-3, 1e-3, 1e-3, dt, eps=eps, source=src), u0, STEPS, masks)
    run = AdjointRun(ProbeEnergyProblem(*n, 1e-3, steps=STEPS, probe_block=block, dt=dt, precision=prec,
                                        checkpoint_every=EVERY, source=src, fields=u0), eps)
    J = run.forward()
    got = run.backward(1.0, out=np.empty_like(eps))
    run.close()
    assert abs(J / J_ref - 1.0) <= (1e-12 if prec == "f64" else 1e-4)
    assert np.linalg.norm(got - g_ref) <= (1e-6 if prec == "f64" else 1e-3) * np.linalg.norm(g_ref)


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_media_set_after_the_context(prec):
    """Media that fdtd_adj_create refuses are refused by the forward pass too
    when they come after it (uniform eps has no per-node arrays to read);
    another per-node eps is taken."""
    import ctypes
    from paper_2011_14043_gb300 import Simulation
    from paper_2011_14043_gb300._lib import lib
    L = lib()
    one = np.ones_like(EPS)
    mu = one.copy()
    mu[:, :, :5] = 2.0
    blk = (ctypes.c_int32 * 6)(*BLOCK)
    for later, want in (((one, None, None), -6), ((EPS, mu, None), -6), ((EPS, None, 1e-3 * one), -6),
                        ((EPS, None, None), 0)):
        sim = Simulation(*N, 1e-3, scheme="fadi", precision=prec, dt=DT)
        sim.set_material(0.5 + EPS)
        sim.set_fields(U0)
        sim.set_source(*SOURCE)
        h, J = ctypes.c_void_p(), ctypes.c_double()
        assert L.fdtd_adj_create(sim._h, blk, STEPS, EVERY, ctypes.byref(h)) == 0
        sim.set_material(*later)
        assert L.fdtd_adj_forward(h, ctypes.byref(J)) == want
        if want == 0:
            g = np.empty_like(EPS)
            assert L.fdtd_adj_backward(h, 1.0, g.ctypes.data_as(ctypes.c_void_p), 0) == 0
            same = start(prec, SOURCE)
            assert same.forward() == J.value
            assert np.array_equal(gradient(same), g)
            same.close()
        L.fdtd_adj_destroy(h)
        sim.close()


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_launch_timing_in_reverse_mode(prec):
    """fdtd_set_timing counts the line solves of the forward and the
    recomputed steps, and changes no result."""
    run = start(prec, SOURCE)
    J = run.forward()
    g = gradient(run)
    run.close()
    run = start(prec, SOURCE)
    run.sim.set_timing(True)
    assert run.forward() == J
    st = run.sim.stats()
    assert st["timed_launches"] == [2 * STEPS] * 3 and min(st["timed_ms"]) > 0
    assert np.array_equal(gradient(run), g)
    assert run.sim.stats()["timed_launches"] == [4 * STEPS] * 3
    run.sim.set_timing(False)       # (and captured steps after timed ones)
    assert np.array_equal(gradient(run), g)
    assert run.sim.stats()["timed_launches"] == [4 * STEPS] * 3
    run.close()


def test_launch_timing_of_long_runs():
    """More timed launches than are kept unresolved (4096), on parallel branches."""
    from paper_2011_14043_gb300.adjoint import AdjointRun, ProbeEnergyProblem
    n, steps = (9, 8, 7), 700
    run = AdjointRun(ProbeEnergyProblem(*n, 1e-3, steps=steps, probe_block=(2, 4, 2, 4, 2, 4), cfl=4.0,
                                        precision="f32", checkpoint_every=50), np.ones(n[::-1]))
    run.sim.set_timing(True)
    run.forward()
    assert run.sim.stats()["timed_launches"] == [2 * steps] * 3
    run.close()
