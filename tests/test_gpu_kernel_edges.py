"""GPU kernels at the sizes where their indexing can go wrong (edges of rows,
segments and tiles, the shortest and longest lines), against the FP64 oracle."""
import numpy as np
import pytest

from gpu_helpers import energy_norm_rel, gpu_run, oracle_problem, random_fields
from oracle import schemes as S

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-12, "f32": 1e-4}   # the library's stated bounds for a few steps


def random_media(nx, ny, nz, seed):
    return np.random.default_rng(seed).uniform(1.0, 6.0, (nz, ny, nx))


def check(nx, ny, nz, scheme, prec, steps=4, eps=None, tune=(0, 0), cfl=4.0):
    d = 1e-3
    dt = cfl * d / (299792458.0 * np.sqrt(3.0 if nz > 1 else 2.0))
    u0 = random_fields(nx, ny, nz, 11)
    out, _, _, sim = gpu_run(nx, ny, nz, d, d, d, dt, scheme, prec, u0, steps, eps=eps, tune=tune)
    sim.close()
    if prec == "f32":
        u0 = {c: v.astype(np.float32).astype(np.float64) for c, v in u0.items()}
    ref, _, _ = S.run_fundamental(oracle_problem(nx, ny, nz, d, d, d, dt, eps=eps), scheme, u0, steps)
    err = energy_norm_rel(out, ref)
    assert err <= TOL[prec], err
    return out


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", [(2, 2, 1), (2, 2, 2), (3, 2, 5), (31, 5, 4), (32, 4, 33), (33, 65, 3), (127, 3, 64)])
def test_media_formed_on_the_device(dims, prec):
    """Per-cell eps: means at the samples and line pivots from the device kernels."""
    check(*dims, "flod", prec, eps=random_media(*dims, 5))


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("media", ["uniform", "blocks"])
@pytest.mark.parametrize("dims", [(2, 2, 2), (15, 9, 8), (16, 32, 7), (17, 33, 31), (64, 31, 32), (65, 64, 5),
                                  (128, 5, 65), (129, 97, 3), (256, 3, 129), (5, 161, 96), (6, 256, 9), (3, 4, 255),
                                  (33, 40, 1)])
def test_procedure_in_one_launch(dims, media, prec):
    """Lines along y, z and x of one procedure in one launch: line lengths on
    both sides of a segment (8), a warp (32) and a tile (256), odd numbers of
    columns, a source on the first and last unknown, runs of 16 steps and
    single ones."""
    from paper_2011_14043_gb300 import Simulation
    nx, ny, nz = dims
    d, steps = 1e-3, 19
    eps = random_media(nx, ny, nz, 3) if media == "blocks" else None
    u0 = random_fields(nx, ny, nz, 7)
    dt = 5.0 * d / (299792458.0 * np.sqrt(3.0 if nz > 1 else 2.0))
    cur = np.random.default_rng(1).standard_normal(steps) * 1e-3
    for scheme, at in (("fadi", (1, 1, 0)), ("fss", (nx - 1, ny - 1, nz - 1)), ("flod2", (nx // 2, ny // 2, nz // 2))):
        # (homogeneous grids with a source take the kernels of a launch per pair)
        src = ("ez",) + at + (cur,) if media == "blocks" or scheme == "flod2" else None
        out, _, _, sim = gpu_run(nx, ny, nz, d, d, d, dt, scheme, prec, u0, steps, eps=eps, source=src)
        sim.close()
        w0 = {c: v.astype(np.float32).astype(np.float64) if prec == "f32" else v for c, v in u0.items()}
        ref, _, _ = S.run_fundamental(oracle_problem(nx, ny, nz, d, d, d, dt, eps=eps, source=src), scheme, w0, steps)
        err = energy_norm_rel(out, ref)
        assert err <= TOL[prec], (scheme, err)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", [(2, 2, 1), (3, 5, 1), (16, 17, 1), (64, 64, 1), (65, 33, 1), (63, 128, 1), (128, 127, 1),
                                  (256, 20, 1)])
def test_plane_steps_in_one_launch(dims, prec):
    """2-D grids whose steps run in one launch: lines on both sides of a
    lane's 2, 4 and 8 nodes, strips of one to several rows, a source and (FP64)
    probes of every component at it, beside it and on the walls."""
    nx, ny, nz = dims
    d, steps = 1e-3, 7
    u0 = random_fields(nx, ny, nz, 5)
    dt = 5.0 * d / (299792458.0 * np.sqrt(2.0))
    cur = np.random.default_rng(2).standard_normal(steps) * 1e-3
    i, j = nx // 2, ny - 1
    probes = [] if prec == "f32" else [("ez", i, j, 0), ("ez", 1, 1, 0), ("hx", nx, 0, 0), ("hy", 0, ny, 0),
                                       ("hz", 0, 0, 1), ("hy", nx - 1, 1, 0), ("hx", 1, ny - 1, 0)]
    w0 = {c: v.astype(np.float32).astype(np.float64) if prec == "f32" else v for c, v in u0.items()}
    for scheme in ("fadi", "flod", "fss", "flod2"):
        src = ("ez", i, j, 0, cur)
        pr = probes if scheme != "flod2" else []
        out, series, _, sim = gpu_run(nx, ny, nz, d, d, d, dt, scheme, prec, u0, steps, source=src, probes=pr)
        sim.close()
        P = oracle_problem(nx, ny, nz, d, d, d, dt, source=src)
        ref, _, want = S.run_fundamental(P, scheme, w0, steps, probes=pr)
        assert energy_norm_rel(out, ref) <= TOL[prec], scheme
        for a, b in zip(series, want):
            assert np.max(np.abs(a - b)) <= TOL[prec] * max(np.max(np.abs(b)), 1e-300), scheme


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", [(2, 3, 1), (31, 4, 3), (32, 5, 2), (255, 3, 4), (256, 2, 3), (257, 3, 2), (520, 2, 2)])
def test_device_copies_of_every_component(dims, prec):
    """Fields set from and read into device memory: rows on both sides of a
    warp (32) and of a lane's 8 elements in flight (256), from tensors that
    start one element into their storage; before a step and after FADI's
    output processing (wall samples of H included)."""
    import torch
    from paper_2011_14043_gb300 import Simulation
    u0 = random_fields(*dims, 3)
    dt = torch.float64 if prec == "f64" else torch.float32
    npt = np.float64 if prec == "f64" else np.float32
    for scheme in ("flod", "fadi"):
        host = Simulation(*dims, 1e-3, scheme=scheme, precision=prec, cfl=3.0)
        dev = Simulation(*dims, 1e-3, scheme=scheme, precision=prec, cfl=3.0)
        for c, v in u0.items():
            host.set_field(c, v)
            store = torch.empty(v.size + 1, dtype=dt, device="cuda")
            t = store[1:].view(*v.shape)
            t.copy_(torch.from_numpy(v))
            dev.set_field(c, t)
            assert np.array_equal(dev.get_field(c, device=True).cpu().numpy(), v.astype(npt)), c
        host.step(2)
        dev.step(2)
        for c in u0:
            a = host.get_field(c)
            assert np.array_equal(dev.get_field(c, device=True).cpu().numpy(), a), (scheme, c)
        for c, w in (("hx", (slice(None), slice(None), 0)), ("hy", (slice(None), -1)), ("hz", (0,))):
            assert np.array_equal(host.get_field(c)[w], u0[c].astype(npt)[w]), c
        host.close()
        dev.close()


@pytest.mark.parametrize("media", ["uniform", "blocks", "both"])
@pytest.mark.parametrize("scheme", ["fadi", "fss"])
def test_batch_in_one_launch_per_procedure(scheme, media):
    """An FP32 batch whose shapes the tuner may choose: grids of one to eight
    warps per tile, x lines on 8, 16 and 32 lanes, runs of 16 steps and single
    ones; against the oracle, and (where the batch took one launch per
    procedure) bit for bit against the grids stepped alone."""
    from paper_2011_14043_gb300 import Batch, Simulation
    grids = [(20, 30, 9), (70, 97, 33), (130, 12, 70), (16, 129, 5), (9, 8, 250)]
    steps = 18
    sims, alone, refs = [], [], []
    for q, (nx, ny, nz) in enumerate(grids):
        u0 = random_fields(nx, ny, nz, 20 + q)
        eps = random_media(nx, ny, nz, q) if media == "blocks" or (media == "both" and q % 2) else None
        for out in (sims, alone):
            s = Simulation(nx, ny, nz, 1e-3, scheme=scheme, precision="f32", cfl=3.0 + q)
            if eps is not None:
                s.set_material(eps)
            s.set_fields(u0)
            out.append(s)
        w0 = {c: v.astype(np.float32).astype(np.float64) for c, v in u0.items()}
        refs.append(S.run_fundamental(oracle_problem(nx, ny, nz, 1e-3, 1e-3, 1e-3, sims[-1].dt, eps=eps), scheme, w0,
                                      steps)[0])
    b = Batch(sims)
    b.step(1)
    b.step(steps - 1)
    procedures = 3 if scheme == "fss" else 2
    fused = b.launches_per_step() <= procedures * (2 if media == "both" else 1)
    for q, s in enumerate(sims):
        got = s.get_fields()
        assert energy_norm_rel(got, refs[q]) <= TOL["f32"], q
        if fused:
            alone[q].step(steps)
            for c in ("hx", "hy", "hz"):
                assert np.array_equal(alone[q].get_state(c), s.get_state(c)), (q, c)
    b.close()


@pytest.mark.parametrize("dims", [(70, 90, 110), (130, 40, 257), (512, 30, 40)])
def test_fourth_order_kernels_of_many_blocks(dims):
    """Fourth-order lines in launches of more than two blocks per SM (E and H
    read twice) and fewer: bit for bit the one-thread-per-line kernel's."""
    from paper_2011_14043_gb300 import Simulation
    u0 = random_fields(*dims, 4)
    out = []
    for tune in ((0, 0), (0, 512)):
        s = Simulation(*dims, 1e-3, scheme="fss", precision="f32", cfl=4.0, tune=tune)
        s.set_order(4)
        s.set_fields(u0)
        s.step(2)
        out.append({c: s.get_field(c) for c in u0})
        s.close()
    for c in u0:
        assert np.array_equal(out[0][c], out[1][c]), c
