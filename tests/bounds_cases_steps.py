"""Cases for the bounds-checked build beside bounds_cases.py: the kernels that
run when a handle has no probe or override to keep it from them.  One launch
per procedure (homogeneous and per-node media, with and without a source),
2-D grids with every step in one launch, both block-tiled fourth-order
kernels, copies into and out of device tensors, batches, and reverse passes of
more probes than one block injects."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

import workloads as W  # noqa: E402
from gpu_helpers import COMPS, random_fields  # noqa: E402


def main(out_path):
    import torch
    from paper_2011_14043_gb300 import Batch, Simulation
    from paper_2011_14043_gb300.adjoint import ProbeEnergyProblem
    out = {}

    def save(tag, sim):
        sim.synchronize()  # raises FdtdError (FDTD_ERR_BOUNDS) after a bounds violation
        dev = {c: sim.get_field(c, device=True) for c in COMPS}
        sim.synchronize()
        for c in COMPS:
            out[f"{tag}/{c}"] = sim.get_field(c)
            assert np.array_equal(dev[c].cpu().numpy(), out[f"{tag}/{c}"]), (tag, c)
        out[f"{tag}/energy"] = np.array(sim.energy())

    def make(dims, scheme, prec, media, tune=(0, 0)):
        nx, ny, nz = dims
        s = Simulation(nx, ny, nz, 1e-3, scheme=scheme, precision=prec, cfl=5.0, tune=tune)
        if media == "blocks":
            s.set_material(W.eps_blocks(7, nx, ny, nz, 1.0, 4.0))
        for c, v in random_fields(nx, ny, nz, seed=nx + ny + nz).items():
            s.set_field(c, torch.from_numpy(v).cuda())
        return s

    current = np.random.default_rng(2).standard_normal(40) * 1e-4

    # one launch per procedure: lines up to the 256 nodes of a tile, odd columns
    for dims in [(37, 29, 23), (20, 256, 7), (256, 12, 9), (7, 9, 255), (2, 2, 2), (65, 64, 33)]:
        for scheme in ("fadi", "fss"):
            for media in ("uniform", "blocks", "source"):
                s = make(dims, scheme, "f32", "blocks" if media == "source" else media)
                if media == "source":
                    s.set_source("ez", dims[0] - 1, 1, dims[2] - 1, current)
                s.step(18)
                save(f"fused/{dims}/{scheme}/{media}", s)
                s.close()
    # planes
    for prec, sizes in (("f64", [(2, 2), (17, 33), (64, 64), (128, 127)]), ("f32", [(3, 2), (65, 33), (256, 250)])):
        for nx, ny in sizes:
            for scheme in ("fadi", "flod", "fss", "flod2"):
                s = make((nx, ny, 1), scheme, prec, "uniform")
                s.set_source("ez", nx - 1, 1, 0, current)
                pid = s.add_probe("ez", nx // 2, ny // 2, 0) if prec == "f64" and scheme != "flod2" else None
                s.step(9)
                if pid is not None:
                    out[f"plane/{prec}/{nx}x{ny}/{scheme}/probe"] = s.get_probe(pid, 9)
                save(f"plane/{prec}/{nx}x{ny}/{scheme}", s)
                s.close()
    # fourth order: launches of many blocks and of few
    for dims in [(70, 90, 110), (33, 20, 17), (512, 30, 40), (5, 3, 2)]:
        s = Simulation(*dims, 1e-3, scheme="fadi", precision="f32", cfl=5.0)
        s.set_order(4)
        s.set_fields(random_fields(*dims, seed=1))
        s.step(2)
        save(f"order4/{dims}", s)
        s.close()
    # batches (the tuner's choice comes from the cache file that both builds share)
    for media in ("uniform", "both"):
        sims = [make(d, "fadi", "f32", "blocks" if media == "both" and q else "uniform")
                for q, d in enumerate([(33, 20, 17), (70, 97, 33), (9, 8, 250)])]
        b = Batch(sims)
        b.step(18)
        b.synchronize()
        out[f"batch/{media}/launches"] = np.array([b.launches_per_step()])
        b.close()
        for q, s in enumerate(sims):
            save(f"batch/{media}/{q}", s)
            s.close()
    # reverse mode
    n = (18, 17, 14)
    eps = np.random.default_rng(8).uniform(1.0, 6.0, n[::-1])
    for prec in ("f32", "f64"):
        run = ProbeEnergyProblem(*n, 1e-3, steps=7, probe_block=(1, 17, 0, 16, 1, 13), cfl=4.0, precision=prec,
                                 checkpoint_every=3, source=("ey", 9, 8, 7, current),
                                 fields=random_fields(*n, seed=9)).run(eps)
        out[f"adjoint/{prec}"] = run.backward(1.0, out=np.empty_like(eps))
        run.close()
    np.savez(out_path, **out)


if __name__ == "__main__":
    main(sys.argv[1])
