"""Shapes that a user's cache file names for a grid are the ones it runs,
also for the FP32 grids that take a fixed shape without one.  The file is read
once per process, so each case is a process of its own; the shape is seen by
its roundings (the segment length decides them)."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

pytestmark = pytest.mark.gpu

N = (40, 100, 90)   # (below a million cells; both lengths are among the fixed shapes)


def child(case, out):
    from gpu_helpers import random_fields
    from paper_2011_14043_gb300 import Simulation
    eps = np.random.default_rng(1).uniform(1.0, 6.0, N[::-1])
    u0 = random_fields(*N, 2)
    if case["what"] == "grid":
        s = Simulation(*N, 1e-3, scheme="fadi", precision="f32", cfl=4.0, tune=(case["tune"], 0))
        s.set_material(eps)
        s.set_fields(u0)
        s.add_probe("ez", 3, 3, 3)
        s.step(3)
        np.savez(out, **{c: s.get_state(c) for c in u0})
    else:
        from paper_2011_14043_gb300.adjoint import ProbeEnergyProblem
        run = ProbeEnergyProblem(*N, 1e-3, steps=4, probe_block=(2, 9, 2, 9, 2, 9), cfl=4.0, checkpoint_every=2,
                                 precision="f32", fields=u0).run(eps)
        np.savez(out, g=run.backward(1.0, out=np.empty_like(eps)))


def run(tmp_path, case, entry=None):
    import torch
    env = {k: v for k, v in os.environ.items() if k != "FDTD_TUNE_CACHE"}
    path = tmp_path / "tune.txt"
    if entry is not None:
        name = torch.cuda.get_device_name().replace(" ", "_")
        key = (f"grid|{name}|p1|s0|" if case["what"] == "grid" else f"adjoint|{name}|p1|") + "x".join(map(str, N))
        path.write_text(f"{key} {entry} 0 0\n")
        env["FDTD_TUNE_CACHE"] = str(path)
    out = tmp_path / "out.npz"
    res = subprocess.run([sys.executable, os.path.abspath(__file__), json.dumps(case), str(out)], env=env,
                         cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    with np.load(out) as z:
        return {k: z[k] for k in z.files}


def equal(a, b):
    return all(np.array_equal(a[k], b[k]) for k in a)


def test_forward_shapes(tmp_path):
    case = {"what": "grid", "tune": 0}
    plain = run(tmp_path, case)
    cached = run(tmp_path, case, "16 32 16 32")
    assert equal(cached, run(tmp_path, dict(case, tune=32)))       # 32 nodes per thread
    assert not equal(cached, plain)
    assert equal(plain, run(tmp_path, case, "16 16 16 16"))        # the lengths of the fixed shapes
    assert equal(plain, run(tmp_path, case, "16 7 16 16"))         # a shape that is not built: as without


def test_reverse_shapes(tmp_path):
    case = {"what": "adjoint"}
    plain = run(tmp_path, case)
    cached = run(tmp_path, case, "16 32 16 32")
    assert not equal(cached, plain)
    assert np.linalg.norm(cached["g"] - plain["g"]) <= 1e-3 * np.linalg.norm(plain["g"])
    assert equal(plain, run(tmp_path, case, "16 8 16 8"))


if __name__ == "__main__":
    child(json.loads(sys.argv[1]), sys.argv[2])
