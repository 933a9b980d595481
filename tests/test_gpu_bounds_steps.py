"""The bounds-checked build on the cases of bounds_cases_steps.py: no
violation, and the arrays of the default build bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def run_cases(lib_path, out_path, tune_cache):
    env = dict(os.environ, FDTD_LIBRARY=lib_path, FDTD_TUNE_CACHE=str(tune_cache))
    res = subprocess.run([sys.executable, os.path.join(HERE, "bounds_cases_steps.py"), str(out_path)], env=env,
                         cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=1200)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    return np.load(out_path)


def batch_entries():
    """Both batches of the cases by one fused launch per procedure and kind."""
    import torch
    name = torch.cuda.get_device_name().replace(" ", "_")
    lines = []
    for kinds in ("uuu", "unn"):
        key = f"batch|{name}|p1|s0" + "".join(f"|{d}{k}" for d, k in zip(("33x20x17", "70x97x33", "9x8x250"), kinds))
        lines += [f"{key} 16 8 16 8 8 1", f"{key}|mode|16,8,16,8,8,1|fused 0 9 9 8 8 1"]
    return "\n".join(lines) + "\n"


def test_bounds_checked_build_runs_the_step_kernels_clean(tmp_path):
    from paper_2011_14043_gb300.build import LIB_PATH, build
    build()
    checked = build(bounds=True)
    cache = tmp_path / "tune_cache.txt"
    cache.write_text(batch_entries())
    ref = run_cases(LIB_PATH, tmp_path / "default.npz", cache)
    chk = run_cases(checked, tmp_path / "checked.npz", cache)
    assert sorted(ref.files) == sorted(chk.files)
    assert len(ref.files) > 400
    assert ref["batch/uniform/launches"][0] == 2 and ref["batch/both/launches"][0] == 4
    for k in ref.files:
        assert np.array_equal(ref[k], chk[k]), k
