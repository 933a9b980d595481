"""Batches that run one fused launch per procedure, with the tuner's choice
given by a cache file (read once per process, so each case is a process of
its own) instead of left to a timing."""
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

GRIDS = [(20, 30, 9), (70, 97, 33), (130, 12, 70), (16, 129, 5), (9, 8, 250)]
SHAPES = "16,8,16,8,8,1"   # y lanes, y L, z lanes, z L, x warps per block, x packing


def media(case, q):
    nx, ny, nz = GRIDS[q]
    if case["media"] == "uniform" or (case["media"] == "both" and q % 2 == 0):
        return None
    return np.random.default_rng(q).uniform(1.0, 6.0, (nz, ny, nx))


def batch_key(case, scheme_id):
    import torch
    name = torch.cuda.get_device_name().replace(" ", "_")
    return f"batch|{name}|p1|s{scheme_id}" + "".join(
        "|%dx%dx%d%s" % (*GRIDS[q], "u" if media(case, q) is None else "n") for q in range(len(GRIDS)))


def run_child(case, tmp_path, lines):
    path = tmp_path / "tune.txt"
    path.write_text("".join(line + "\n" for line in lines))
    env = dict(os.environ, FDTD_TUNE_CACHE=str(path))
    res = subprocess.run([sys.executable, os.path.abspath(__file__), json.dumps(case)], env=env,
                         cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    return json.loads(res.stdout.splitlines()[-1]), path.read_text().splitlines()


def sim(case, q, tune=(0, 0)):
    from gpu_helpers import random_fields
    from paper_2011_14043_gb300 import Simulation
    s = Simulation(*GRIDS[q], 1e-3, scheme=case["scheme"], precision="f32", cfl=3.0 + q, tune=tune)
    if media(case, q) is not None:
        s.set_material(media(case, q))
    s.set_fields(random_fields(*GRIDS[q], 20 + q))
    return s


def child_launches(case):
    """Launches per step of a batch of `tune` handles."""
    from paper_2011_14043_gb300 import Batch
    sims = [sim(case, q, tuple(case["tune"])) for q in range(len(GRIDS))]
    b = Batch(sims)
    b.step(2)
    b.synchronize()
    return {"launches": b.launches_per_step()}


def entry(key, fused, mode):
    return [f"{key} {SHAPES.replace(',', ' ')}", f"{key}|mode|{SHAPES}{mode} 0 9 9 8 8 {fused}"]


SCHEMES = {"fadi": 0, "fss": 2}


@pytest.mark.parametrize("scheme", ["fadi", "fss"])
def test_choices_with_and_without_the_fused_launches_are_kept_apart(scheme, tmp_path):
    procedures = 3 if scheme == "fss" else 2
    case = {"what": "launches", "scheme": scheme, "media": "uniform", "tune": [0, 0]}
    key = batch_key(case, SCHEMES[scheme])
    # an entry made with them among the candidates
    got, lines = run_child(case, tmp_path, entry(key, 1, "|fused"))
    assert got["launches"] == procedures and len(lines) == 2
    got, lines = run_child(case, tmp_path, entry(key, 0, "|fused"))
    assert got["launches"] > procedures and len(lines) == 2
    # an entry made without them answers nothing here: timed again
    got, lines = run_child(case, tmp_path, entry(key, 0, ""))
    assert len(lines) == 3 and lines[2].split()[0] == f"{key}|mode|{SHAPES}|fused"
    # and an entry made with them does not reach handles that the fused kernel refuses
    case["tune"] = [8, 0]
    got, lines = run_child(case, tmp_path, entry(key, 1, "|fused"))
    assert got["launches"] > procedures
    assert len(lines) == 3 and lines[2].split()[0] == f"{key}|mode|{SHAPES}"


def child_own_steps(case):
    """From one state, `steps` steps by the batch and by each handle itself
    (in between and again): the grids whose bits differ."""
    from paper_2011_14043_gb300 import Batch
    sims = [sim(case, q) for q in range(len(GRIDS))]
    b = Batch(sims)
    b.step(1)
    differ = []
    for n in (1, 18):
        before = [{c: s.get_state(c) for c in ("ex", "ey", "ez", "hx", "hy", "hz")} for s in sims]
        b.step(n)
        after = [{c: s.get_state(c) for c in before[0]} for s in sims]
        for q, s in enumerate(sims):
            for c in before[q]:
                s.set_state(c, before[q][c])
            s.step(n)
            if not all(np.array_equal(s.get_state(c), after[q][c]) for c in before[q]):
                differ.append(q)
    out = {"launches": b.launches_per_step(), "differ": differ}
    b.close()
    return out


@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("media_kind", ["uniform", "blocks", "both"])
@pytest.mark.parametrize("scheme", ["fadi", "fss"])
def test_a_batch_runs_the_arithmetic_of_its_handles(scheme, media_kind, fused, tmp_path):
    """Bit for bit (per-node media outside the fused launches: only where the
    tuned segment lengths agree, so those grids are left out)."""
    case = {"what": "own_steps", "scheme": scheme, "media": media_kind}
    got, _ = run_child(case, tmp_path, entry(batch_key(case, SCHEMES[scheme]), fused, "|fused"))
    if fused:
        assert got["launches"] == (3 if scheme == "fss" else 2) * (2 if media_kind == "both" else 1)
    assert [q for q in got["differ"] if fused or media(case, q) is None] == []


def child_values(case):
    """Errors of the batch against the FP64 oracle, and the grids whose bits
    differ from those of the same grid stepped alone."""
    from gpu_helpers import energy_norm_rel, oracle_problem, random_fields
    from oracle import schemes as S
    from paper_2011_14043_gb300 import Batch
    steps = 18
    sims = [sim(case, q) for q in range(len(GRIDS))]
    b = Batch(sims)
    b.step(1)
    b.step(steps - 1)
    out = {"launches": b.launches_per_step(), "errors": [], "differ": []}
    states = [{c: s.get_state(c) for c in ("ex", "ey", "ez", "hx", "hy", "hz")} for s in sims]
    for q, s in enumerate(sims):
        u0 = {c: v.astype(np.float32).astype(np.float64) for c, v in random_fields(*GRIDS[q], 20 + q).items()}
        P = oracle_problem(*GRIDS[q], 1e-3, 1e-3, 1e-3, s.dt, eps=media(case, q))
        out["errors"].append(energy_norm_rel(s.get_fields(), S.run_fundamental(P, case["scheme"], u0, steps)[0]))
        alone = sim(case, q)
        alone.step(steps)
        if not all(np.array_equal(alone.get_state(c), states[q][c]) for c in states[q]):
            out["differ"].append(q)
        alone.close()
    b.close()
    return out


@pytest.mark.parametrize("media_kind", ["uniform", "blocks", "both"])
@pytest.mark.parametrize("scheme", ["fadi", "fss"])
def test_fused_batch_against_the_oracle_and_grids_stepped_alone(scheme, media_kind, tmp_path):
    case = {"what": "values", "scheme": scheme, "media": media_kind}
    got, _ = run_child(case, tmp_path, entry(batch_key(case, SCHEMES[scheme]), 1, "|fused"))
    assert got["launches"] == (3 if scheme == "fss" else 2) * (2 if media_kind == "both" else 1)
    assert max(got["errors"]) <= 1e-4     # the library's stated bound for a few steps
    assert got["differ"] == []


if __name__ == "__main__":
    CASE = json.loads(sys.argv[1])
    print(json.dumps(globals()["child_" + CASE["what"]](CASE)))
