"""Work lists in the bounds-check build: every position a kernel appends at or reads from and every entry it reads back
is checked like the stencils' indices. On the CPU the sources are searched for subscripts of the lists that are not; on
the GPU the checked library steps grids that take lists (and grids that do not), the persistent step and batches."""
import json
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2208_04488_gb300", "csrc")
LISTS = r"(?<![\w.])(?:list|cells|lists\.list\[d\]|A\.listed|A\.deferred)\[(?!d\]\[)([^;]*)"


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cuh")))
def test_every_subscript_of_a_list_is_checked(name):
    for line in open(os.path.join(CSRC, name)):
        if line.lstrip().startswith("//") or "lists.list[d] " in line or "* list[" in line:
            continue
        for index in re.findall(LISTS, line):
            assert "HRM_IDX" in index, line


CHILD = r"""
import json, sys
import numpy as np
sys.path.insert(0, ROOT)
from paper_2208_04488_gb300 import build, hrm, problems as P
build.build()
out = {}
# FP64 takes lists above 16384 cells, the precision form above 65536 (one stage at a time: above 262144)
cases = [(P.shock_tube_1d_baseline(400), 0), (P.shock_tube_1d_baseline(17001), 0), (P.shock_bubble_2d(180, 93), 0),
         (P.dirichlet_box([131, 127]), 0), (P.dirichlet_box([27, 26, 25]), 0), (P.interface_3d(26), 0),
         (P.shock_tube_1d_baseline(66001), 1), (P.shock_bubble_2d(371, 179), 1), (P.dirichlet_box([263, 251]), 1),
         (P.interface_3d(41), 1), (P.shock_bubble_2d(731, 363), 1), (P.shock_bubble_2d(97, 45), 1)]
for pr, prec in cases:
    s = hrm.Solver.from_problem(pr, params=hrm.params_default(cfl=0.4, check=0, precision=prec))
    s.step(0.0, 4)
    s.begin_step(s.step_tau())
    for k in range(s.stages()):
        s.stage(k)
    for d in range(pr.D):
        s.set_gate(d, (np.arange(s.face_count(d)) % 3 == 0).astype(np.uint8))
    s.set_params(hrm.params_default(cfl=0.4, check=0, precision=prec, learned=hrm.LEARNED_FIXED))
    s.step(0.0, 2)
    s.set_params(hrm.params_default(cfl=0.4, check=0, precision=prec, screen=0))
    s.step(0.0, 2)
    if prec and pr.D == 2 and not pr.boundary:
        s.set_params(hrm.params_default(cfl=0.4, check=0, precision=prec))
        s.set_step_path(1)
        s.step(0.0, 3)
        assert s.step_launches() == 3
        det = hrm.Detector(capacity=1 << 14, seed=1)
        s.set_step_path(0)
        s.set_detector(det)
        s.set_params(hrm.params_default(cfl=0.4, check=0, precision=prec, learned=hrm.LEARNED_GATE))
        s.step(0.0, 2)
    out[f"{pr.name}_{'x'.join(map(str, pr.n))}_{prec}"] = s.bounds_violations()
    s.close()
for prec in (0, 1):
    b = hrm.BatchSolver(P.batch_instances(count=5, scale=24, seed=7) + [P.advection_2d_smooth(40)],
                        params=hrm.params_default(cfl=0.4, check=0, precision=prec))
    b.step(5)
    b.tune(1)
    b.step(2)
    out[f"batch_{prec}"] = b.bounds_violations()
print(json.dumps(out))
"""


@pytest.mark.gpu
def test_lists_meet_no_out_of_range_index():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, HRM_BOUNDS_CHECK="1")
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CHILD], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    counts = json.loads(r.stdout.strip().splitlines()[-1])
    assert counts and all(v == 0 for v in counts.values()), counts
