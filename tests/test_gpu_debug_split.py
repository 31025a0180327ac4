"""The index-checking debug build on the kernels that are launched by default in FP64 (the two passes and what prepares them,
after initialisation and after a checkpoint) and on the tile shapes of small grids and of wall sides: no failed check, and the
parity bound against the oracle (FP64 1e-10, FP32 1e-4).  Reads of other cells in the two-pass kernels go through plane_at(),
which carries the check."""
import json
import os
import re
import subprocess
import sys

import pytest

from test_gpu_debug_build import builds  # noqa: F401

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, os, sys
sys.path.insert(0, os.environ["HLBM_ROOT"]); sys.path.insert(0, os.path.join(os.environ["HLBM_ROOT"], "tests"))
import numpy as np
import torch
torch.cuda.set_device(0)
from paper_2002_03644_gb300 import hlbm, inputs
from test_gpu_parity import run_pair, compare, TOL
out = {"library": hlbm.library_path(), "checks": []}
bs = np.array([[1.02, 0.08, 0.01, 0.21], [0.98, 0.05, -0.02, 0.19], [1.01, 0.06, 0.03, 0.2], [0.99, 0.07, 0.0, 0.205]])
mixed, plates = (1, 2, 2, 1), (0, 0, 3, 3)
runs = [(101, 67, 0, (0, 0, 0, 0), 0.5, 0), (101, 67, 0, mixed, 0.5, 0), (101, 67, 0, mixed, 0.0, 1), (101, 67, 0, (2, 1, 0, 0), 0.0, 0),
        (2, 100, 0, (1, 1, 1, 1), 0.0, 0), (1, 9, 0, (0, 0, 0, 0), 0.0, 1), (800, 760, 0, mixed, 0.0, 0),
        (2, 100, 0, plates, 0.5, 0), (101, 110, 0, plates, 0.5, 0), (300, 200, 0, plates, 0.0, 0), (101, 67, 1, plates, 0.5, 0),
        (101, 67, 1, mixed, 0.0, 1), (101, 67, 2, mixed, 0.5, 0), (101, 67, 3, (0, 0, 0, 0), 0.0, 0)]
for nx, ny, prec, bc, sigma, phi in runs:
    case = inputs.random_smooth(nx, ny, seed=3, amp=0.04, u0=(0.06, 0.01), theta0=0.2, mu=3e-3, sigma=sigma, bc=bc, bc_state=bs)
    case.phi_mode = phi
    s, _, got, ref = run_pair(hlbm, case, prec, 5)
    site = hlbm.hlbm_debug_check()
    if prec < 2 and 3 not in bc:
        compare(got, ref, case.gamma, TOL[prec])
    out["checks"].append([str((nx, ny, prec, bc, sigma, phi)), list(site)])
    if prec == 0:
        s.set_state(s.state())
        s.step(2)
        s.synchronize()
        out["checks"].append(["from a checkpoint", list(hlbm.hlbm_debug_check())])
    s.close()
print(json.dumps(out))
"""


def test_reads_of_other_cells_are_checked():
    src = open(os.path.join(ROOT, "paper_2002_03644_gb300", "csrc", "hlbm_split.cuh")).read()
    for name in ("plane_at", "split_level_kernel", "split_collide_kernel", "split_prepare_kernel"):
        body = src[re.search(r"\b%s\(const double|\b%s\(double" % (name, name), src).start():]
        assert "HLBM_CELL_OK" in body[:body.index("\n}\n")], name
    # one cell's plane values are read at its own offset o, a neighbour's through plane_at
    for index in re.findall(r"\bp[uvts]\[(\w+)\]|\bp[sd]\[(\w+)\]|sp\.\w+\[([\w.]+)\]", src):
        assert set(index) <= {"o", ""}, index


@pytest.mark.gpu
def test_debug_build_runs_the_default_kernels_clean(builds):  # noqa: F811
    build, _ = builds
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = build.build_library(debug=True)
    env = dict(os.environ, HLBM_LIBRARY="debug", HLBM_ROOT=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["library"] == lib
    for name, (site, a, b) in out["checks"]:
        assert site == 0, (name, site, a, b)
