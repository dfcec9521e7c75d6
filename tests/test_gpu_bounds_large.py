"""The index-checked build on a lattice whose hopping kernels are those of larger
lattices: one thread a site in FP32 and BF16, two in df64 and FP64, with partial
last warps and blocks, natural output, and FP32 fields at the ends of a df64
smoother.  test_gpu_bounds runs lattices that the twelve-thread kernels take.
"""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_large_lattice_index_checks_and_canaries_clean():
    from paper_2407_08092_gb300 import build
    lib = build.build(checked=True)
    r = subprocess.run([sys.executable, os.path.join(HERE, "bounds_large_child.py")],
                       env=dict(os.environ, LQ_LIBRARY=lib), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    rep = json.loads(r.stdout.strip().splitlines()[-1])
    assert rep["checked"] == 1, rep
    assert rep["violations"] == 0 and rep["status"] == 0, rep
    assert rep["bad_canaries"] == [], rep
    assert rep["failed"] == [], rep
