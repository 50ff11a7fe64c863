"""Bounds-checked run of the tile, split and D3Q19 kernels and of the other
routes that need no launch shape (bounds_tile_workload.py), as test_gpu_bounds
does for the strip and batched kernels."""
import json
import os
import subprocess
import sys
from pathlib import Path

import pytest

from paper_2012_11075_gb300 import _build
from tests.gpu_helpers import need_gpu

ROOT = Path(__file__).resolve().parents[1]


@pytest.mark.gpu
def test_tile_and_d3q19_kernels_stay_in_bounds():
    need_gpu()
    lib = _build.build(debug_bounds=True)
    env = dict(os.environ, WBLBE_LIBRARY=str(lib),
               PYTHONPATH=str(ROOT) + os.pathsep + os.environ.get("PYTHONPATH", ""))
    out = subprocess.run([sys.executable, "-m", "tests.bounds_tile_workload"], cwd=ROOT, env=env,
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stderr[-2000:]
    res = json.loads(out.stdout.strip().splitlines()[-1])
    assert res["runs"] == 2 * (2 * (17 + 12 + 1) + 1)
    assert res["errors"] == 0, res


def test_every_d3q19_kernel_checks_its_accesses():
    """The D3Q19 file has kernels of its own: each has a check, directly or in
    the function that reads for it, and the count is part of the total."""
    csrc = ROOT / "paper_2012_11075_gb300" / "csrc"
    text = (csrc / "d3q19.cu").read_text()
    for kernel in text.split("__global__")[1:]:
        assert any(w in kernel for w in ("WB_IN(", "elem3_at(", "Node3<")), kernel[:120]
    assert "d3_bounds_errors(reset" in (csrc / "wblbe.cu").read_text()
