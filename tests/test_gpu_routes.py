"""Calls whose route is chosen by size take one that is not slower than the
other routes they have: each comparison is of two calls of the library on the
same device, with bounds far from the run-to-run noise (a few per cent) and
from the difference a wrong choice makes (stated in each test)."""
import ctypes

import numpy as np
import pytest

from paper_2012_11075_gb300 import wblbe
from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()
    wblbe.load_library()


def _us(fn, calls=1, repeats=7):
    """Least device time of one of `calls` calls in fn(), after a first run."""
    import torch
    fn()
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / calls)
    return best


def test_batch_is_not_cut_finer_than_it_needs():
    """Four cases whose 256-column, 16-row tiles are 1.4 per resident CTA:
    halved to 8 rows they took 1.24 times the time.  15 rows per tile are
    never halved."""
    rng = np.random.default_rng(4)
    sizes = [(617, 512), (1043, 395), (330, 871), (702, 640)]
    prm = [wblbe.Params(nx, ny, 0.95, 0.01, 0.01, 1.0, 0.2, precision=wblbe.FP32_SHIFTED)
           for nx, ny in sizes]
    lib = wblbe.load_library()
    room = sum(int(lib.wblbe_batch_case_bytes(ctypes.byref(p.c()))) for p in prm) + (1 << 20)
    t = {}
    for rows in (15, 16):
        b = wblbe.Batch(precision=wblbe.FP32_SHIFTED, max_cases=4, max_tiles=4096,
                        max_case_nodes=max(p.nx * p.ny for p in prm), arena_bytes=room,
                        tile_x=256, rows_per_tile=rows, steps_per_launch=32)
        for p in prm:
            b.admit(p, 0.6 + 0.1 * rng.uniform(-1, 1, (p.ny, p.nx)), 0.0, 10 ** 12)
        t[rows] = _us(lambda: b.advance(3), 3 * 32)
        b.close()
    assert t[16] < 1.12 * t[15], t
