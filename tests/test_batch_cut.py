"""The finer cut of a batch whose tiles would not occupy the device: rows per
tile are halved down to 8, so tiles with runs of 8 to 15 rows, ragged strips
and cases of one run appear; every case must still equal its lattice run
alone, bit for bit, and stop decisions must not change."""
import numpy as np
import pytest

from paper_2012_11075_gb300 import wblbe
from paper_2012_11075_gb300 import workloads as wl
from tests.gpu_helpers import gpu_params, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()
    wblbe.load_library()


@pytest.mark.parametrize("precision", [wblbe.FP64, wblbe.FP32_SHIFTED])
@pytest.mark.parametrize("tile_x,rows", [(32, 128), (128, 64), (64, 15), (64, 16)])
def test_finer_cut_keeps_every_case(precision, tile_x, rows):
    sizes = [(8, 8), (33, 9), (35, 17), (129, 31), (131, 64), (64, 250), (257, 40)]
    cases = [wl.droplet(radius=0.25 * min(nx, ny), tau=0.95, rho_g=0.2, nx=nx, ny=ny)
             for nx, ny in sizes]
    b = wblbe.Batch(precision=precision, max_cases=len(cases), arena_bytes=1 << 28,
                    tile_x=tile_x, rows_per_tile=rows, steps_per_launch=7)
    ids = [b.admit(gpu_params(pr, wblbe.WELL_BALANCED, precision), pr.rho, 0.0,
                   28 if k % 2 else 10 ** 9) for k, pr in enumerate(cases)]
    b.advance(6)                             # the odd cases stop after 28 steps
    for k, (pr, cid) in enumerate(zip(cases, ids)):
        steps = 28 if k % 2 else 42
        assert b.info(cid)["steps"] == steps
        s = wblbe.Solver(gpu_params(pr, wblbe.WELL_BALANCED, precision))
        s.init_rho(pr.rho)
        s.step(steps)
        assert np.array_equal(b.get_populations(cid), s.get_populations()), (pr.nx, pr.ny)
        s.close()
    b.close()
