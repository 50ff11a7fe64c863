"""D3Q19 lattices whose rows are whole 128-thread blocks (nodes keep the grid's
coordinates; other widths are numbered in one run), and FP32 marches of many
planes with a short last run (each slot of the four-plane rings is rewritten
several times, and the values a thread carries from plane to plane live
through the whole run)."""
import numpy as np
import pytest

from paper_2012_11075_gb300 import wblbe
from tests.gpu_helpers import need_gpu
from tests.test_gpu_d3q19 import _check, _run_both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()
    wblbe.load_library()


@pytest.mark.parametrize("shape", [(128, 1, 1), (128, 3, 2), (128, 6, 5), (256, 2, 3), (384, 3, 1)])
@pytest.mark.parametrize("scheme", [wblbe.WELL_BALANCED, wblbe.STANDARD])
def test_rows_of_whole_blocks_match_the_oracle(shape, scheme):
    nx, ny, nz = shape
    rng = np.random.default_rng(nx * 10000 + ny * 100 + nz)
    rho = 0.6 + 0.3 * rng.uniform(-1, 1, (nz, ny, nx))
    out = _run_both(nx, ny, nz, rho, scheme, 50, tau=0.85, kappa=0.0128, beta=0.01,
                    rho_l=1.0, rho_g=0.2)
    _check(*out, 0.01, 1.0, 0.2)


def _planes_per_run(nx, ny, nz):
    """Planes a CTA of the FP32 step marches: fewest iterations over all waves
    of four CTAs per SM, a run of n planes taking n + 4."""
    import torch
    resident = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-nx // 32) * -(-ny // 8)
    runs = [-(-nz // k) for k in range(1, nz + 1)]
    return min(runs, key=lambda n: -(-tiles * -(-nz // n) // resident) * (n + 4))


# (nx, ny, nz, least planes per run): whole blocks and others, long runs whose
# last is shorter, and short ones
@pytest.mark.parametrize("nx,ny,nz,least", [
    (130, 100, 101, 9), (256, 200, 31, 9), (250, 251, 29, 9), (128, 96, 75, 5), (128, 5, 3, 1),
    (256, 9, 4, 1)])
@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
def test_fp32_marches_follow_fp64(nx, ny, nz, least, scheme):
    """5 steps: populations are O(1), so the float storage and arithmetic stay
    within 40 ulps of 1 (2^-24 each), as at the tiles' edges."""
    run = _planes_per_run(nx, ny, nz)
    assert run >= least and (least == 1 or nz % run != 0)
    rng = np.random.default_rng(nx * 100 + ny * 10 + nz)
    rho = 0.6 + 0.1 * rng.uniform(-1, 1, (nz, ny, nx))
    f = []
    for precision in (wblbe.FP64, wblbe.FP32_SHIFTED):
        s = wblbe.Solver3(wblbe.Params3(nx, ny, nz, 0.9, 0.01, 0.005, 1.0, 0.2, scheme=scheme,
                                        precision=precision))
        s.init_rho(rho)
        s.step(5)
        f.append(s.get_populations())
        s.close()
    assert np.max(np.abs(f[0] - f[1])) < 40 * 2.0 ** -24
