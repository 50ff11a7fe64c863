"""The tile kernel of small and medium lattices against the strip kernel, at
the sizes where it can go wrong: lattices smaller than a tile's frame (its
columns and rows wrap onto themselves), one node more or less than a tile, a
last tile with one row, and each tile shape's range.  Both kernels evaluate a
node with the same operations, so populations, fields and the order-free
statistics are equal bit for bit; the sums are folded in another order."""
import numpy as np
import pytest

from paper_2012_11075_gb300 import wblbe
from tests.gpu_helpers import need_gpu

pytestmark = pytest.mark.gpu

# FP64 shapes: 8 x 4 up to 380 tiles, 16 x 8 up to 152, then 16 x 16;
# FP32: 16 x 8 up to 456 tiles, then 32 x 16
SIZES = [(1, 1), (2, 5), (5, 2), (7, 3), (8, 4), (9, 5), (15, 9), (16, 8), (17, 17), (33, 16),
         (31, 49), (4, 301), (301, 4), (104, 121), (161, 145), (257, 241)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()
    wblbe.load_library()


def _solver(nx, ny, scheme, precision, strip):
    s = wblbe.Solver(wblbe.Params(nx, ny, 0.9, 0.0128, 0.01, 1.0, 0.2, scheme=scheme,
                                  precision=precision))
    if strip:
        s.set_launch(*s.get_launch())
    return s


@pytest.mark.parametrize("precision", [wblbe.FP64, wblbe.FP32_SHIFTED])
@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
def test_tile_kernel_equals_strip_kernel_bitwise(scheme, precision):
    for nx, ny in SIZES:
        rng = np.random.default_rng(nx * 1000 + ny)
        rho = 0.6 + 0.3 * rng.uniform(-1, 1, (ny, nx))
        runs = []
        for strip in (False, True):
            s = _solver(nx, ny, scheme, precision, strip)
            s.init_rho(rho)
            s.step(70)                       # graph replays and direct steps
            f = s.get_populations()
            code, done, st = s.run_until_equilibrium(0.0, 13, 5)   # steps with statistics
            runs.append((f, s.get_populations(), s.moments()[0], code, done, st))
            s.close()
        (fa, ga, ma, ca, da, sa), (fb, gb, mb, cb, db, sb) = runs
        assert np.array_equal(fa, fb) and np.array_equal(ga, gb), (nx, ny)
        for k in ("rho", "ux", "uy", "mu"):
            assert np.array_equal(ma[k], mb[k]), (nx, ny, k)
        assert (ca, da) == (cb, db)
        for k in ("umax", "mu_min", "mu_max", "nonfinite", "step"):
            assert sa[k] == sb[k], (nx, ny, k)
        # up to nx ny positive terms summed in another order, in float64
        tol = nx * ny * 2.0 ** -52
        assert sa["mass"] == pytest.approx(sb["mass"], rel=tol)
        assert sa["kinetic"] == pytest.approx(sb["kinetic"], rel=tol, abs=1e-300)


@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
@pytest.mark.parametrize("precision,nx,ny", [(wblbe.FP64, 1201, 1001),
                                             (wblbe.FP32_SHIFTED, 901, 889)])
def test_steps_on_tiles_with_statistics_on_strips(scheme, precision, nx, ny):
    # just above the node count at which passes with statistics leave the tiles
    rng = np.random.default_rng(nx)
    rho = 0.6 + 0.3 * rng.uniform(-1, 1, (ny, nx))
    runs = []
    for strip in (False, True):
        s = _solver(nx, ny, scheme, precision, strip)
        s.init_rho(rho)
        code, done, st = s.run_until_equilibrium(0.0, 7, 3)
        runs.append((s.get_populations(), s.moments()[0], code, done, st))
        s.close()
    (fa, ma, ca, da, sa), (fb, mb, cb, db, sb) = runs
    assert np.array_equal(fa, fb) and (ca, da, sa) == (cb, db, sb)
    for k in ("rho", "ux", "uy", "mu"):
        assert np.array_equal(ma[k], mb[k]), k
