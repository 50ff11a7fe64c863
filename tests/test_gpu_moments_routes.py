"""The moments pass on its two kernels.  A single lattice's moments take the
tile kernel up to 1.2 (FP64) and 0.8 (FP32) million nodes whatever launch
shape was set, so they are compared here with the row slabs' pass, which is
the strip kernel at every size (one slab: the same lattice): the fields and
extrema are equal bit for bit, the sums folded in another order.  Above those
counts both are strips, and an independent kernel gives the values."""
import numpy as np
import pytest

from paper_2012_11075_gb300 import wblbe
from paper_2012_11075_gb300 import workloads as wl
from tests.gpu_helpers import gpu_params, need_gpu
from tests.test_gpu_tile import SIZES
from tests.test_zz_no_alloc import _compare, _noalloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()
    wblbe.load_library()


@pytest.mark.parametrize("precision,extra", [
    (wblbe.FP64, [(1095, 1095), (1201, 1001)]),          # below and above the count
    (wblbe.FP32_SHIFTED, [(893, 895), (901, 889)])])
@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
def test_moments_on_tiles_equal_moments_on_strips(scheme, precision, extra):
    for nx, ny in [s for s in SIZES if s[1] >= 3] + extra:     # a slab has at least 3 rows
        rng = np.random.default_rng(nx * 1000 + ny)
        rho = 0.6 + 0.3 * rng.uniform(-1, 1, (ny, nx))
        params = wblbe.Params(nx, ny, 0.9, 0.0128, 0.01, 1.0, 0.2, scheme=scheme,
                              precision=precision)
        out = []
        for make in (lambda: wblbe.Solver(params), lambda: wblbe.Slabs(params, 1)):
            s = make()
            s.init_rho(rho)
            s.step(9)
            out.append(s.moments())
            s.close()
        (ma, sa), (mb, sb) = out
        for k in ("rho", "ux", "uy", "mu"):
            assert np.array_equal(ma[k], mb[k]), (nx, ny, k)
        for k in ("umax", "mu_min", "mu_max", "nonfinite", "step"):
            assert sa[k] == sb[k], (nx, ny, k)
        tol = nx * ny * 2.0 ** -52          # nx ny positive terms in another order
        assert sa["mass"] == pytest.approx(sb["mass"], rel=tol)
        assert sa["kinetic"] == pytest.approx(sb["kinetic"], rel=tol, abs=1e-300)


@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
@pytest.mark.parametrize("nx,ny", [(1095, 1095), (1201, 1001)])
def test_moments_on_either_kernel_match_an_independent_one(scheme, nx, ny):
    torch = need_gpu()
    lib = wblbe.load_library()
    rng = np.random.default_rng(nx)
    pr = wl.Problem(nx, ny, 0.85, 0.0128, 0.01, 1.0, 0.2,
                    0.6 + 0.3 * rng.uniform(-1, 1, (ny, nx)), name="random")
    params = gpu_params(pr, scheme)
    s = wblbe.Solver(params)
    s.init_rho(pr.rho)
    s.step(20)
    ref, ref_st = s.moments()
    got, st = _noalloc(lib, params, torch.from_numpy(s.get_populations()).cuda(), torch)
    s.close()
    _compare(ref, ref_st, got, st, pr)
