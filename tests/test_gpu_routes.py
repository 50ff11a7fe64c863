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


# few rows, many columns: the tile kernel's padding made the default step 1.3
# to 3.6 times slower than the strip kernel's (which set_launch selects)
@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
@pytest.mark.parametrize("precision,nx,ny", [
    (wblbe.FP64, 200000, 1), (wblbe.FP64, 200000, 4), (wblbe.FP64, 40000, 2),
    (wblbe.FP64, 200000, 17), (wblbe.FP64, 10000, 1), (wblbe.FP32_SHIFTED, 200000, 2),
    (wblbe.FP32_SHIFTED, 40000, 1), (wblbe.FP32_SHIFTED, 500000, 5),
    # and a few that stay on the tiles
    (wblbe.FP64, 10000, 5), (wblbe.FP64, 40000, 12), (wblbe.FP32_SHIFTED, 25000, 6)])
def test_flat_lattices_take_the_faster_kernel(scheme, precision, nx, ny):
    rng = np.random.default_rng(nx + ny)
    rho = 0.6 + 0.3 * rng.uniform(-1, 1, (ny, nx))
    out = []
    for strip in (False, True):
        s = wblbe.Solver(wblbe.Params(nx, ny, 0.9, 0.0128, 0.01, 1.0, 0.2, scheme=scheme,
                                      precision=precision))
        if strip:
            s.set_launch(*s.get_launch())
        s.init_rho(rho)
        s.step(6)
        code, done, st = s.run_until_equilibrium(0.0, 5, 3)
        out.append((s.get_populations(), s.moments()[0], st["mu_min"], st["mu_max"], st["umax"],
                    _us(lambda: s.step(32), 32)))
        s.close()
    (fa, ma, *sa, ta), (fb, mb, *sb, tb) = out
    assert np.array_equal(fa, fb) and sa == sb
    for k in ("rho", "ux", "uy", "mu"):
        assert np.array_equal(ma[k], mb[k]), k
    assert ta < 1.2 * tb, (ta, tb)


def _d3_moments_us(nx, ny, nz, precision, scheme):
    import torch
    s = wblbe.Solver3(wblbe.Params3(nx, ny, nz, 0.95, 0.01, 0.01, 1.0, 0.2, scheme=scheme,
                                    precision=precision))
    s.init_rho(0.6 + 0.1 * np.random.default_rng(nz).uniform(-1, 1, (nz, ny, nx)))
    out = torch.empty(5, nz, ny, nx, dtype=torch.float64, device="cuda")
    st = wblbe.CStats()
    us = _us(lambda: s._check(s.lib.wblbe3_moments(s.h, out[0].data_ptr(), out[1].data_ptr(),
                                                   out[4].data_ptr(), 1, ctypes.byref(st))),
             repeats=25)
    s.close()
    return us


@pytest.mark.parametrize("scheme", [wblbe.STANDARD, wblbe.WELL_BALANCED])
@pytest.mark.parametrize("n", [8, 16])
def test_moments_of_a_small_d3q19_lattice_are_not_serial(n, scheme):
    """A CTA that took eight planes of a small lattice one after another made
    its FP64 moments 1.4 to 1.5 times those of a lattice of one plane."""
    one = _d3_moments_us(n, n, 1, wblbe.FP64, scheme)
    cube = _d3_moments_us(n, n, n, wblbe.FP64, scheme)
    assert cube < 1.2 * one, (cube, one)


@pytest.mark.parametrize("precision", [wblbe.FP64, wblbe.FP32_SHIFTED])
@pytest.mark.parametrize("shape", [(5, 4, 3), (30, 20, 19), (40, 50, 33), (130, 60, 33)])
def test_d3q19_moments_whatever_the_planes_per_cta(shape, precision):
    """1, 1, 4 and 8 planes per CTA, the last CTA's short: every node is
    counted once.  The sums against the fields' in float64, to the rounding of
    nx ny nz additions of positive terms."""
    nx, ny, nz = shape
    s = wblbe.Solver3(wblbe.Params3(nx, ny, nz, 0.95, 0.01, 0.01, 1.0, 0.2, precision=precision))
    s.init_rho(0.6 + 0.1 * np.random.default_rng(nx).uniform(-1, 1, (nz, ny, nx)))
    s.step(3)
    m, st = s.moments()
    s.close()
    tol = nx * ny * nz * 2.0 ** -52
    u2 = (m["u"] ** 2).sum(axis=0)
    assert st["mass"] == pytest.approx(m["rho"].sum(), rel=tol)
    assert st["kinetic"] == pytest.approx(0.5 * (m["rho"] * u2).sum(), rel=tol)
    assert st["umax"] == pytest.approx(np.sqrt(u2.max()), rel=1e-15)
    assert st["mu_min"] == m["mu"].min() and st["mu_max"] == m["mu"].max()


def _d3_issue_us(nz):
    """Host time of issuing one FP32 step of a 1 x 1 x nz lattice."""
    import time

    import torch
    s = wblbe.Solver3(wblbe.Params3(1, 1, nz, 0.95, 0.01, 0.01, 1.0, 0.2,
                                    precision=wblbe.FP32_SHIFTED))
    s.init_rho(np.full((nz, 1, 1), 0.6))
    best = float("inf")
    for _ in range(7):
        torch.cuda.synchronize()
        t = time.perf_counter()
        s.step(20)                       # 40 launches: well within the launch queue
        best = min(best, (time.perf_counter() - t) / 20 * 1e6)
    torch.cuda.synchronize()
    s.close()
    return best


def test_host_work_of_a_d3q19_step_does_not_grow_with_the_lattice():
    """Choosing the run of planes again in every step cost some hundred us of
    host time for 65535 planes; two launches take about ten."""
    assert _d3_issue_us(65535) < _d3_issue_us(64) + 30.0
