"""Lattices the D3Q19 kernels cannot index are refused on the host: their
element offsets within a population plane are 32 bits wide."""
import ctypes

import pytest

from paper_2012_11075_gb300 import wblbe


def _call(nx, ny, nz, precision):
    lib = wblbe.load_library()
    p = wblbe.Params3(nx, ny, nz, 0.9, 0.01, 0.01, 1.0, 0.1, precision=precision).c()
    nbytes = lib.wblbe3_workspace_bytes(ctypes.byref(p))
    h = ctypes.c_void_p()
    # 255 bytes never suffice: a lattice that is accepted answers ENOMEM, and
    # no memory is touched
    st = lib.wblbe3_create(ctypes.byref(p), ctypes.c_void_p(256), 255, None, ctypes.byref(h))
    assert not h
    return nbytes, st


@pytest.mark.parametrize("precision", [wblbe.FP64, wblbe.FP32_SHIFTED])
@pytest.mark.parametrize("nx,ny,nz", [
    (1, 65535, 4097),            # 16 x 65535 x 4097 elements, just above 2^32
    (65536, 65536 - 1, 2), (2048, 2048, 1024), (1 << 16, 1 << 15, 2), (1 << 30, 2, 2)])
def test_planes_of_2_to_32_elements_are_refused(nx, ny, nz, precision):
    assert _call(nx, ny, nz, precision) == (0, wblbe.EINVAL)


@pytest.mark.parametrize("precision", [wblbe.FP64, wblbe.FP32_SHIFTED])
@pytest.mark.parametrize("nx,ny,nz", [(65536, 65535, 1), (2048, 2048, 1023), (1, 65535, 4095),
                                      (256, 256, 256)])
def test_planes_below_are_accepted(nx, ny, nz, precision):
    nbytes, st = _call(nx, ny, nz, precision)
    plane = (nx + 15) // 16 * 16 * ny * nz
    assert nbytes >= 2 * 19 * plane * (8 if precision == wblbe.FP64 else 4)
    assert st == wblbe.ENOMEM
