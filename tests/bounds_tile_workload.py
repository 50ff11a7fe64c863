"""The kernels that bounds_workload.py does not reach, through the library that
WBLBE_LIBRARY names (the bounds-checked build, in test_gpu_bounds_tile.py):
the tile and split kernels of single lattices in every mode and tile shape
(no launch shape is set), the strip kernel of larger and of flat lattices, a
refined batch cut, and the D3Q19 kernels.  Prints the number of out-of-bounds
accesses as one JSON line."""
import json

import numpy as np

from paper_2012_11075_gb300 import wblbe

# FP64: split up to 304 tiles of 8 x 4, then 8 x 4 up to 380, 16 x 8 up to 152,
# 16 x 16; FP32: 16 x 8 up to 456 tiles, 32 x 16; flat ones on strips
SHAPES = [(1, 1), (2, 5), (5, 2), (7, 3), (9, 5), (17, 17), (31, 49), (4, 301), (301, 4),
          (99, 101), (104, 121), (121, 125), (161, 145), (257, 241), (33, 700), (20001, 3),
          (40000, 1)]
# just above the node counts at which statistics leave the tiles
STATS = [(wblbe.FP64, 1201, 1001), (wblbe.FP32_SHIFTED, 901, 889)]
SHAPES3 = [(1, 1, 1), (3, 4, 5), (1, 1, 17), (7, 6, 5), (33, 9, 8), (40, 7, 31), (130, 3, 2),
           (128, 4, 6), (256, 3, 3), (128, 1, 1), (45, 30, 61), (130, 60, 33)]


def single(nx, ny, scheme, precision):
    rng = np.random.default_rng(nx * 1000 + ny)
    s = wblbe.Solver(wblbe.Params(nx, ny, 0.85, 0.0128, 0.01, 1.0, 0.2, scheme=scheme,
                                  precision=precision))
    s.init_rho(0.6 + 0.3 * rng.uniform(-1, 1, (ny, nx)))
    s.step(35)                               # a captured chunk and direct steps
    s.run_until_equilibrium(0.0, 3, 2)       # steps with statistics
    s.moments()
    s.close()


def cube(nx, ny, nz, scheme, precision):
    rng = np.random.default_rng(nx * 1000 + ny * 10 + nz)
    s = wblbe.Solver3(wblbe.Params3(nx, ny, nz, 0.85, 0.0128, 0.01, 1.0, 0.2, scheme=scheme,
                                    precision=precision))
    s.init_rho(0.6 + 0.3 * rng.uniform(-1, 1, (nz, ny, nx)))
    s.step(3)
    s.moments()
    s.get_populations()
    s.close()


def main():
    wblbe.debug_bounds_errors(reset=True)
    runs = 0
    for precision in (wblbe.FP64, wblbe.FP32_SHIFTED):
        for scheme in (wblbe.STANDARD, wblbe.WELL_BALANCED):
            for nx, ny in SHAPES:
                single(nx, ny, scheme, precision)
                runs += 1
            for shape in SHAPES3:
                cube(*shape, scheme, precision)
                runs += 1
            for p, nx, ny in STATS:
                if p == precision:
                    single(nx, ny, scheme, precision)
                    runs += 1
        b = wblbe.Batch(precision=precision, max_cases=4, arena_bytes=64 << 20, tile_x=32,
                        rows_per_tile=128, steps_per_launch=3)
        for nx, ny in [(8, 8), (33, 17), (129, 31), (64, 250)]:
            b.admit(wblbe.Params(nx, ny, 0.85, 0.0128, 0.01, 1.0, 0.2, precision=precision),
                    np.full((ny, nx), 0.6), 0.0, 10 ** 6)
        b.advance(2)
        b.close()
        runs += 1
    print(json.dumps({"errors": wblbe.debug_bounds_errors(), "runs": runs}), flush=True)


if __name__ == "__main__":
    main()
