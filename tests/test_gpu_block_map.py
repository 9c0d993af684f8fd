"""The block map of the 2D sweeps against the same arithmetic without it.

- The right-hand side through a context (block map, tile lists, dead blocks
  written without a sweep) equals enomr_rhs_euler2d_noalloc(), which has no
  map, bit for bit: jumps, single cells and thin lines on and beside block
  edges, odd and even sizes, ragged last blocks, both boundary kinds.
- Whole steps: a state that varies along one direction only gives the same
  rows (columns) on a grid of few lines, below the size that has a map.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2311_15504_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def state(ny, nx, marks, seed=0):
    """One constant state with rectangles (y0, y1, x0, x1) of others on it."""
    rng = np.random.default_rng(seed)
    prim = np.empty((4, ny, nx))
    prim[:] = np.array([1.0, 0.3, -0.2, 1.0])[:, None, None]
    for y0, y1, x0, x1 in marks:
        prim[:, y0:y1, x0:x1] = rng.uniform([0.5, -0.4, -0.4, 0.5], [1.5, 0.4, 0.4, 1.5])[:, None, None]
    return wl.conserved_2d(*prim)


MARKS = {
    "none": [],
    "corner_cell": [(0, 1, 0, 1)],
    "last_cell": [(-1, None, -1, None)],
    "block_edge_cells": [(31, 32, 95, 96), (64, 65, 160, 161)],
    "thin_lines": [(0, None, 127, 128), (100, 101, 0, None)],
    "quadrants": [(0, 150, 0, 170), (150, None, 170, None)],
    "many": [(7 * i, 7 * i + 1, 13 * i, 13 * i + 2) for i in range(18)],
}


@pytest.mark.parametrize("bc", (0, 1))
@pytest.mark.parametrize("shape", ((256, 256), (257, 301), (300, 258), (1100, 70)))
def test_rhs_with_and_without_map(shape, bc):
    from paper_2311_15504_gb300 import enomr
    ny, nx = shape
    for order in (5, 17):
        s = enomr.Solver(enomr.EULER, shape, order=order, dx=0.1, dy=0.2, bc=bc)
        for name, marks in MARKS.items():
            U = torch.from_numpy(state(ny, nx, [m for m in marks if (m[0] or 0) < ny
                                                and (m[2] or 0) < nx])).cuda()
            ref = torch.empty_like(U)
            p = ctypes.c_void_p
            rc = enomr._lib.enomr_rhs_euler2d_noalloc(
                p(U.data_ptr()), p(ref.data_ptr()), nx, ny, 0.1, 0.2, order, 1.4, bc,
                p(torch.cuda.current_stream().cuda_stream))
            assert rc == 0
            got = torch.full_like(U, 7.0)  # every cell must be written
            for occupancy in (enomr.OCCUPANCY_HIGH, enomr.OCCUPANCY_LOW):
                s.set_occupancy(occupancy)
                s.rhs(U, out=got)
                assert torch.equal(got.view(torch.int64), ref.view(torch.int64)), (name, order)
        s.check_status()


@pytest.mark.parametrize("along", ("x", "y"))
@pytest.mark.parametrize("dt", (0.0, 0.02))
def test_steps_with_and_without_map(along, dt):
    from paper_2311_15504_gb300 import enomr
    n, few, many = 500, 40, 300
    line = state(1, n, [(0, 1, 0, 200), (0, 1, 401, 402)], seed=3)  # [4][1][n]
    if along == "y":
        line = line[[0, 2, 1, 3]].transpose(0, 2, 1)

    def run(lines):
        U = np.repeat(line, lines, axis=1 if along == "x" else 2)
        shape = U.shape[1:]
        s = enomr.Solver(enomr.EULER, shape, order=9, dx=0.1, dy=0.1)
        U = torch.from_numpy(np.ascontiguousarray(U)).cuda()
        for _ in range(4):
            s.step(U, dt, 0.4)
        s.check_status()
        return U

    a, b = run(few), run(many)
    one = a[:, :1] if along == "x" else a[:, :, :1]
    assert torch.equal(a, one.expand_as(a)) and torch.equal(b, one.expand_as(b))
