"""The block map of the 2D sweeps: non-finite patches, and whole steps.

- A patch of equal cells without a finite flux is no constant block: its
  flux differences are NaN, as the sweeps without a map have them.
- enomr_step keeps block maps from stage to stage (blocks known to be constant
  are not read again, and the combination of a block known in U^n too reads one
  cell of it); three enomr_stage calls make each stage's map from that state
  alone.  The same bits, on states that vary in both directions.
"""
import ctypes

import numpy as np
import pytest

from paper_2311_15504_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PATCHES = {  # conserved state of the patch
    "nan": (np.nan,) * 4,
    "nan_energy": (1.0, 0.3, -0.2, np.nan),
    "inf_energy": (1.0, 0.3, -0.2, np.inf),
    "overflow": (1.0, 0.3, -0.2, 1.7e308),
    "vacuum": (0.0, 0.3, -0.2, 1.0),
    "negative_density": (-1.0, 0.3, -0.2, 1.0),
    "negative_pressure": (1.0, 3.0, -0.2, 1.0),
    "large": (2.0 ** 120, 2.0 ** 120, 0.0, 2.0 ** 122),
}


@pytest.mark.parametrize("order", (5, 9, 17))
@pytest.mark.parametrize("patch", sorted(PATCHES))
def test_rhs_of_a_non_finite_patch(patch, order):
    from paper_2311_15504_gb300 import enomr
    ny, nx = 300, 330
    U = wl.conserved_2d(*(np.full((ny, nx), v) for v in (1.0, 0.3, -0.2, 1.0)))
    U[:, 37:221, 50:270] = np.array(PATCHES[patch])[:, None, None]
    for bc in (0, 1):
        s = enomr.Solver(enomr.EULER, (ny, nx), order=order, dx=0.1, dy=0.2, bc=bc)
        Ud = torch.from_numpy(U).cuda()
        ref, p = torch.empty_like(Ud), ctypes.c_void_p
        rc = enomr._lib.enomr_rhs_euler2d_noalloc(
            p(Ud.data_ptr()), p(ref.data_ptr()), nx, ny, 0.1, 0.2, order, 1.4, bc,
            p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        got = s.rhs(Ud)
        assert torch.equal(got.isnan(), ref.isnan())
        ok = ~ref.isnan()
        assert torch.equal(got[ok].view(torch.int64), ref[ok].view(torch.int64))
        if patch not in ("large",):
            with pytest.raises(enomr.EnomrError):
                s.check_status()


def varied(ny, nx, kind):
    rng = np.random.default_rng(len(kind))
    prim = np.empty((4, ny, nx))
    prim[:] = np.array([1.0, 0.3, -0.2, 1.0])[:, None, None]

    def box(y0, y1, x0, x1):
        prim[:, y0:y1, x0:x1] = rng.uniform([0.5, -0.4, -0.4, 0.5], [1.5, 0.4, 0.4, 1.5])[:, None, None]
    if kind == "quadrants":
        box(0, 150, 0, 170)
        box(150, None, 170, None)
    elif kind == "block_corners":
        for y, x in ((31, 95), (64, 160), (96, 31), (159, 191)):
            box(y, y + 1, x, x + 1)
    elif kind == "edges":
        box(0, 1, 0, 1)
        box(ny - 1, ny, nx - 1, nx)
        box(100, 103, 0, 2)
    elif kind == "lines":
        box(0, ny, 127, 128)
        box(100, 101, 0, nx)
    return wl.conserved_2d(*prim)


@pytest.mark.parametrize("kind", ("quadrants", "block_corners", "edges", "lines"))
@pytest.mark.parametrize("bc", (0, 1))
@pytest.mark.parametrize("shape", ((257, 301), (288, 256), (1100, 70)))
def test_step_equals_its_stages(shape, bc, kind):
    """The front crosses block edges from the first stage on (an edge lies on a
    block edge or a cell beside it), so live blocks appear in every stage."""
    from paper_2311_15504_gb300 import enomr
    for order in (5, 17):
        s = enomr.Solver(enomr.EULER, shape, order=order, dx=0.1, dy=0.2, bc=bc)
        U = torch.from_numpy(varied(*shape, kind)).cuda()
        a, b = torch.empty_like(U), torch.empty_like(U)
        for i in range(6):
            dt = s.cfl_dt(U, 0.4) if i % 2 else 0.02
            V = U.clone()
            s.stage(1, U, U, a, dt)
            s.stage(2, U, a, b, dt)
            s.stage(3, U, b, a, dt)
            if i % 2:
                assert s.step(V, 0.0, 0.4, return_dt=True) == dt
            else:
                s.step(V, dt)
            assert torch.equal(a.view(torch.int64), V.view(torch.int64)), (order, i)
            U.copy_(V)
        s.check_status()
