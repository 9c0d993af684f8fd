"""The adjoint beside a strong jump: no cell outside the chosen stencils enters.

With the choices frozen, the cotangent of a cell of L depends on the cells of
the stencils that its two interfaces chose (each field and side), on the two
cells beside each interface (Roe average) and on the argmax cells of alpha; on
no other.  Smooth flow on the left of a jump by K in density and pressure:

- dL/dU of cells left of the jump is exactly 0 in every cell outside that set;
- the left side's part of it is the same for K = 2^10 and 2^20, bit for bit:
  powers of two leave every velocity, and so every alpha, as it is, and with
  equal choices nothing else reads the far side.
"""
import numpy as np
import pytest

import oracle
from paper_2311_15504_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, JUMP, NY = 96, 48, 12


def state(K, dims):
    x = (np.arange(N) + 0.5) / N
    k = np.where(np.arange(N) < JUMP, 1.0, K)
    rho = k * (1.0 + 0.2 * np.sin(7 * x))
    p = k * (1.0 + 0.3 * np.cos(5 * x))
    u = 0.3 + 0.1 * np.sin(6 * x)
    if dims == 1:
        return wl.conserved_1d(rho, u, p)
    v = 0.1 * np.cos(4 * x)
    return np.ascontiguousarray(np.repeat(wl.conserved_2d(rho, u, v, p)[:, None, :], NY, axis=1))


def stencil_cells(order, sel, k, side):
    """Cells that interface x_{k-1/2} reads on `side` with choice sel."""
    T = oracle.num_tested(order)
    m, n = ((0, 1), (1, 0), (0, 0))[sel - T] if sel >= T else oracle.candidate(order, sel)[:2]
    return range(k - 1 - m, k + n) if side == 0 else range(k - n, k + m + 1)


def gradient(order, K, dims):
    """dL/dU^T applied to a cotangent on the cells left of the jump, the x
    selections [2][fields][rows][N + 1] and the argmax cells of alpha [rows][3]."""
    from paper_2311_15504_gb300 import enomr
    U = torch.from_numpy(state(K, dims)).cuda()
    shape = N if dims == 1 else (NY, N)
    s = enomr.Solver(enomr.EULER, shape, order=order, dx=1.0 / N, dy=1.0 / N, bc=enomr.TRANSMISSIVE)
    sel = s.selection(U).cpu().numpy().astype(int)
    C, rows = (3, 1) if dims == 1 else (4, NY)
    sel = sel[:2 * C * rows * (N + 1)].reshape(2, C, rows, N + 1)
    bar = torch.zeros_like(U)
    bar[..., 16:JUMP - 1] = torch.from_numpy(
        np.random.default_rng(order).standard_normal(tuple(U[..., 16:JUMP - 1].shape))).cuda()
    g = s.rhs_vjp(U, bar).cpu().numpy().reshape(C, rows, N)
    argmax = s.debug_alpha()[4].cpu().numpy()
    s.check_status()
    return g, sel, argmax


@pytest.mark.parametrize("dims", (1, 2))
@pytest.mark.parametrize("order", (5, 7, 9, 13, 17))
def test_adjoint_reads_the_chosen_stencils_only(order, dims):
    grads = {}
    for K in (2.0 ** 10, 2.0 ** 20):
        g, sel, argmax = gradient(order, K, dims)
        for row in range(g.shape[1]):
            near = set()
            for k in range(16, JUMP):
                near |= {k - 1, k}
                for side in (0, 1):
                    for f in range(g.shape[0]):
                        near |= set(stencil_cells(order, sel[side, f, row, k], k, side))
            assert max(near) < JUMP  # the choices avoid the jump
            far = np.ones(N, bool)
            far[sorted(near)] = False
            far[argmax[row]] = False
            assert far[JUMP:].sum() > 40
            assert not g[:, row, far].any(), (K, row, np.abs(g[:, row, far]).max())
        grads[K] = (g, sel[..., :JUMP], argmax)
    (a, sa, ma), (b, sb, mb) = grads.values()
    assert (sa == sb).all() and (ma == mb).all()
    inner = slice(None) if dims == 1 else slice(2, NY - 2)  # ghost rows add to the first and last row
    for row in range(a.shape[1])[inner]:
        cells = np.setdiff1d(np.arange(JUMP), ma[row])
        assert np.array_equal(a[:, row, cells], b[:, row, cells]), \
            np.abs(a[:, row, cells] - b[:, row, cells]).max() / np.abs(a).max()
