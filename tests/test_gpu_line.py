"""The single-problem 1D Euler step against the batched one, bit for bit.

enomr_step on a line runs the window-per-warp sweep (tiles of 31 cells; on long
lines the interface-per-lane one) with the next stage's wave speeds in its
epilogue; the batch runs its own tile function and reductions.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2311_15504_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 5, 30, 31, 32, 33, 61, 62, 63, 64, 93, 500, 2017)


def states(sizes, seed):
    rng = np.random.default_rng(seed)
    out = []
    for n in sizes:
        x = (np.arange(n) + 0.5) / n
        rho = np.where(x < 0.4, 1.0, 0.3) * (1 + 0.1 * np.sin(9 * x + rng.uniform(0, 3)))
        out.append(wl.conserved_1d(np.where(x > 0.8, 0.5, rho), np.where(x < 0.6, 0.3, -0.2),
                                   np.where(x < 0.4, 1.0, 0.2)))
    return out


def compare(sizes, order, bc, steps):
    from paper_2311_15504_gb300 import enomr
    Us, hs = states(sizes, order), 1.0 / np.array(sizes)
    B = enomr.Batch(sizes, hs, order=order, bc=bc)
    Ub = B.pack(Us)
    Ul = [torch.from_numpy(u).cuda() for u in Us]
    S = [enomr.Solver(enomr.EULER, int(n), order=order, dx=float(h), bc=bc)
         for n, h in zip(sizes, hs)]
    for _ in range(steps):
        B.step(Ub, 0.4)
        for s, u in zip(S, Ul):
            s.step(u, 0.0, 0.4)
    for p, u in enumerate(Ul):
        assert torch.equal(B.view(Ub, p), u), (sizes[p], order, bc)


@pytest.mark.parametrize("order", (5, 9, 17))
@pytest.mark.parametrize("bc", (0, 1))
def test_line_equals_batch(order, bc):
    compare([n for n in SIZES if bc == 1 or n >= order + 1], order, bc, 3)


@pytest.mark.parametrize("order", (5, 17))
def test_long_line_equals_batch(order):
    compare([2 ** 17, 2 ** 17 + 1], order, 1, 1)


def test_fixed_step_equals_its_stages():
    from paper_2311_15504_gb300 import enomr
    u = torch.from_numpy(states([500], 1)[0]).cuda()
    s = enomr.Solver(enomr.EULER, 500, order=9, dx=0.002)
    a, b, v = torch.empty_like(u), torch.empty_like(u), u.clone()
    dt = 2e-4
    s.stage(1, u, u, a, dt)
    s.stage(2, u, a, b, dt)
    s.stage(3, u, b, a, dt)
    s.step(v, dt)
    assert torch.equal(a, v)
    s.check_status()


@pytest.mark.parametrize("order, longest", ((5, 40000), (9, 40000), (11, 65000), (17, 65000)))
def test_lines_beside_the_change_of_sweep_equal_batch(order, longest):
    """The longest line that the window-per-warp sweep takes, and one cell more."""
    for bc in (0, 1):
        compare([longest, longest + 1], order, bc, 2)
