"""The forms of the scalar kernels against one another, bit for bit.

- Lines of few CTAs run instances with more registers than long ones: a
  periodic line repeated end to end has the same right-hand side in each copy.
- The one-launch step spreads a line over a cluster: the sizes at which the
  number of its CTAs changes, against the stages one at a time.
- The speed reduction takes eight cells per thread, the last ones of a line too.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ORDERS = (5, 7, 9, 11, 13, 15, 17)
EQS = ("advection", "advection_left", "burgers", "burgers_left", "burgers_mixed")


def line(n, eq):
    """Smooth, a plateau, noise of a few ulp, a jump and random cells."""
    rng = np.random.default_rng(n)
    u = 1.2 + 0.3 * np.sin(2 * np.pi * np.arange(n) / n)
    q = n // 5
    u[q:2 * q] = 1.1
    u[2 * q:3 * q] = 0.9 + 2.2e-16 * rng.integers(0, 9, q)
    u[3 * q:4 * q] = rng.uniform(0.5, 1.5, q)
    return -u if eq == "burgers_left" else (u - 1.0 if eq == "burgers_mixed" else u)


def solver(eq, n, order, h, bc):
    from paper_2311_15504_gb300 import enomr
    return enomr.Solver(enomr.BURGERS if eq.startswith("burgers") else enomr.ADVECTION, n,
                        order=order, dx=h, bc=bc, adv_speed=-0.7 if eq.endswith("left") else 1.0)


@pytest.mark.parametrize("eq", EQS)
@pytest.mark.parametrize("order", ORDERS)
def test_long_line_equals_its_period(order, eq):
    n, copies = 5003, 16  # 20 CTAs of 255 cells, and 314
    u = torch.from_numpy(line(n, eq)).cuda()
    a = solver(eq, n, order, 0.01, 0).rhs(u)
    b = solver(eq, n * copies, order, 0.01, 0).rhs(u.repeat(copies))
    assert torch.equal(b.view(copies, n), a.expand(copies, n))


@pytest.mark.parametrize("n", (254, 255, 256, 509, 510, 511, 765, 766, 1020, 1021, 1024))
@pytest.mark.parametrize("eq", EQS)
@pytest.mark.parametrize("order", (5, 9, 17))
def test_step_over_a_cluster_equals_its_stages(order, eq, n):
    U = torch.from_numpy(line(n, eq)).cuda()
    for bc in (0, 1):
        s = solver(eq, n, order, 2.0 / n, bc)
        a, b, v = torch.empty_like(U), torch.empty_like(U), U.clone()
        for _ in range(3):
            w = v.clone()
            dt = s.cfl_dt(w, 0.4)
            s.stage(1, w, w, a, dt)
            s.stage(2, w, a, b, dt)
            s.stage(3, w, b, a, dt)
            assert s.step(v, 0.0, 0.4, return_dt=True) == dt
            assert torch.equal(a, v)
        s.check_status()


@pytest.mark.parametrize("n", (20, 255, 1025, 2047, 2048, 2049, 30001, 2490367, 2490369, 4980737))
def test_speed_of_a_line(n):
    """cfl / max |u| with the largest cell at the ends and in the middle."""
    s = solver("burgers", n, 5, 0.5, 0)
    for at in (0, 1, n // 3, n - 2, n - 1):
        u = torch.full((n,), 0.25, dtype=torch.float64, device="cuda")
        u[at] = -2.0
        assert s.cfl_dt(u, 0.5) == 0.5 / (2.0 * (1.0 / 0.5))
    s.check_status()
