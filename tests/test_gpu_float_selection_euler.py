"""The float form of the Euler selections against the FP64 form, bit for bit.

- With boundary sides the 2D sweeps select in FP64 throughout: four explicit
  transmissive sides and the plain transmissive grid are the same problem.
- A state times 2^200 takes every difference out of the range of the float
  form, so each window is left to FP64; velocities, sound speeds and Roe
  averages do not change, and the scheme commutes with a power of two exactly.

The data make the float form decide, nearly decide and leave open: exact ties,
differences of a few ulp, jumps, and fields whose differences cancel in the
projection.
"""
import numpy as np
import pytest

from paper_2311_15504_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ORDERS = (5, 7, 9, 11, 13, 15, 17)
FACTOR = 2.0 ** 200
KINDS = ("smooth", "isentropic", "ties", "steps", "rounding", "nearly_flat", "jumps", "random")


def primitives(shape, kind):
    """(rho, u, v, p) arrays."""
    rng = np.random.default_rng(len(kind))
    y, x = np.meshgrid(*((np.arange(n) + 0.5) / n for n in shape), indexing="ij")
    wave = np.sin(2 * np.pi * (x + 0.3 * y)) + 0.1 * np.sin(14 * np.pi * x + 6 * y)
    one = np.ones(shape)
    if kind == "smooth":
        return 1.3 + 0.2 * wave, 0.3 + 0.1 * wave, 0.2 * np.cos(5 * x - 3 * y), 1 + 0.1 * wave
    if kind == "isentropic":  # the entropy field's differences cancel
        rho = 1 + 0.05 * wave
        return rho, 0.3 * one, 0.1 * wave, rho ** 1.4
    if kind == "ties":
        q = rng.integers(1, 4, (4,) + shape).astype(float)
        return q[0], 0.25 * q[1], 0.125 * q[2], q[3]
    if kind == "steps":
        q = rng.integers(1, 5, (4, shape[0] // 5 + 1, shape[1] // 7 + 1)).astype(float)
        q = np.repeat(np.repeat(q, 5, 1), 7, 2)[:, :shape[0], :shape[1]]
        return q[0], 0.25 * q[1], 0.125 * q[2], q[3]
    if kind == "rounding":
        q = 1.0 + 2.2e-16 * rng.integers(0, 9, (4,) + shape)
        return q[0], 0.3 * q[1], -0.2 * q[2], q[3]
    if kind == "nearly_flat":
        return 1 + 1e-12 * wave, 0.3 + 1e-13 * wave, 0.2 * one, 1 + 1e-11 * wave
    if kind == "jumps":
        left = (x + 0.2 * y) % 0.31 < 0.12
        return (np.where(left, 1.0, 1e-3) * (1 + 0.01 * wave), np.where(left, 0.3, -0.2),
                0.1 * wave, np.where(left, 1.0, 2e-2))
    q = rng.uniform(-1, 1, (4,) + shape)
    return 1.5 + q[0], q[1], q[2], 1.5 + q[3]


def same(a, b):
    return torch.equal(a.view(torch.int64), b.view(torch.int64))


@pytest.mark.parametrize("shape", ((37, 300), (260, 257)))  # without and with a block map
@pytest.mark.parametrize("order", ORDERS)
def test_2d_equals_the_fp64_selecting_sweeps(order, shape):
    from paper_2311_15504_gb300 import enomr
    plain = enomr.Solver(enomr.EULER, shape, order=order, dx=0.1, dy=0.2, bc=enomr.TRANSMISSIVE)
    sided = enomr.Solver(enomr.EULER, shape, order=order, dx=0.1, dy=0.2, bc=enomr.TRANSMISSIVE)
    for i in range(4):
        sided.set_side(i, "transmissive")
    for kind in KINDS:
        U = torch.from_numpy(wl.conserved_2d(*primitives(shape, kind))).cuda()
        assert torch.equal(plain.selection(U), sided.selection(U)), kind
        # elsewhere D_x + D_y is rounded alike; signs of zeros are not compared
        assert torch.equal(plain.rhs(U), sided.rhs(U)), kind


@pytest.mark.parametrize("staging", ("STAGING_LOADS", "STAGING_TMA"))
@pytest.mark.parametrize("order", ORDERS)
def test_2d_commutes_with_a_power_of_two(order, staging):
    from paper_2311_15504_gb300 import enomr
    shape = (258, 260)
    s = enomr.Solver(enomr.EULER, shape, order=order, dx=0.1, dy=0.2, bc=enomr.PERIODIC)
    s.set_staging(getattr(enomr, staging))
    for kind in KINDS:
        U = torch.from_numpy(wl.conserved_2d(*primitives(shape, kind))).cuda()
        assert torch.equal(s.selection(U), s.selection(U * FACTOR)), kind
        assert same(s.rhs(U) * FACTOR, s.rhs(U * FACTOR)), kind
    s.check_status()


# the window-per-warp sweep at its tiles' edges, and the interface-per-lane one
@pytest.mark.parametrize("n", (40, 62, 63, 2000, 65001))
@pytest.mark.parametrize("order", ORDERS)
def test_1d_commutes_with_a_power_of_two(order, n):
    from paper_2311_15504_gb300 import enomr
    s = enomr.Solver(enomr.EULER, n, order=order, dx=1.0 / n, bc=enomr.PERIODIC)
    for kind in KINDS:
        rho, u, _, p = (q[0] for q in primitives((1, n), kind))
        U = torch.from_numpy(np.ascontiguousarray(wl.conserved_1d(rho, u, p))).cuda()
        assert torch.equal(s.selection(U), s.selection(U * FACTOR)), kind
        assert same(s.rhs(U) * FACTOR, s.rhs(U * FACTOR)), kind
    s.check_status()


@pytest.mark.parametrize("order", ORDERS)
def test_batch_commutes_with_a_power_of_two(order):
    from paper_2311_15504_gb300 import enomr
    sizes = [40, 61, 62, 63, 64, 500, 1201]
    b = enomr.Batch(sizes, [1.0 / n for n in sizes], order=order, bc=enomr.PERIODIC)
    for kind in KINDS:
        q = [[a[0] for a in primitives((1, n), kind)] for n in sizes]
        U = b.pack([wl.conserved_1d(rho, u, p) for rho, u, _, p in q])
        V = U * FACTOR
        for _ in range(2):
            b.step(U, 0.2)
            b.step(V, 0.2)
        assert same(U * FACTOR, V), kind
