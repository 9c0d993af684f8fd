"""The float form of the selection and of the value sum against the FP64 form.

A state times 2^200 takes every difference out of the range of the float
form, so the kernels evaluate it in FP64 throughout, and the scheme commutes
with a power of two bit for bit.  Selections must therefore be equal with and
without the factor, and right-hand sides equal to the rounding of the value
sums: W products of weights with sum |a| <= 2.7 on both forms.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FACTOR = 2.0 ** 200
ORDERS = (5, 9, 13, 17)


def lines(n):
    """Windows at which the float form decides, nearly decides and cannot decide."""
    rng = np.random.default_rng(n)
    x = np.arange(n) / n
    smooth = 1.2 + np.sin(2 * np.pi * x) + 0.1 * np.sin(14 * np.pi * x + 1)
    plateau = 1 + 0.3 * np.sin(4 * np.pi * x)
    plateau[n // 3:n // 2] = plateau[n // 3]
    return {
        "smooth": smooth,
        "zeros": np.sin(2 * np.pi * x),
        "steps": np.repeat(rng.integers(1, 5, n // 7 + 1), 7)[:n].astype(float),  # exact ties
        "ints": rng.integers(-4, 5, n).astype(float),
        "rounding": 1.0 + 2.2e-16 * rng.integers(0, 9, n),  # differences of a few ulp
        "nearly_flat": 1.0 + 1e-12 * smooth,
        "range_edge": 1.0 + 2.0 ** -6 * (1 + 1e-3 * rng.standard_normal(n)) * (np.arange(n) % 2),
        "plateau": plateau,
    }


def close(a, b, scale, order):
    # both sums round W products of size at most 2.7 scale; a difference of two
    # faces over h and the products of the flux double it
    tol = 2 * (order + 4) * 2.7 * 2.0 ** -53 * scale
    return np.abs(a - b).max() <= tol


@pytest.mark.parametrize("n", (40, 255, 256, 511, 1500))  # tiles of 255 cells
@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("eq", ("advection", "advection_left", "burgers", "burgers_left"))
def test_scalar_float_form(eq, order, n):
    from paper_2311_15504_gb300 import enomr
    h = 2.0 / n
    left = eq.endswith("left")
    for name, u in lines(n).items():
        burgers = eq.startswith("burgers")
        # the flux is quadratic for Burgers: the factor enters it squared
        k = np.sqrt(FACTOR) if burgers else FACTOR
        s = enomr.Solver(enomr.BURGERS if burgers else enomr.ADVECTION, n, order=order, dx=h,
                         bc=enomr.PERIODIC, adv_speed=-0.7 if left else 1.0)
        u = -u if burgers and left else u
        U = torch.from_numpy(u).cuda()
        assert torch.equal(s.selection(U), s.selection(U * k)), (name, eq)
        a, b = s.rhs(U).cpu().numpy(), s.rhs(U * k).cpu().numpy() / FACTOR
        flux = 0.5 * np.abs(u).max() ** 2 * (2 if burgers else 0) + np.abs(u).max()
        assert close(a, b, flux / h, order), (name, eq)
        s.check_status()


@pytest.mark.parametrize("n", (18, 31, 32, 33, 200, 511, 512, 513, 1023, 1024, 1025, 5000))
@pytest.mark.parametrize("order", (5, 17))
@pytest.mark.parametrize("eq", ("advection", "advection_left", "burgers", "burgers_left",
                                "burgers_mixed"))
def test_short_line_step_equals_its_stages(eq, order, n):
    """enomr_step of at most 1024 cells is one launch, a longer Burgers step takes
    the next stage's speed in each stage; enomr_stage is one launch each."""
    from paper_2311_15504_gb300 import enomr
    h = 2.0 / n
    u = lines(n)["plateau"]
    u = -u if eq == "burgers_left" else (u - 1.0 if eq == "burgers_mixed" else u)
    for bc in (enomr.PERIODIC, enomr.TRANSMISSIVE):
        s = enomr.Solver(enomr.BURGERS if eq.startswith("burgers") else enomr.ADVECTION, n,
                         order=order, dx=h, bc=bc, adv_speed=-0.7 if eq.endswith("left") else 1.0)
        U = torch.from_numpy(u).cuda()
        a, b, v = torch.empty_like(U), torch.empty_like(U), U.clone()
        dt = s.cfl_dt(U, 0.4)
        s.stage(1, U, U, a, dt)
        s.stage(2, U, a, b, dt)
        s.stage(3, U, b, a, dt)
        assert s.step(v, 0.0, 0.4, return_dt=True) == dt
        assert torch.equal(a, v)
        s.check_status()
