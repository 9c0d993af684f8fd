"""Small batches run instances with more registers than large ones: a problem
gives the same bits in either, for every tile shape that autotuning can choose."""
import numpy as np
import pytest

from paper_2311_15504_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", (5, 7, 9, 11, 13, 15, 17))
def test_problem_alone_and_among_many(order):
    from paper_2311_15504_gb300 import enomr
    rng = np.random.default_rng(order)
    n, copies = 301, 700  # 10, 5 or 3 tiles; 2100 to 7000 tiles
    x = (np.arange(n) + 0.5) / n
    rho = np.where(x < 0.4, 1.0, 0.3) * (1 + 0.1 * np.sin(9 * x))
    rho[200:260] = 0.5 + 2.2e-16 * rng.integers(0, 9, 60)
    u = torch.from_numpy(wl.conserved_1d(rho, np.where(x < 0.6, 0.3, -0.2), np.where(x < 0.5, 1.0, 0.2)))
    for bc in (0, 1):
        one = enomr.Batch([n], [1.0 / n], order=order, bc=bc)
        many = enomr.Batch([n] * copies, [1.0 / n] * copies, order=order, bc=bc)
        a, b = one.pack([u]), many.pack([u] * copies)
        for _ in range(2):
            one.autotune(a, 1)
            many.autotune(b, 1)
            one.step(a, 0.4)
            many.step(b, 0.4)
            assert torch.equal(b.view(copies, -1), a.expand(copies, -1))
        one.check_status()
        many.check_status()
