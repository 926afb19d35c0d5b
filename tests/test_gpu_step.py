"""The Arnoldi step of a single complex64 problem (its vector in registers, 2 to
16 elements a thread, and the kernel for longer vectors) against the step of
several problems: same problem, same number of iterations up to rounding, and a
residual, formed with the complex128 operator, below the tolerance (the solver
stops on the same quantity; 1e-3 of it for the other order of summation)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie, workloads  # noqa: E402

pytestmark = pytest.mark.gpu


def _solve(grid, restart, tol=1e-8):
    eps_bg = 2.085
    eps = eps_bg + 0.25 * (workloads.random_permittivity(grid, seed=11) - eps_bg)
    b = torch.from_numpy(workloads.random_currents(grid, seed=12).astype(np.complex128).ravel()).cuda()
    plans = [vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, eps_bg) for _ in range(2)]
    for p in plans:
        vie.vie_set_permittivity(p, eps)
    x = torch.zeros_like(b)
    one = vie.vie_solve(plans[0], b, x, tol, restart=restart)
    y = torch.empty_like(b)
    vie.vie_matvec(plans[0], x, y)
    assert one["converged"]
    assert torch.linalg.vector_norm(b - y).item() <= 1.001 * tol * torch.linalg.vector_norm(b).item()
    xs = [torch.zeros_like(b) for _ in range(2)]
    _, two = vie.vie_solve_batch(plans, [b, b], xs, tol, restart=restart)
    assert abs(one["iterations"] - two[0]["iterations"]) <= 2 + one["iterations"] // 10


# 3 unknowns; one block; the largest vectors of 2 elements a thread; 4, 6, 8, 12, 16 elements; longer vectors
@pytest.mark.parametrize("grid", [(1, 1, 1), (7, 5, 3), (101, 51, 10), (128, 80, 10), (150, 100, 10), (128, 160, 10),
                                  (300, 100, 10), (400, 100, 10), (420, 100, 10)])
def test_vector_lengths(grid):
    _solve(grid, 30)


# bases below, at and past the 16 and 32 vectors that are swept at a time
@pytest.mark.parametrize("restart", [1, 2, 16, 17, 33, 70])
def test_basis_lengths(restart):
    _solve((40, 12, 9), restart)
