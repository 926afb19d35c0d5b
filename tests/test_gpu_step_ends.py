"""How the one-problem Arnoldi step ends where the several-problem step is the
reference: an operator output that is not finite, or whose norm is not, ends
the cycle by its breakdown flag (no time-out, no non-finite iterate); and JM-VIE
vectors (6N) of several lengths, against the complex128 solve (the several-
problem kernel)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie, workloads  # noqa: E402

pytestmark = pytest.mark.gpu


# 1 + chi = -1e-30 j: M = 1e30, entries of w are finite in complex64 and |w|^2 is not; 1e-60: M itself is not
@pytest.mark.parametrize("near_zero", [-1e-30j, -1e-60j])
@pytest.mark.parametrize("grid", [(3, 2, 2), (40, 12, 9)])
def test_non_finite_output_ends_by_breakdown(grid, near_zero):
    eps = workloads.random_permittivity(grid, seed=51)
    eps[0, 1, 1] = 2.085 * near_zero
    b = torch.from_numpy(workloads.random_currents(grid, seed=52).astype(np.complex128).ravel()).cuda()
    plans = [vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, 2.085) for _ in range(2)]
    for p in plans:
        vie.vie_set_permittivity(p, eps)
    x = torch.zeros_like(b)
    one = vie.vie_solve(plans[0], b, x, 1e-8, restart=20, timeout_s=20.0, raise_on_not_converged=False)
    xs = [torch.zeros_like(b) for _ in range(2)]
    status, two = vie.vie_solve_batch(plans, [b, b], xs, 1e-8, restart=20, timeout_s=20.0,
                                      raise_on_not_converged=False)
    assert status == 4 and one["status"] == 4            # VIE_ERR_NOT_CONVERGED: no progress
    assert not one["converged"] and not two[0]["converged"]
    assert one["iterations"] == two[0]["iterations"]
    assert torch.isfinite(torch.view_as_real(x)).all()
    # the plan stays usable
    vie.vie_set_permittivity(plans[0], 2.085 + 0.1 * (workloads.random_permittivity(grid, seed=51) - 2.085))
    assert vie.vie_solve(plans[0], b, x, 1e-8, restart=20)["converged"]


# 2, 4, 8 and 12 elements a thread
@pytest.mark.parametrize("grid", [(10, 9, 5), (100, 50, 8), (300, 30, 10), (450, 30, 10)])
def test_jm_vectors(grid):
    plan = vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, 2.085)
    vie.vie_set_permittivity(plan, 2.085 + 0.1 * (workloads.random_permittivity(grid, seed=53) - 2.085))
    vie.vie_set_permeability(plan, 1.0 + 0.1 * (workloads.random_permittivity(grid, seed=54) - 1.0))
    b = torch.from_numpy(np.concatenate([workloads.random_currents(grid, seed=s) for s in (55, 56)])
                         .astype(np.complex128).ravel()).cuda()
    x, y, r = torch.zeros_like(b), torch.zeros_like(b), torch.empty_like(b)
    tol = 1e-8
    mixed = vie.vie_jm_solve(plan, b, x, tol, mode=vie.VIE_SOLVE_MIXED, restart=30)
    full = vie.vie_jm_solve(plan, b, y, tol, mode=vie.VIE_SOLVE_FP64, restart=30)
    assert mixed["converged"] and full["converged"]
    vie.vie_jm_matvec(plan, x, r)
    assert torch.linalg.vector_norm(b - r).item() <= 1.001 * tol * torch.linalg.vector_norm(b).item()
    # two solutions of residual tol of a well-conditioned system
    assert torch.linalg.vector_norm(x - y).item() <= 1e-6 * torch.linalg.vector_norm(y).item()
