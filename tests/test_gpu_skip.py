"""A batch of two shapes in which the last shape's problem stops at its first
step: its passes are skipped from then on while the other shape's run.  The
solution of the other one, whose residual is formed with the complex128
operator, and its number of steps are those of the problem solved alone (up to
the order of summation)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie, workloads  # noqa: E402

pytestmark = pytest.mark.gpu


# second grid: compiled x and y-z passes, run-time radices, the split pass B
@pytest.mark.parametrize("done", [(600, 23, 11), (90, 30, 12), (40, 24, 24), (5, 150, 6)])
def test_skipped_shape_behind_a_running_one(done):
    def problem(grid, scale):
        plan = vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, 2.085)
        eps = 2.085 + scale * (workloads.random_permittivity(grid, seed=21) - 2.085)
        vie.vie_set_permittivity(plan, eps)
        b = torch.from_numpy(workloads.random_currents(grid, seed=22).astype(np.complex128).ravel()).cuda()
        return plan, b

    tol = 1e-6
    (p0, b0), (p1, b1) = problem((200, 27, 11), 0.5), problem(done, 0.0)
    x0, x1 = torch.zeros_like(b0), torch.zeros_like(b1)
    alone = vie.vie_solve(p0, b0, x0, tol, restart=30)
    xs = [torch.zeros_like(b0), torch.zeros_like(b1)]
    status, infos = vie.vie_solve_batch([p0, p1], [b0, b1], xs, tol, restart=30)
    assert status == 0 and all(i["converged"] for i in infos) and infos[1]["iterations"] == 1
    assert abs(infos[0]["iterations"] - alone["iterations"]) <= 2 + alone["iterations"] // 10
    for plan, b, x in ((p0, b0, xs[0]), (p1, b1, xs[1])):
        y = torch.empty_like(b)
        vie.vie_matvec(plan, x, y)
        assert torch.linalg.vector_norm(b - y).item() <= 1.001 * tol * torch.linalg.vector_norm(b).item()
